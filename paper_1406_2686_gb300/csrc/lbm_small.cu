// Many steps of a small D2Q9 lattice in one launch.  A step of a few thousand
// nodes is two kernels of about one microsecond of work, and launching,
// draining and reloading them from L2 takes the other two thirds of its time.
// Here one thread-block cluster holds the whole state in the shared memory of
// its blocks, one node per thread, and the step's two phases (collision and
// streaming; densities, FENE-P update and feedback stress) are separated by
// cluster barriers instead of kernel boundaries.  Neighbours in another block
// are read and pushed to through distributed shared memory; their addresses
// are worked out once per launch.  The node arithmetic is that of k_lattice and
// k_post, in the same order.
// Bound by the latency of one step's chain of dependent operations (one warp
// per scheduler at 64 x 32): 1.58 us a step there, 1.8 with two components, against
// 3.5 and 4.1 of the launch pairs; 64 x 64 1.8 / 3.5, 100 x 60 with two components
// 2.9 / 4.5, 128 x 64 2.5 / 3.6 and 3.4 / 4.4.  16 blocks, the largest cluster:
// 8 take 1.76 us at 64 x 32 and 2.4 at 64 x 64.  The populations stay in registers
// between moments and collision (read again from shared memory: 1.60 and, with
// two components, 2.0 us).
#include "fd_impl.cuh"
#include "lbm_impl.cuh"

namespace vefd {

namespace {

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// Address of this block's shared-memory location in block `rank` of the cluster.
__device__ __forceinline__ unsigned cluster_addr(unsigned local, unsigned rank) {
    unsigned a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    return a;
}

__device__ __forceinline__ float cluster_ld(unsigned a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}

__device__ __forceinline__ void cluster_st(unsigned a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

// Hardware barrier of all threads of the cluster; their shared-memory writes
// before it are visible after it.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// Planes of one float per node in a block's shared memory: two population
// buffers, densities, stress, velocity, two conformation buffers.
template <int NCOMP>
struct SmallPlanes {
    static constexpr int P = NCOMP * (D2Q9::Q - 1);
    static constexpr int F = 0, D = 2 * P, Q = D + NCOMP, U = Q + D2Q9::NQ, C = U + 2, total = C + 2 * D2Q9::NC;
};

// `nsteps` steady steps of b.fin, b.Cin, b.R, b.drho, b.Q, b.frest.  The state
// after them is written back to where as many single steps leave it: after an
// odd count to b.fout and (FD) b.Cout, else to b.fin and b.Cin.
template <class PT, int NCOMP, int COLL, bool FD>
__global__ void __launch_bounds__(kSmallMaxThreads) k_small(StepBufs b, StepParams p, int nsteps) {
    using L = D2Q9;
    using S = SmallPlanes<NCOMP>;
    extern __shared__ float sm[];
    const int M = blockDim.x, t = threadIdx.x, N = (int)p.N;
    const int i = (int)cluster_rank() * M + t;
    const bool active = i < N;
    const unsigned base = smem_u32(sm), pitch = 4u * (unsigned)M;
    const unsigned own = base + 4u * (unsigned)t;
    const int y = active ? i / p.nx : 0, x = active ? i - y * p.nx : 0;
    const bool wall_lo = p.walls && y == 0, wall_hi = p.walls && y == p.ny - 1;
    // this node's slot of every plane, and its neighbours' (clamped at walls, so
    // that a stencil point beyond one is the node itself)
    unsigned nb[L::Q];
    nb[0] = own;
#pragma unroll
    for (int a = 1; a < L::Q; ++a) {
        nb[a] = own;
        if (active) {
            const int j = y_clamped(y + L::cy(a), p.ny, p.walls) * p.nx + wrap1(x + L::cx(a), p.nx);
            if (idx_ok(j, N, b.status)) nb[a] = cluster_addr(base + 4u * (unsigned)(j % M), (unsigned)(j / M));
        }
    }
    auto at = [&](unsigned node, int plane) { return node + (unsigned)plane * pitch; };

    float rest[NCOMP], R[L::NC];
    const PT* fin = static_cast<const PT*>(b.fin);
    if (active) {
#pragma unroll
        for (int k = 0; k < S::P; ++k) cluster_st(at(own, S::F + k), pop_load(fin + (long long)k * N + i));
        float d[NCOMP];
        dens_ldg<NCOMP>(b.drho, i, d);
#pragma unroll
        for (int s = 0; s < NCOMP; ++s) {
            rest[s] = b.frest[s * N + i];
            cluster_st(at(own, S::D + s), d[s]);
        }
#pragma unroll
        for (int k = 0; k < L::NQ; ++k) cluster_st(at(own, S::Q + k), p.feedback != 0.0f ? b.Q[k * N + i] : 0.0f);
#pragma unroll
        for (int k = 0; k < L::NC; ++k) {
            cluster_st(at(own, S::C + k), b.Cin[k * N + i]);
            R[k] = FD && p.have_prev ? b.R[k * N + i] : 0.0f;
        }
    }
    cluster_barrier();

    for (int n = 0; n < nsteps; ++n) {
        const int cur = S::F + (n & 1) * S::P, nxt = S::F + (1 - (n & 1)) * S::P;
        const int cc = S::C + (FD ? n & 1 : 0) * L::NC, cn = S::C + (FD ? 1 - (n & 1) : 0) * L::NC;
        if (active) {
            // moments
            float dr[NCOMP], pif[NCOMP][6], f[NCOMP][L::Q];
            float jx = 0.0f, jy = 0.0f;
#pragma unroll
            for (int s = 0; s < NCOMP; ++s) {
                dr[s] = cluster_ld(at(own, S::D + s));
#pragma unroll
                for (int k = 0; k < 6; ++k) pif[s][k] = 0.0f;
#pragma unroll
                for (int a = 1; a < L::Q; ++a) {
                    const float fa = f[s][a] = cluster_ld(at(own, cur + s * (L::Q - 1) + a - 1));
                    if (L::cx(a)) jx += L::cx(a) * fa;
                    if (L::cy(a)) jy += L::cy(a) * fa;
                    if (COLL == 1) pi_add<L>(pif[s], a, fa);
                }
            }
            // Shan-Chen sums and polymer force, as neighbour_forces
            float acc[2][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}}, Fp[3] = {0.f, 0.f, 0.f}, qloc[L::NQ];
            if (NCOMP == 2) {
                float sa[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, sd[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
                for (int a = 1; a < L::Q; ++a) {
                    const bool axis = L::w(a) == L::w(1);
#pragma unroll
                    for (int s = 0; s < NCOMP; ++s) {
                        const float v = cluster_ld(at(nb[a], S::D + s));
                        float* acc_s = axis ? sa[s] : sd[s];
                        if (L::cx(a)) acc_s[0] += L::cx(a) * v;
                        if (L::cy(a)) acc_s[1] += L::cy(a) * v;
                    }
                }
#pragma unroll
                for (int s = 0; s < 2; ++s)
#pragma unroll
                    for (int k = 0; k < 2; ++k) acc[s][k] = L::w(1) * sa[s][k] + L::w(L::Q - 1) * sd[s][k];
            }
#pragma unroll
            for (int k = 0; k < L::NQ; ++k) qloc[k] = 0.0f;
            if (p.feedback != 0.0f) {
                if (p.coupling == 1) {
#pragma unroll
                    for (int k = 0; k < L::NQ; ++k) qloc[k] = cluster_ld(at(own, S::Q + k));
                } else {
                    // nb[1..4]: +x, -x, +y, -y
                    float div[2] = {0.f, 0.f};
                    const float h = wall_lo || wall_hi ? 1.0f : 0.5f;
#pragma unroll
                    for (int jj = 0; jj < 2; ++jj) {
                        const int kx = S::Q + qidx<L>(0, jj), ky = S::Q + qidx<L>(1, jj);
                        div[jj] += 0.5f * (cluster_ld(at(nb[1], kx)) - cluster_ld(at(nb[2], kx)));
                        div[jj] += h * (cluster_ld(at(nb[3], ky)) - cluster_ld(at(nb[4], ky)));
                    }
#pragma unroll
                    for (int k = 0; k < 2; ++k) Fp[k] = p.feedback * div[k];
                }
            }
            Local<NCOMP> st;
            local_state<L, NCOMP>(p, dr, jx, jy, 0.0f, acc, Fp, st, b.status);
            cluster_st(at(own, S::U), st.ux);
            cluster_st(at(own, S::U + 1), st.uy);
            collide_emit<PT, L, NCOMP, COLL>(
                p, st, qloc, pif, wall_lo, wall_hi,
                [&](int s, int a) { return f[s][a]; },
                [&](int s, int a, PT va, PT vb, bool ba, bool bb) {
                    const int pl = nxt + s * (L::Q - 1) + a - 1;  // plane of direction a; a + 1 is its opposite
                    cluster_st(ba ? at(own, pl + 1) : at(nb[a], pl), pop_get(va));
                    cluster_st(bb ? at(own, pl) : at(nb[a + 1], pl + 1), pop_get(vb));
                },
                rest);
        }
        cluster_barrier();
        if (active) {
            float d[NCOMP], c[L::NC];
#pragma unroll
            for (int s = 0; s < NCOMP; ++s) {
                d[s] = rest[s];
#pragma unroll
                for (int a = 1; a < L::Q; ++a) d[s] += cluster_ld(at(own, nxt + s * (L::Q - 1) + a - 1));
            }
            if (FD) {
                const unsigned pt[5] = {own, nb[2], nb[1], nb[4], nb[3]};
                auto v = [&](int k, int q) { return cluster_ld(at(pt[q], k < L::NC ? cc + k : S::U + k - L::NC)); };
                const bool wall = wall_lo || wall_hi;
                StepParams ps = p;
                ps.have_prev = p.have_prev || n > 0;
                float Rnew[L::NC];
                const unsigned bits = fenep_compute<L::D, L::NC>(v, wall ? 1.0f : 0.5f, wall ? 0.0f : 1.0f, R, ps, c, Rnew);
#pragma unroll
                for (int k = 0; k < L::NC; ++k) {
                    cluster_st(at(own, cn + k), c[k]);
                    R[k] = Rnew[k];
                }
                if (bits) atomicOr(b.status, bits);
            } else {
#pragma unroll
                for (int k = 0; k < L::NC; ++k) c[k] = cluster_ld(at(own, cc + k));
            }
#pragma unroll
            for (int s = 0; s < NCOMP; ++s) cluster_st(at(own, S::D + s), d[s]);
            if (p.feedback != 0.0f) store_feedback<L, NCOMP>(c, d, p, sm + S::Q * M + t, M, 0);
        }
        // also keeps every block here until no other one reads its planes
        cluster_barrier();
    }

    if (!active) return;
    const bool odd = nsteps & 1;
    const int fl = S::F + (odd ? S::P : 0), cl = S::C + (FD && odd ? L::NC : 0);
    PT* fo = odd ? static_cast<PT*>(b.fout) : const_cast<PT*>(fin);
    float* Co = odd ? b.Cout : const_cast<float*>(b.Cin);
#pragma unroll
    for (int k = 0; k < S::P; ++k) fo[(long long)k * N + i] = pop_put<PT>(cluster_ld(at(own, fl + k)));
    float d[NCOMP];
#pragma unroll
    for (int s = 0; s < NCOMP; ++s) {
        b.frest[s * N + i] = rest[s];
        d[s] = cluster_ld(at(own, S::D + s));
    }
    dens_store<NCOMP>(b.drho, i, d);
#pragma unroll
    for (int k = 0; k < 2; ++k) b.u[k * N + i] = cluster_ld(at(own, S::U + k));
    if (p.feedback != 0.0f) {
#pragma unroll
        for (int k = 0; k < L::NQ; ++k) b.Q[k * N + i] = cluster_ld(at(own, S::Q + k));
    }
    if (FD) {
#pragma unroll
        for (int k = 0; k < L::NC; ++k) {
            Co[k * N + i] = cluster_ld(at(own, cl + k));
            b.R[k * N + i] = R[k];
        }
    }
}

// Prepares the kernel on the current device; whether it takes the cluster there.
template <class K>
bool small_cluster(K kernel, int smem_max) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max) != cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kSmallBlocks;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(kSmallBlocks);
    cfg.blockDim = dim3(kSmallMaxThreads);
    cfg.dynamicSmemBytes = smem_max;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n > 0;
}

template <class PT, int NCOMP, int COLL, bool FD>
cudaError_t small_steps(const StepParams& p, const StepBufs& b, int nsteps, cudaStream_t s) {
    constexpr int node_bytes = SmallPlanes<NCOMP>::total * (int)sizeof(float);
    constexpr int blocks = kSmallBlocks;
    static PerDevice site;
    int takes = 0;  // 1 the device takes the cluster, 2 it does not
    const cudaError_t e = site.get(&takes, [&](int* v) {
        *v = small_cluster(k_small<PT, NCOMP, COLL, FD>, node_bytes * kSmallMaxThreads) ? 1 : 2;
        return cudaSuccess;
    });
    if (e != cudaSuccess) return e;
    if (takes != 1) return cudaErrorNotSupported;
    const int m = (((int)p.N + blocks - 1) / blocks + 31) / 32 * 32;
    if (m > kSmallMaxThreads) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = blocks;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(m);
    cfg.dynamicSmemBytes = (size_t)node_bytes * m;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_small<PT, NCOMP, COLL, FD>, b, p, nsteps);
}

template <class PT, int NCOMP>
cudaError_t small_dispatch(bool fd, const StepParams& p, const StepBufs& b, int nsteps, cudaStream_t s) {
    if (p.collision == 1)
        return fd ? small_steps<PT, NCOMP, 1, true>(p, b, nsteps, s) : small_steps<PT, NCOMP, 1, false>(p, b, nsteps, s);
    return fd ? small_steps<PT, NCOMP, 0, true>(p, b, nsteps, s) : small_steps<PT, NCOMP, 0, false>(p, b, nsteps, s);
}

}  // namespace

cudaError_t launch_small(int ncomp, bool fd, const StepParams& p, const StepBufs& b, int nsteps, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    VEFD_WITH_PT(p.prec, {
        e = ncomp == 2 ? small_dispatch<PT, 2>(fd, p, b, nsteps, s) : small_dispatch<PT, 1>(fd, p, b, nsteps, s);
    });
    return e;
}

}  // namespace vefd

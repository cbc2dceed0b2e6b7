// Finite-difference FENE-P update of the conformation tensor (Eq. FENE of
// Gupta, Sbragaglia & Scagliarini, with the artificial diffusivity and the
// time integration described at the end of Sec. 2):
//   R = -(u.grad)C + C.grad u + (grad u)^T.C - (f(r_P) C - I)/tau_P + kappa lap C,
//   (grad u)_ij = d_i u_j, f(r_P) = (L^2 - 3)/(L^2 - tr C),
//   C^{n+1} = C^n + 3/2 R^n - 1/2 R^{n-1}   (forward Euler without history).
// Second-order central differences, periodic in x and z; at walls the ghost
// row is the linear extrapolation v(-1) = 2 v(0) - v(1), which makes the
// first derivative one-sided and the second derivative vanish.
// Stored variable: Ct = C - I, so (f C - I) = f Ct + (f - 1) I with
// f - 1 = tr Ct / (L^2 - 3 - tr Ct), evaluated without cancellation.
// Optionally (StepParams::chol) the AB2 step advances the log-Cholesky factor
// of sigma_P = f C instead of C (the Cholesky scheme of Sec. 2).
// The update runs in the same pass as the densities of the new populations
// (k_post), since both only wait for the lattice kernel.
#include <cuda.h>

#include "fd_impl.cuh"

namespace vefd {

namespace {

__device__ __forceinline__ int wrap1(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// One FENE-P update at node (x, y, z) with its stencil read from global
// memory; writes C - I of the next time level and the new history.
template <int D, int NC>
__device__ __forceinline__ void fenep_node(const float* __restrict__ Ct, float* __restrict__ Cout,
                                           float* __restrict__ R, const float* __restrict__ u,
                                           unsigned* __restrict__ status, const StepParams& p, int x, int y, int z,
                                           float cnew[NC]) {
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const long long N = p.N;
    const long long i = ((long long)z * ny + y) * nx + x;
    long long idx[7];
    idx[0] = i;
    idx[1] = i - x + wrap1(x - 1, nx);
    idx[2] = i - x + wrap1(x + 1, nx);
    float hy1 = 0.5f, hy2 = 1.0f;
    if (p.walls && y == 0) {
        idx[3] = i;
        idx[4] = i + nx;
        hy1 = 1.0f;
        hy2 = 0.0f;
    } else if (p.walls && y == ny - 1) {
        idx[3] = i - nx;
        idx[4] = i;
        hy1 = 1.0f;
        hy2 = 0.0f;
    } else {
        idx[3] = ((long long)z * ny + wrap1(y - 1, ny)) * nx + x;
        idx[4] = ((long long)z * ny + wrap1(y + 1, ny)) * nx + x;
    }
    idx[5] = idx[6] = i;
    if (D == 3) {
        idx[5] = ((long long)wrap1(z - 1, nz) * ny + y) * nx + x;
        idx[6] = ((long long)wrap1(z + 1, nz) * ny + y) * nx + x;
    }
    auto v = [&](int k, int d) -> float {
        const float* base = k < NC ? Ct + k * N : u + (k - NC) * N;
        return idx_ok(idx[d], N, status) ? __ldg(base + idx[d]) : 0.0f;
    };
    float Rprev[NC], Rnew[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) Rprev[k] = p.have_prev ? R[k * N + i] : 0.0f;
    const unsigned bits = fenep_compute<D, NC>(v, hy1, hy2, Rprev, p, cnew, Rnew);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        Cout[k * N + i] = cnew[k];
        R[k * N + i] = Rnew[k];
    }
    if (bits) atomicOr(status, bits);
}

// After the lattice kernel of step n: densities of the new populations
// (same summation order as the moments kernel), the FENE-P update of C from
// time n to n+1 when the polymer is evolved, and the feedback stress of time
// n+1 for the next lattice step.  All of it only reads data the lattice kernel
// has finished writing, so one pass over the lattice does it.
// One thread per node over runs of 128 consecutive nodes (x fastest), so no lane
// is spent on the padding of a box; stencil neighbours come from L1 and L2.
// Bound by the latency of its 107 loads a node: five blocks per SM (102
// registers) measure 25.1 us on 100 x 50 x 70 FP32 against 28.8 without the
// bound, 26.1 with 6 and 28.5 with 8.  32 x 4 x 2 boxes with the populations
// staged by a tensor copy, which the run form replaced, took 33.1 us there, 20.6
// against 18.1 on 88 x 48 x 64 and 19.4 against 16.8 on 64^3.
constexpr int kPostBlocks = 5;

template <class PT, class L, int NCOMP, bool FD>
__global__ void __launch_bounds__(128, kPostBlocks) k_post(const PT* __restrict__ fnew, const float* __restrict__ frest,
                                              float* __restrict__ drho,
                                              const float* __restrict__ Ct, float* __restrict__ Cout,
                                              float* __restrict__ R, const float* __restrict__ u,
                                              float* __restrict__ Q, unsigned* __restrict__ status, StepParams p,
                                              int rev) {
    // everything below reads or overwrites data of the preceding lattice kernel
    pdl_wait();
    const long long N = p.N;
    const int i = (rev ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x) * 128 + threadIdx.x;
    if (i >= N) return;
    const int row = (int)((unsigned)i / (unsigned)p.nx), x = i - row * p.nx;
    const int z = (int)((unsigned)row / (unsigned)p.ny), y = row - z * p.ny;
    float d[NCOMP];
#pragma unroll
    for (int s = 0; s < NCOMP; ++s) {
        d[s] = __ldg(frest + s * N + i);
#pragma unroll
        for (int a = 1; a < L::Q; ++a) d[s] += pop_load(fnew + (s * (L::Q - 1) + a - 1) * N + i);
    }
    float c[L::NC];
    if (FD) {
        fenep_node<L::D, L::NC>(Ct, Cout, R, u, status, p, x, y, z, c);
    } else {
#pragma unroll
        for (int k = 0; k < L::NC; ++k) c[k] = __ldg(Ct + k * N + i);
    }
    pdl_trigger();
    dens_store<NCOMP>(drho, i, d);
    if (p.feedback != 0.0f) store_feedback<L, NCOMP>(c, d, p, Q, N, i);
}

// D3Q19 variant of the pass that marches along z through a column of
// 32 x 8 nodes.  C - I and u of four consecutive planes (with a one-node halo
// in x and y) live in a shared-memory ring, so every stencil value is read
// from global memory about 1.3 times instead of 7; each plane's new
// populations arrive by one bulk tensor copy (box 32 x 8 x 1 x P) that
// overlaps the stencil arithmetic.  Needs NX % 32 == 0 and NY % 8 == 0.
constexpr int kZmBX = 32, kZmBY = 8, kZmHX = kZmBX + 2, kZmHY = kZmBY + 2, kZmNF = 9;
constexpr int kZmPlane = kZmNF * kZmHY * kZmHX;  // floats per ring plane

template <class PT, int NCOMP>
constexpr int zm_smem_bytes() {
    return NCOMP * 18 * kZmBX * kZmBY * (int)sizeof(PT) + 4 * kZmPlane * (int)sizeof(float);
}

// MODE 0: the densities of the new populations, staged plane by plane.
// MODE 1 (FUSED): after the column-marching lattice kernel.  drho then holds
// each node's partial density (the rest population and every population that
// arrived from inside its 32 x 8 column and lattice-kernel z-segment of
// length zl); the pass adds, from fnew, the populations that crossed a column
// side or a segment end, in direction order, and needs no population copy.
// MODE 2 (PARTS): after the staged lattice kernel with partial densities
// (tile_partials): each node's density is its slot-0 sum plus, in slot
// order, the slots its position in its lattice tile (32 x part_by x part_bz)
// implies; no population is read.
// One 32 x 8 column (origin x0, y0) over the planes [z0, z0 + zs) of the
// pass; tm_fnew is the tensor map of the new populations (box 32 x 8 x 1 x P).
template <class PT, int NCOMP, bool FD, int MODE>
__device__ __forceinline__ void post_column(const CUtensorMap* tm_fnew, const float* __restrict__ frest,
                                            float* __restrict__ drho, const float* __restrict__ Ct,
                                            float* __restrict__ Cout, float* __restrict__ R,
                                            const float* __restrict__ u, float* __restrict__ Q,
                                            unsigned* __restrict__ status, const StepParams& p, int x0, int y0, int z0,
                                            int zs, const PT* __restrict__ fnew, int zl,
                                            const float* __restrict__ part = nullptr, int part_by = 1,
                                            int part_bz = 1) {
    constexpr bool FUSED = MODE == 1, PARTS = MODE == 2;
    using L = D3Q19;
    constexpr int P = NCOMP * (L::Q - 1);  // moving populations
    constexpr int T = kZmBX * kZmBY;
    constexpr unsigned kBytes = (unsigned)(P * T * sizeof(PT));
    extern __shared__ __align__(128) unsigned char sraw[];
    PT* sP = reinterpret_cast<PT*>(sraw);  // [P][BY][BX] populations of the current plane (MODE 0)
    float* ring = reinterpret_cast<float*>(sraw + (MODE != 0 ? 0 : P * T * sizeof(PT)));  // [4][NF][HY][HX]
    __shared__ __align__(8) unsigned long long bar;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int N = (int)p.N, plane = nx * ny;
    const int z1 = min(z0 + zs, nz);
    const int x = x0 + tx, y = y0 + ty;
    const bool leader = (tx | ty) == 0;
    const unsigned bar_a = smem_u32(&bar);
    if (leader) mbar_init(bar_a);
    // everything below reads or overwrites data of the preceding lattice kernel
    pdl_wait();

    // which ring cells this thread stages: its own (interior) cell and, for
    // some warps, one halo cell (rows y0-1 / y0+8, columns x0-1 / x0+32)
    int hr = -1, hc = -1;
    if (ty == 0) {
        hr = 0;
        hc = tx + 1;
    } else if (ty == kZmBY - 1) {
        hr = kZmHY - 1;
        hc = tx + 1;
    } else if (ty == 1 && tx < 2 * kZmHY) {
        hr = tx % kZmHY;
        hc = tx < kZmHY ? 0 : kZmHX - 1;
    }
    int hx = 0, hyg = 0;
    bool hvalid = false;
    if (hr >= 0) {
        hx = wrap1(x0 - 1 + hc, nx);
        const int yy = y0 - 1 + hr;
        if (p.walls) {
            hvalid = yy >= 0 && yy < ny;  // ghost rows beyond walls are never read
            hyg = yy;
        } else {
            hvalid = true;
            hyg = wrap1(yy, ny);
        }
    }
    auto load_plane = [&](int zp, float v_in[kZmNF], float v_h[kZmNF]) {
        const int zz = wrap1(zp, nz);
        const int gi = zz * plane + y * nx + x;
        const int gh = zz * plane + hyg * nx + hx;
#pragma unroll
        const bool ok_i = idx_ok(gi, N, status), ok_h = hvalid && idx_ok(gh, N, status);
        for (int k = 0; k < kZmNF; ++k) {
            const float* base = k < 6 ? Ct + k * N : u + (k - 6) * N;
            v_in[k] = ok_i ? __ldg(base + gi) : 0.0f;
            if (hvalid) v_h[k] = ok_h ? __ldg(base + gh) : 0.0f;
        }
    };
    auto store_plane = [&](int slot, const float v_in[kZmNF], const float v_h[kZmNF]) {
        float* rp = ring + slot * kZmPlane;
#pragma unroll
        for (int k = 0; k < kZmNF; ++k) {
            rp[(k * kZmHY + ty + 1) * kZmHX + tx + 1] = v_in[k];
            if (hvalid) rp[(k * kZmHY + hr) * kZmHX + hc] = v_h[k];
        }
    };
    float vi[kZmNF], vh[kZmNF];
    // prologue: planes z0-1, z0, z0+1 into slots 0, 1, 2
    for (int q = 0; q < 3; ++q) {
        load_plane(z0 - 1 + q, vi, vh);
        store_plane(q, vi, vh);
    }
    __syncthreads();

    const bool wall_lo = p.walls && y == 0, wall_hi = p.walls && y == ny - 1;
    const float hy1 = (wall_lo || wall_hi) ? 1.0f : 0.5f;
    const float hy2 = (wall_lo || wall_hi) ? 0.0f : 1.0f;
    const int ry = ty + 1, rc = tx + 1;
    const int rym = wall_lo ? ry : ry - 1, ryp = wall_hi ? ry : ry + 1;
    const int t = ty * kZmBX + tx;

    const ColumnTopo topo{nx == 32, ny == 8 && !p.walls, nz == 1};
    for (int k = 0; k < z1 - z0; ++k) {
        const int z = z0 + k;
        // the next step's lattice kernel may be scheduled once every block is on its last plane
        if (k == z1 - z0 - 1) pdl_trigger();
        // new populations of this plane: one bulk copy (the buffer was released
        // by every thread at the barrier ending the previous iteration)
        if (MODE == 0 && leader) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tma_load_4d(smem_u32(sP), tm_fnew, x0, y0, z, 0, bar_a, kBytes);
        }
        // stage plane z+2 while this plane is computed
        const bool more = z + 2 <= z1;
        if (more) load_plane(z + 2, vi, vh);
        const int i = z * plane + y * nx + x;
        float rest[NCOMP];
        if (FUSED) {
            // partial density plus what crossed a column side or a segment end
            const bool wlo = p.walls && y == 0, whi = p.walls && y == ny - 1;
            const int zs_lo = (z / zl) * zl, zs_hi = min(zs_lo + zl, nz);  // this plane's lattice-kernel segment
            float part[NCOMP];
            dens_get<NCOMP>(drho, i, part);
#pragma unroll
            for (int s = 0; s < NCOMP; ++s) {
                float d = part[s];
#pragma unroll
                for (int a = 1; a < L::Q; ++a) {
                    const int cx = L::cx(a), cy = L::cy(a), cz = L::cz(a);
                    if ((cy > 0 && wlo) || (cy < 0 && whi)) continue;  // bounce-back: counted in the partial
                    const int zsrc = z - cz;
                    const bool same_seg = topo.nz1 || (zsrc >= zs_lo && zsrc < zs_hi);
                    const bool same_col = (topo.nx32 || (unsigned)(tx - cx) < 32u) && (topo.ny8p || (unsigned)(ty - cy) < 8u);
                    if (same_seg && same_col) continue;
                    d += pop_get(fnew[(s * (L::Q - 1) + a - 1) * N + i]);
                }
                rest[s] = d;
            }
        } else if (PARTS) {
            // slot 0, then the neighbouring tiles' pushes (x, y, z, xy, xz, yz)
            const int ly = y % part_by, lz = z % part_bz;
            const bool xe = tx == 0 || tx == kZmBX - 1;
            const bool ye = (ly == 0 && (y > 0 || !p.walls)) || (ly == part_by - 1 && (y < ny - 1 || !p.walls));
            const bool ze = lz == 0 || lz == part_bz - 1;
            const bool use[7] = {true, xe, ye, ze, xe && ye, xe && ze, ye && ze};
#pragma unroll
            for (int s = 0; s < NCOMP; ++s) rest[s] = 0.0f;
#pragma unroll
            for (int q = 0; q < 7; ++q) {
                if (!use[q]) continue;
                float w[NCOMP] = {};
                if (idx_ok(i, N, status)) dens_ldg<NCOMP>(part + (long long)q * N * NCOMP, i, w);
#pragma unroll
                for (int s = 0; s < NCOMP; ++s) rest[s] = q == 0 ? w[s] : rest[s] + w[s];
            }
        } else {
#pragma unroll
            for (int s = 0; s < NCOMP; ++s) rest[s] = __ldg(frest + s * N + i);
        }
        float c[6];
        if (FD) {
            const float* pm = ring + (k % 4) * kZmPlane;
            const float* pc = ring + ((k + 1) % 4) * kZmPlane;
            const float* pp = ring + ((k + 2) % 4) * kZmPlane;
            auto v = [&](int f, int d) -> float {
                const int o = f * kZmHY * kZmHX;
                switch (d) {
                case 0: return pc[o + ry * kZmHX + rc];
                case 1: return pc[o + ry * kZmHX + rc - 1];
                case 2: return pc[o + ry * kZmHX + rc + 1];
                case 3: return pc[o + rym * kZmHX + rc];
                case 4: return pc[o + ryp * kZmHX + rc];
                case 5: return pm[o + ry * kZmHX + rc];
                default: return pp[o + ry * kZmHX + rc];
                }
            };
            float Rprev[6], Rnew[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) Rprev[q] = p.have_prev ? R[q * N + i] : 0.0f;
            const unsigned bits = fenep_compute<3, 6>(v, hy1, hy2, Rprev, p, c, Rnew);
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                Cout[q * N + i] = c[q];
                R[q * N + i] = Rnew[q];
            }
            if (bits) atomicOr(status, bits);
        } else {
            const float* pc = ring + ((k + 1) % 4) * kZmPlane;
#pragma unroll
            for (int q = 0; q < 6; ++q) c[q] = pc[(q * kZmHY + ry) * kZmHX + rc];
        }
        // densities of the new populations (same summation order as elsewhere)
        float d[NCOMP];
        if (FUSED || PARTS) {
#pragma unroll
            for (int s = 0; s < NCOMP; ++s) d[s] = rest[s];
            dens_store<NCOMP>(drho, i, d);
        } else {
            const bool ok = mbar_wait_bounded_parity(bar_a, (unsigned)(k & 1));
            if (__syncthreads_or(!ok)) {
                if (leader) {
                    atomicOr(status, kStTimeout);
                    mbar_wait_bounded_parity(bar_a, (unsigned)(k & 1));  // bounded: let the copy land
                }
                return;
            }
#pragma unroll
            for (int s = 0; s < NCOMP; ++s) {
                d[s] = rest[s];
#pragma unroll
                for (int a = 1; a < L::Q; ++a) d[s] += pop_get(sP[(s * (L::Q - 1) + a - 1) * T + t]);
            }
            dens_store<NCOMP>(drho, i, d);
        }
        if (p.feedback != 0.0f) store_feedback<L, NCOMP>(c, d, p, Q, N, i);
        if (more) store_plane((k + 3) % 4, vi, vh);
        __syncthreads();
    }
}

template <class PT, int NCOMP, bool FD, int MODE>
__global__ void __launch_bounds__(kZmBX * kZmBY, 2) k_post_zm(const __grid_constant__ CUtensorMap tm_fnew,
                                                               const float* __restrict__ frest,
                                                               float* __restrict__ drho, const float* __restrict__ Ct,
                                                               float* __restrict__ Cout, float* __restrict__ R,
                                                               const float* __restrict__ u, float* __restrict__ Q,
                                                               unsigned* __restrict__ status, StepParams p, int zs,
                                                               int rev, const PT* __restrict__ fnew, int zl,
                                                               const float* __restrict__ part, int part_by,
                                                               int part_bz) {
    const int x0 = (rev ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x) * kZmBX;
    const int y0 = p.ylo + (rev ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y) * kZmBY;
    const int z0 = (rev ? (int)(gridDim.z - 1 - blockIdx.z) : (int)blockIdx.z) * zs;
    post_column<PT, NCOMP, FD, MODE>(&tm_fnew, frest, drho, Ct, Cout, R, u, Q, status, p, x0, y0, z0, zs, fnew, zl,
                                     part, part_by, part_bz);
}

// Batched ensemble form: block i (taken in reverse order, so the pass starts on
// the tiles the lattice kernel touched last) runs column item i - start[m] of
// member m: columns x-fastest, then y, then z-segments of the member's zs planes.
template <class PT, int NCOMP, bool FD>
__global__ void __launch_bounds__(kZmBX * kZmBY, 2)
    k_post_batch(const EnsMember* __restrict__ members, const int* __restrict__ start, int nm, int parity) {
    const int item = (int)(gridDim.x - 1 - blockIdx.x);
    const int m = batch_member(start, nm, item);
    const EnsMember& M = members[m];
    const int t = item - start[m];
    const StepParams p = M.p;
    const StepBufs b = M.b[parity];
    const int r = t / M.ncx;
    const CUtensorMap* tm = &M.tm_post[1 - (M.cur0 ^ parity)];      // the populations just written
    if ((threadIdx.x | threadIdx.y) == 0) tensormap_acquire(tm);  // the thread that issues the copies
    post_column<PT, NCOMP, FD, 0>(tm, b.frest, b.drho, b.Cin, b.Cout, b.R, b.u, b.Q, b.status, p,
                                      (t % M.ncx) * kZmBX, (r % M.ncy) * kZmBY, (r / M.ncy) * M.zs, M.zs,
                                      static_cast<const PT*>(b.fout), 1);
}

// Densities and feedback stress of a given state (no time step).
template <class PT, class L, int NCOMP>
__global__ void __launch_bounds__(128) k_pre(const PT* __restrict__ f, const float* __restrict__ frest,
                                             float* __restrict__ drho,
                                             const float* __restrict__ Ct, float* __restrict__ Q, StepParams p) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= p.nx || y >= p.ny) return;
    const long long N = p.N;
    const long long i = ((long long)z * p.ny + y) * p.nx + x;
    float d[NCOMP];
#pragma unroll
    for (int s = 0; s < NCOMP; ++s) {
        d[s] = __ldg(frest + s * N + i);
#pragma unroll
        for (int a = 1; a < L::Q; ++a) d[s] += pop_load(f + (s * (L::Q - 1) + a - 1) * N + i);
    }
    dens_store<NCOMP>(drho, i, d);
    float c[L::NC];
#pragma unroll
    for (int k = 0; k < L::NC; ++k) c[k] = __ldg(Ct + k * N + i);
    if (p.feedback != 0.0f) store_feedback<L, NCOMP>(c, d, p, Q, N, i);
}

}  // namespace

cudaError_t launch_post(int lattice, int ncomp, bool fd, const StepParams& p, const StepBufs& b,
                        const void* fnew, cudaStream_t s, int rev) {
    const dim3 blk(128), grd((unsigned)((p.N + 127) / 128));
    cudaError_t e = cudaSuccess;
#define VEFD_POST(LT, NCP)                                                                                  \
    do {                                                                                                    \
        const PT* fn = static_cast<const PT*>(fnew);                                                        \
        e = launch_pdl(p.pdl != 0, fd ? k_post<PT, LT, NCP, true> : k_post<PT, LT, NCP, false>, grd, blk, 0, s, fn, \
                       (const float*)b.frest, b.drho, b.Cin, b.Cout, b.R, (const float*)b.u, b.Q, b.status, p, rev); \
    } while (0)
    VEFD_WITH_PT(p.prec, {
        if (lattice == 1) {
            if (ncomp == 2) VEFD_POST(D3Q19, 2);
            else VEFD_POST(D3Q19, 1);
        } else {
            if (ncomp == 2) VEFD_POST(D2Q9, 2);
            else VEFD_POST(D2Q9, 1);
        }
    });
#undef VEFD_POST
    return e;
}

bool post_zm_eligible(int lattice, int nx, int ny) { return lattice == 1 && nx % kZmBX == 0 && ny % kZmBY == 0; }

namespace {
int g_sm_count = 0;

template <class PT, int NCOMP, bool FD, int MODE>
cudaError_t post_zm(const CUtensorMap* tm, const StepParams& p, const StepBufs& b, cudaStream_t s, int rev, int zl,
                    Parts parts = Parts{}) {
    constexpr bool FUSED = MODE == 1;
    constexpr int smem = MODE != 0 ? 4 * kZmPlane * (int)sizeof(float) : zm_smem_bytes<PT, NCOMP>();
    static PerDevice site;
    const cudaError_t e = allow_smem(site, k_post_zm<PT, NCOMP, FD, MODE>, smem);
    if (e != cudaSuccess) return e;
    if (!g_sm_count) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&g_sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) g_sm_count = 152;
    }
    // one wave: split z so that the columns x z-segments fill two blocks per SM
    const int bxy = (p.nx / kZmBX) * (p.ny / kZmBY);
    int nzb = (2 * g_sm_count) / bxy;
    if (nzb < 1) nzb = 1;
    if (nzb > p.nz) nzb = p.nz;
    const int zs = p.post_zs > 0 ? (p.post_zs < p.nz ? p.post_zs : p.nz) : (p.nz + nzb - 1) / nzb;
    nzb = (p.nz + zs - 1) / zs;
    dim3 blk(kZmBX, kZmBY, 1), grd(p.nx / kZmBX, (p.yhi - p.ylo) / kZmBY, nzb);
    // FUSED reads the partial densities of the new time level and completes them in place
    float* dens = FUSED ? b.drho_next : b.drho;
    const CUtensorMap dummy{};
    return launch_pdl(p.pdl != 0, k_post_zm<PT, NCOMP, FD, MODE>, grd, blk, smem, s, MODE != 0 ? dummy : *tm,
                      (const float*)b.frest, dens, (const float*)b.Cin, b.Cout, b.R, (const float*)b.u, b.Q, b.status,
                      p, zs, rev, static_cast<const PT*>(b.fout), zl, (const float*)parts.part, parts.by, parts.bz);
}
}  // namespace

cudaError_t launch_post_zm(int ncomp, bool fd, const StepParams& p, const StepBufs& b, const void* tensor_map_fnew,
                           cudaStream_t s, int rev, Parts parts) {
    const CUtensorMap* tm = static_cast<const CUtensorMap*>(tensor_map_fnew);
    cudaError_t e = cudaSuccess;
    if (parts.part && (parts.by < 2 || parts.bz < 2)) return cudaErrorInvalidValue;
    VEFD_WITH_PT(p.prec, {
        if (parts.part) {
            if (ncomp == 2)
                e = fd ? post_zm<PT, 2, true, 2>(tm, p, b, s, rev, 1, parts)
                       : post_zm<PT, 2, false, 2>(tm, p, b, s, rev, 1, parts);
            else
                e = fd ? post_zm<PT, 1, true, 2>(tm, p, b, s, rev, 1, parts)
                       : post_zm<PT, 1, false, 2>(tm, p, b, s, rev, 1, parts);
        } else if (ncomp == 2) {
            e = fd ? post_zm<PT, 2, true, 0>(tm, p, b, s, rev, 1) : post_zm<PT, 2, false, 0>(tm, p, b, s, rev, 1);
        } else {
            e = fd ? post_zm<PT, 1, true, 0>(tm, p, b, s, rev, 1) : post_zm<PT, 1, false, 0>(tm, p, b, s, rev, 1);
        }
    });
    return e;
}

cudaError_t launch_post_zm_fused(int ncomp, bool fd, const StepParams& p, const StepBufs& b, cudaStream_t s, int zs,
                                 int rev) {
    cudaError_t e = cudaSuccess;
    VEFD_WITH_PT(p.prec, {
        if (ncomp == 2)
            e = fd ? post_zm<PT, 2, true, 1>(nullptr, p, b, s, rev, zs) : post_zm<PT, 2, false, 1>(nullptr, p, b, s, rev, zs);
        else
            e = fd ? post_zm<PT, 1, true, 1>(nullptr, p, b, s, rev, zs) : post_zm<PT, 1, false, 1>(nullptr, p, b, s, rev, zs);
    });
    return e;
}

namespace {
template <class PT, int NCOMP, bool FD>
cudaError_t post_batch(const EnsMember* members, const int* start, int nm, int items, int parity, bool pdl,
                       cudaStream_t s) {
    constexpr int smem = zm_smem_bytes<PT, NCOMP>();
    static PerDevice site;
    const cudaError_t e = allow_smem(site, k_post_batch<PT, NCOMP, FD>, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(pdl, k_post_batch<PT, NCOMP, FD>, dim3(items), dim3(kZmBX, kZmBY, 1), smem, s, members, start,
                      nm, parity);
}
}  // namespace

cudaError_t launch_post_batch(int ncomp, int prec, bool fd, const EnsMember* members, const int* start, int nm,
                              int items, int parity, bool pdl, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    VEFD_WITH_PT(prec, {
        if (ncomp == 2)
            e = fd ? post_batch<PT, 2, true>(members, start, nm, items, parity, pdl, s)
                   : post_batch<PT, 2, false>(members, start, nm, items, parity, pdl, s);
        else
            e = fd ? post_batch<PT, 1, true>(members, start, nm, items, parity, pdl, s)
                   : post_batch<PT, 1, false>(members, start, nm, items, parity, pdl, s);
    });
    return e;
}

cudaError_t launch_pre(int lattice, int ncomp, const StepParams& p, const StepBufs& b, cudaStream_t s) {
    dim3 blk(32, 4, 1), grd((p.nx + 31) / 32, (p.ny + 3) / 4, p.nz);
    VEFD_WITH_PT(p.prec, {
        const PT* f = static_cast<const PT*>(b.fin);
        if (lattice == 1) {
            if (ncomp == 2) k_pre<PT, D3Q19, 2><<<grd, blk, 0, s>>>(f, b.frest, b.drho, b.Cin, b.Q, p);
            else k_pre<PT, D3Q19, 1><<<grd, blk, 0, s>>>(f, b.frest, b.drho, b.Cin, b.Q, p);
        } else {
            if (ncomp == 2) k_pre<PT, D2Q9, 2><<<grd, blk, 0, s>>>(f, b.frest, b.drho, b.Cin, b.Q, p);
            else k_pre<PT, D2Q9, 1><<<grd, blk, 0, s>>>(f, b.frest, b.drho, b.Cin, b.Q, p);
        }
    });
    return cudaGetLastError();
}

}  // namespace vefd

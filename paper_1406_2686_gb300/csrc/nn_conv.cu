// 3x3x3 convolution layers of the warm-start network as implicit GEMMs on the
// tcgen05 tensor cores (channels-last activations, zero padding 1, stride 1 or 2).
//
// The BF16 copy of the activations, xb[voxel][Cp] (Cp = channels rounded up to
// 8), is all that is gathered: a column (tap, 8 channels) of the im2col matrix
// is one 16-byte piece of a neighbouring voxel, so the producer threads build
// the operand tiles in shared memory directly and no im2col matrix, no
// gradient columns and no transposed copies exist in memory.
//   k_conv      rows = voxels, K = (tap, channel), N = output channels, with
//               bias and ReLU in the epilogue: the forward pass, and with the
//               gradient as input the backward-data pass (for stride 2 the rows
//               are grouped by the parity of their coordinates, so that each
//               128-row tile has one short list of contributing taps);
//   k_conv_dw   dW^T[(tap, channel)][o] = sum over voxels, both operands
//               MN-major so that the gathered rows are used as they lie.
// Both run a ring of shared-memory stages between 128 producer threads
// (cp.async, zero fill at the borders) and one thread that issues the matrix
// operations; accumulation over K runs tap by tap, 16 columns at a time.
// What bounds them: the gather's L2/L1 traffic, 27 reads of each activation.
// Measured against explicit im2col matrices (scalar kernels writing [V][27 C]
// and its transpose, GEMMs over them, FP32 gradient columns folded back):
// 48 -> 16 channels at 64^3, forward and backward, 6747 -> 449 us; the whole
// network's prediction at 64^3 12263 -> 1096 us, the same bits (the order of
// the sums over K is the GEMM's).
#include <algorithm>

#include "nn_tc.cuh"
#include "vefd_nn.h"

namespace vefd_nn {
namespace {

constexpr int kRows = 128;     // rows of a tile (tcgen05 M)
constexpr int kSlabs = 8;      // 16-byte pieces (8 channels) of a K chunk: K = 64
constexpr int kLag = 3;        // chunks a producer keeps in flight before announcing the oldest
constexpr int kMaxStages = 8;
constexpr int kTaps = 27;

// Rows and gathered neighbours of one pass.  Class c (one class, or eight
// parity classes) covers a sub-grid rz x ry x rx of row voxels; its row (z, y,
// x) sits at gathered voxel (z, y, x) * scale and reads the entries
// [cbeg[c], cbeg[c + 1]): tap id[], voxel offset off[] from that centre.
struct Gather {
    int B, D, H, W, C8;            // gathered grid, 16-byte pieces per voxel
    int Dr, Hr, Wr;                // row grid (the output's layout)
    int scale, ncls;               // gathered centre = row * scale (one class) or the sub-grid index (parity classes)
    int cbeg[9], tile0[9];
    int rz[8], ry[8], rx[8];
    int off[kTaps], id[kTaps];
    unsigned neg[8][3], pos[8][3];  // entries of a class that step below / above the centre along z, y, x
};

struct Row {
    bool ok;
    long long out;   // row voxel in the output grid
    long long base;  // gathered centre voxel * C8
    unsigned mask;   // entries inside the gathered grid
};

__device__ __forceinline__ Row row_of(const Gather& g, int cls, int mt, int r) {
    Row w;
    const int rx = g.rx[cls], ry = g.ry[cls], rz = g.rz[cls];
    unsigned m = (unsigned)(mt - g.tile0[cls]) * kRows + r;
    w.ok = m < (unsigned)(g.B * rz * ry * rx);
    if (!w.ok) m = 0;
    const unsigned x = m % rx, q = m / rx;
    const unsigned y = q % ry, p = q / ry;
    const unsigned z = p % rz, b = p / rz;
    const bool par = g.ncls > 1;
    const int gz = z * g.scale, gy = y * g.scale, gx = x * g.scale;
    const int oz = par ? 2 * z + (cls >> 2) : z, oy = par ? 2 * y + ((cls >> 1) & 1) : y, ox = par ? 2 * x + (cls & 1) : x;
    w.out = (((long long)b * g.Dr + oz) * g.Hr + oy) * g.Wr + ox;
    w.base = ((((long long)b * g.D + gz) * g.H + gy) * g.W + gx) * g.C8;
    unsigned bad = 0;
    if (gz == 0) bad |= g.neg[cls][0];
    if (gz + 1 >= g.D) bad |= g.pos[cls][0];
    if (gy == 0) bad |= g.neg[cls][1];
    if (gy + 1 >= g.H) bad |= g.pos[cls][1];
    if (gx == 0) bad |= g.neg[cls][2];
    if (gx + 1 >= g.W) bad |= g.pos[cls][2];
    w.mask = w.ok ? ~bad : 0u;
    return w;
}

__device__ __forceinline__ int class_of(const Gather& g, int mt) {
    int c = 0;
    while (c + 1 < g.ncls && mt >= g.tile0[c + 1]) ++c;
    return c;
}

// Y[row][n] = sum over (entry, channel) of the gathered row times Wk, n < N,
// then + bias[n] and max(., 0).  Wk[(tap * C8 + c8)][Np][8] BF16 with one zero
// slab at the end; Np = N rounded up to 16, tiles of bn columns.  Warps 0-3
// gather A (thread = row), 4-7 are the epilogue, 8 issues the matrix
// operations, 9 copies the B slabs.  Shared-memory layout of both operands:
// [slab][row][16 bytes], the no-swizzle K-major core-matrix layout.
constexpr int kConvThreads = 320;

__global__ void __launch_bounds__(kConvThreads)
    k_conv(const uint4* __restrict__ A, const __grid_constant__ Gather g, const uint4* __restrict__ Wk, int Np, int bn,
           int acc_cols, int stages, float* __restrict__ Y, const float* __restrict__ bias, int N, int relu, int vec,
           unsigned* __restrict__ status) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) unsigned long long full[kMaxStages], bfull[kMaxStages], empty[kMaxStages], acc_full[2],
        acc_empty[2];
    __shared__ unsigned tmem_base;
    __shared__ int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned base = smem_addr(dsm);
    const unsigned a_bytes = kSlabs * kRows * 16, stage_bytes = a_bytes + kSlabs * bn * 16;
    const int ntn = (Np + bn - 1) / bn, ntiles = g.tile0[g.ncls] * ntn;
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init_n(smem_addr(&full[s]), 4);
            mbar_init_n(smem_addr(&bfull[s]), 1);
            mbar_init_n(smem_addr(&empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init_n(smem_addr(&acc_full[a]), 1);
            mbar_init_n(smem_addr(&acc_empty[a]), 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    if (warp == 8) tmem_alloc(&tmem_base, 2 * acc_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = tmem_base;
    volatile int* abortp = &abort_flag;
    bool failed = false;

    if (warp < 4) {
        const int r = threadIdx.x;
        int it = 0, s = 0, rel = 0;  // chunk counter, its stage, stage to announce next
        unsigned ph = 0;
        for (int t = blockIdx.x; t < ntiles && !failed; t += gridDim.x) {
            const int mt = t / ntn, cls = class_of(g, mt);
            const Row w = row_of(g, cls, mt, r);
            const int e0 = g.cbeg[cls], nk8 = (g.cbeg[cls + 1] - e0) * g.C8, nk8r = (nk8 + 1) & ~1;
            const uint4* src = A + w.base;
            int ti = 0, c8 = 0;
            const uint4* tap = src + (long long)g.off[e0] * g.C8;
            bool ok = w.mask & 1u;
            for (int q0 = 0; q0 < nk8r; q0 += kSlabs, ++it) {
                if (it >= stages && !mbar_wait(smem_addr(&empty[s]), ph ^ 1u)) failed = true;
                if (__any_sync(0xffffffffu, failed || *abortp)) {
                    failed = true;
                    break;
                }
                const unsigned dst = base + (unsigned)s * stage_bytes + r * 16;
#pragma unroll
                for (int j = 0; j < kSlabs; ++j) {
                    if (q0 + j >= nk8r) break;
                    const bool in = ok && q0 + j < nk8;
                    cp_async16(dst + j * (kRows * 16), in ? tap + c8 : A, in);
                    if (++c8 == g.C8) {
                        c8 = 0;
                        ++ti;
                        if (e0 + ti < g.cbeg[cls + 1]) {
                            tap = src + (long long)g.off[e0 + ti] * g.C8;
                            ok = (w.mask >> ti) & 1u;
                        }
                    }
                }
                cp_async_commit();
                if (it >= kLag) {
                    cp_async_wait<kLag>();
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_addr(&full[rel]));
                    if (++rel == stages) rel = 0;
                }
                if (++s == stages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        }
        cp_async_wait<0>();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (!failed && lane == 0)
            for (int q = it < kLag ? it : kLag; q > 0; --q) {
                mbar_arrive(smem_addr(&full[rel]));
                if (++rel == stages) rel = 0;
            }
        if (failed) *abortp = 1;
    } else if (warp == 9) {
        if (lane == 0) {
            int it = 0, s = 0;
            unsigned ph = 0;
            for (int t = blockIdx.x; t < ntiles && !failed; t += gridDim.x) {
                const int mt = t / ntn, n0 = (t % ntn) * bn, cls = class_of(g, mt);
                const int e0 = g.cbeg[cls], nk8 = (g.cbeg[cls + 1] - e0) * g.C8, nk8r = (nk8 + 1) & ~1;
                const unsigned slab = (unsigned)min(bn, Np - n0) * 16u;
                int ti = 0, c8 = 0;
                for (int q0 = 0; q0 < nk8r; q0 += kSlabs, ++it) {
                    if ((it >= stages && !mbar_wait(smem_addr(&empty[s]), ph ^ 1u)) || *abortp) {
                        failed = true;
                        break;
                    }
                    const unsigned bb = smem_addr(&bfull[s]);
                    const int ns = min(kSlabs, nk8r - q0);
                    mbar_expect(bb, slab * ns);
                    const unsigned dst = base + (unsigned)s * stage_bytes + a_bytes;
                    for (int j = 0; j < ns; ++j) {
                        const int k8 = q0 + j < nk8 ? g.id[e0 + ti] * g.C8 + c8 : kTaps * g.C8;
                        bulk_load(dst + (unsigned)j * bn * 16, Wk + (long long)k8 * Np + n0, slab, bb);
                        if (++c8 == g.C8) {
                            c8 = 0;
                            ++ti;
                        }
                    }
                    if (++s == stages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
            if (failed) *abortp = 1;
            // bounded: the copies in flight (the last `stages` issued) land before the block leaves
            for (int q = it > stages ? it - stages : 0; q < it; ++q)
                mbar_wait(smem_addr(&bfull[q % stages]), (unsigned)((q / stages) & 1));
        }
    } else if (warp == 8) {
        if (lane == 0) {
            int s = 0, j = 0;
            unsigned ph = 0;
            for (int t = blockIdx.x; t < ntiles && !failed; t += gridDim.x, ++j) {
                const int mt = t / ntn, n0 = (t % ntn) * bn, cls = class_of(g, mt);
                const int nk8r = ((g.cbeg[cls + 1] - g.cbeg[cls]) * g.C8 + 1) & ~1;
                const uint32_t idesc = instr_desc(kRows, min(bn, Np - n0));
                const int acc = j & 1;
                if (j >= 2 && !mbar_wait(smem_addr(&acc_empty[acc]), (unsigned)((j / 2 - 1) & 1))) {
                    failed = true;
                    break;
                }
                tc_fence_after();
                const unsigned d = tmem + (unsigned)(acc * acc_cols);
                for (int q0 = 0; q0 < nk8r; q0 += kSlabs) {
                    if (!mbar_wait(smem_addr(&full[s]), ph) || !mbar_wait(smem_addr(&bfull[s]), ph) || *abortp) {
                        failed = true;
                        break;
                    }
                    tc_fence_after();
                    const unsigned sa = base + (unsigned)s * stage_bytes, sb = sa + a_bytes;
                    const int steps = min(kSlabs, nk8r - q0) / 2;
                    for (int k = 0; k < steps; ++k)
                        mma_f16(d, smem_desc(sa + k * 2 * kRows * 16, kRows * 16, 128),
                                smem_desc(sb + (unsigned)k * 2 * bn * 16, bn * 16, 128), idesc, (q0 > 0 || k > 0) ? 1u : 0u);
                    mma_commit(smem_addr(&empty[s]));
                    if (++s == stages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                if (failed) break;
                mma_commit(smem_addr(&acc_full[acc]));
            }
            if (failed) {
                *abortp = 1;
                // bounded: every matrix operation issued has completed before tensor memory is freed
                mma_commit(smem_addr(&acc_full[j & 1]));
                mbar_wait(smem_addr(&acc_full[j & 1]), (unsigned)((j / 2) & 1));
            }
        }
    } else {
        // epilogue: warp 4 + q owns tensor-memory lanes 32 q ... 32 q + 31
        const int q = warp & 3;
        int j = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++j) {
            const int mt = t / ntn, n0 = (t % ntn) * bn, cls = class_of(g, mt), acc = j & 1;
            const Row w = row_of(g, cls, mt, q * 32 + lane);
            const bool ready = mbar_wait(smem_addr(&acc_full[acc]), (unsigned)((j / 2) & 1)) && !*abortp;
            if (!__all_sync(0xffffffffu, ready)) {
                failed = true;
                break;
            }
            tc_fence_after();
            float* y = Y + w.out * N;
            for (int c0 = 0; c0 < bn && n0 + c0 < N; c0 += 16) {
                uint32_t v[16];
                tmem_ld16(tmem + ((unsigned)(q * 32) << 16) + (unsigned)(acc * acc_cols + c0), v);
                if (!w.ok) continue;
                float f[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const int n = n0 + c0 + k;
                    f[k] = __uint_as_float(v[k]);
                    if (bias && n < N) f[k] += __ldg(bias + n);
                    if (relu) f[k] = fmaxf(f[k], 0.0f);
                }
#pragma unroll
                for (int k = 0; k < 16; k += 4) {
                    const int n = n0 + c0 + k;
                    if (vec) {
                        if (n < N) *reinterpret_cast<float4*>(y + n) = make_float4(f[k], f[k + 1], f[k + 2], f[k + 3]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (n + i < N) y[n + i] = f[k + i];
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&acc_empty[acc]));
        }
        if (failed) *abortp = 1;
    }
    __syncwarp();
    if (failed && lane == 0) atomicOr(status, kStatusTimeout);
    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_free(tmem, 2 * acc_cols);
}

// parts[split][k][o] = sum over the split's voxels v of xb[neighbour of v by
// k's tap][k's channels] * gb[v][o], k = tap * 8 C8 + channel (128 of them per
// block), o < Cout (bn per block).  Stage of 64 voxels: A [16 slabs][64][16 B],
// B [bn / 8 slabs][64][16 B]: MN-major core matrices (8 channels contiguous, 8
// voxels 16 bytes apart), so M groups lie a slab (1024 B) and K groups 128 B apart.
constexpr int kDwThreads = 160, kDwVox = 64;

__global__ void __launch_bounds__(kDwThreads)
    k_conv_dw(const uint4* __restrict__ X, const __grid_constant__ Gather g, const uint4* __restrict__ G, int Cout, int bn,
              int acc_cols, int stages, int nchunks, int chunks_per, float* __restrict__ parts,
              unsigned* __restrict__ status) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) unsigned long long full[kMaxStages], empty[kMaxStages], acc_full;
    __shared__ unsigned tmem_base;
    __shared__ int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned base = smem_addr(dsm);
    const unsigned slab_bytes = kDwVox * 16, a_bytes = 16 * slab_bytes, stage_bytes = a_bytes + (bn / 8) * slab_bytes;
    const int C8 = g.C8, K8 = kTaps * C8, O8 = Cout / 8;
    const int mt = blockIdx.x, n0 = blockIdx.y * bn;
    const int ch0 = blockIdx.z * chunks_per, ch1 = min(nchunks, ch0 + chunks_per);
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init_n(smem_addr(&full[s]), 4);
            mbar_init_n(smem_addr(&empty[s]), 1);
        }
        mbar_init_n(smem_addr(&acc_full), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    if (warp == 4) tmem_alloc(&tmem_base, acc_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = tmem_base;
    volatile int* abortp = &abort_flag;
    bool failed = false;
    if (warp < 4) {
        const int r = threadIdx.x & 63, half = threadIdx.x >> 6;
        // this thread's eight columns of A: neighbour offset and tap
        int off[8], tap[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int q = mt * 16 + half * 8 + j;
            tap[j] = q < K8 ? q / C8 : -1;
            off[j] = q < K8 ? g.off[q / C8] * C8 + q % C8 : 0;
        }
        const unsigned nvox = (unsigned)(g.B * g.Dr * g.Hr * g.Wr);
        const int nb = min(bn, Cout - n0) / 8;  // slabs of B (the columns beyond Cout are never read back)
        int it = 0, s = 0, rel = 0;
        unsigned ph = 0;
        for (int ch = ch0; ch < ch1; ++ch, ++it) {
            if (it >= stages && !mbar_wait(smem_addr(&empty[s]), ph ^ 1u)) failed = true;
            if (__any_sync(0xffffffffu, failed || *abortp)) {
                failed = true;
                break;
            }
            const unsigned v = (unsigned)ch * kDwVox + r;
            const bool ok = v < nvox;
            const unsigned m = ok ? v : 0;
            const unsigned x = m % g.Wr, p1 = m / g.Wr;
            const unsigned y = p1 % g.Hr, p2 = p1 / g.Hr;
            const unsigned z = p2 % g.Dr, b = p2 / g.Dr;
            const int gz = z * g.scale, gy = y * g.scale, gx = x * g.scale;
            unsigned bad = ok ? 0u : ~0u;
            if (gz == 0) bad |= g.neg[0][0];
            if (gz + 1 >= g.D) bad |= g.pos[0][0];
            if (gy == 0) bad |= g.neg[0][1];
            if (gy + 1 >= g.H) bad |= g.pos[0][1];
            if (gx == 0) bad |= g.neg[0][2];
            if (gx + 1 >= g.W) bad |= g.pos[0][2];
            const uint4* src = X + ((((long long)b * g.D + gz) * g.H + gy) * g.W + gx) * C8;
            const unsigned dst = base + (unsigned)s * stage_bytes + r * 16;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (tap[j] < 0) continue;  // rows of the product that are never read back
                const bool in = !((bad >> tap[j]) & 1u);
                cp_async16(dst + (unsigned)(half * 8 + j) * slab_bytes, in ? src + off[j] : X, in);
            }
            const uint4* gs = G + (long long)m * O8 + n0 / 8;
            for (int o = half; o < nb; o += 2) cp_async16(dst + a_bytes + (unsigned)o * slab_bytes, gs + o, ok);
            cp_async_commit();
            if (it >= kLag) {
                cp_async_wait<kLag>();
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_addr(&full[rel]));
                if (++rel == stages) rel = 0;
            }
            if (++s == stages) {
                s = 0;
                ph ^= 1u;
            }
        }
        cp_async_wait<0>();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (!failed && lane == 0)
            for (int q = it < kLag ? it : kLag; q > 0; --q) {
                mbar_arrive(smem_addr(&full[rel]));
                if (++rel == stages) rel = 0;
            }
        if (failed) *abortp = 1;
        // epilogue: this warp's tensor-memory lanes
        const bool ready = !failed && mbar_wait(smem_addr(&acc_full), 0u) && !*abortp;
        if (__all_sync(0xffffffffu, ready)) {
            tc_fence_after();
            const int k = mt * 128 + warp * 32 + lane;
            float* out = parts + ((long long)blockIdx.z * (K8 * 8) + k) * Cout;
            for (int c0 = 0; c0 < bn && n0 + c0 < Cout; c0 += 16) {
                uint32_t v[16];
                tmem_ld16(tmem + ((unsigned)(warp * 32) << 16) + (unsigned)c0, v);
                if (k >= K8 * 8) continue;
#pragma unroll
                for (int j = 0; j < 16; j += 4)
                    if (n0 + c0 + j < Cout)
                        *reinterpret_cast<float4*>(out + n0 + c0 + j) =
                            make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]), __uint_as_float(v[j + 2]),
                                        __uint_as_float(v[j + 3]));
            }
        } else {
            failed = true;
            *abortp = 1;
        }
    } else if (lane == 0) {
        const uint32_t idesc = instr_desc_mn(128, bn);
        int s = 0;
        unsigned ph = 0;
        for (int ch = ch0; ch < ch1; ++ch) {
            if (!mbar_wait(smem_addr(&full[s]), ph) || *abortp) {
                failed = true;
                break;
            }
            tc_fence_after();
            const unsigned sa = base + (unsigned)s * stage_bytes, sb = sa + a_bytes;
#pragma unroll
            for (int k = 0; k < kDwVox / 16; ++k)
                mma_f16(tmem, smem_desc(sa + k * 256, 128, slab_bytes), smem_desc(sb + k * 256, 128, slab_bytes), idesc,
                        (ch > ch0 || k > 0) ? 1u : 0u);
            mma_commit(smem_addr(&empty[s]));
            if (++s == stages) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (failed) *abortp = 1;
        mma_commit(smem_addr(&acc_full));
        if (failed) mbar_wait(smem_addr(&acc_full), 0u);  // bounded: nothing in flight when tensor memory is freed
    }
    __syncwarp();
    if (failed && lane == 0) atomicOr(status, kStatusTimeout);
    tc_fence_before();
    __syncthreads();
    if (warp == 4) tmem_free(tmem, acc_cols);
}

// FP32 [V][C] -> BF16 [V][8 C8], zero padded; one thread per 8 channels.
__global__ void k_pad_bf16(const float* __restrict__ x, long long V, int C, int C8, int vec, uint4* __restrict__ xb) {
    const long long n = V * C8;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        float f[8];
        if (vec) {  // C = 8 C8, 16-byte aligned
            const float4 a = reinterpret_cast<const float4*>(x)[2 * e], b = reinterpret_cast<const float4*>(x)[2 * e + 1];
            f[0] = a.x, f[1] = a.y, f[2] = a.z, f[3] = a.w, f[4] = b.x, f[5] = b.y, f[6] = b.z, f[7] = b.w;
        } else {
            const long long v = e / C8;
            const int c = (int)(e - v * C8) * 8;
#pragma unroll
            for (int j = 0; j < 8; ++j) f[j] = c + j < C ? x[v * C + c + j] : 0.0f;
        }
        __nv_bfloat162 h[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]);
        xb[e] = *reinterpret_cast<uint4*>(h);
    }
}

// g = dy, zero where relu and the output y <= 0, as BF16 [V][C]; column sums of
// g over the block's rows (rows blockIdx.x * rows ...) to part[blockIdx.x][C].
// A thread keeps 8 fixed columns; C8 * rpi threads work, rpi rows at a time.
constexpr int kActThreads = 256;
__global__ void __launch_bounds__(kActThreads)
    k_act_back_sum(const float* __restrict__ dy, const float* __restrict__ y, long long V, int C8, int relu, int rows,
                   uint4* __restrict__ gb, float* __restrict__ part) {
    __shared__ float red[kActThreads * 8];
    const long long r0 = (long long)blockIdx.x * rows, r1 = min(V, r0 + rows);
    for (int cb = 0; cb < C8; cb += kActThreads) {  // one pass for C <= 2048
        const int w = min(kActThreads, C8 - cb), rpi = kActThreads / w;
        const int c = threadIdx.x % w, rr = threadIdx.x / w;
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (rr < rpi)
            for (long long r = r0 + rr; r < r1; r += rpi) {
                const long long e = r * C8 + cb + c;
                const float4 a = reinterpret_cast<const float4*>(dy)[2 * e], b = reinterpret_cast<const float4*>(dy)[2 * e + 1];
                const float4 p = reinterpret_cast<const float4*>(y)[2 * e], q = reinterpret_cast<const float4*>(y)[2 * e + 1];
                float f[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
                const float o[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
                __nv_bfloat162 h[4];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (relu && !(o[j] > 0.0f)) f[j] = 0.0f;
                    acc[j] += f[j];
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]);
                gb[e] = *reinterpret_cast<uint4*>(h);
            }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 8; ++j) red[j * kActThreads + threadIdx.x] = acc[j];
        __syncthreads();
        for (int k = threadIdx.x; k < w * 8; k += kActThreads) {
            const int col = k >> 3, j = k & 7;
            float sum = 0.0f;
            for (int q = 0; q < rpi; ++q) sum += red[j * kActThreads + q * w + col];
            part[(long long)blockIdx.x * C8 * 8 + (cb + col) * 8 + j] = sum;
        }
    }
}

// dw[o][tap C + c] (+)= sum_s parts[s][tap 8 C8 + c][o], db[o] (+)= sum_b part[b][o], in order.
__global__ void k_dw_reduce(const float* __restrict__ parts, int splits, int C, int Cp, int Cout,
                            const float* __restrict__ dbpart, int nparts, float* __restrict__ dw, float* __restrict__ db,
                            int accumulate) {
    const int n = kTaps * Cp * Cout;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) {
        const int o = e % Cout, k = e / Cout, tap = k / Cp, c = k % Cp;
        if (c >= C) return;
        float acc = 0.0f;
#pragma unroll 8
        for (int s = 0; s < splits; ++s) acc += parts[(long long)s * n + e];
        float* d = dw + ((long long)o * kTaps + tap) * C + c;
        *d = accumulate ? *d + acc : acc;
    } else if (e < n + Cout) {
        const int o = e - n;
        float acc = 0.0f;
#pragma unroll 8
        for (int s = 0; s < nparts; ++s) acc += dbpart[(long long)s * Cout + o];
        db[o] = accumulate ? db[o] + acc : acc;
    }
}

// wk[(tap C8 + c8)][Np][8] = w[n][tap C + 8 c8 + j] (forward) and
// wd[(tap O8 + o8)][Cn][8] = w[8 o8 + j][tap C + n] (backward data), zero
// elsewhere; one zero slab ends each.
__global__ void k_conv_pack(const float* __restrict__ w, int Cout, int C, int C8, int Np, int O8, int Cn,
                            __nv_bfloat16* __restrict__ wk, __nv_bfloat16* __restrict__ wd) {
    const long long nk = (long long)(kTaps * C8 + 1) * Np * 8, nd = (long long)(kTaps * O8 + 1) * Cn * 8;
    const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (e < nk) {
        const int j = (int)(e & 7);
        const long long q = e >> 3;
        const int n = (int)(q % Np), slab = (int)(q / Np), tap = slab / C8, c = (slab % C8) * 8 + j;
        wk[e] = __float2bfloat16_rn(tap < kTaps && n < Cout && c < C ? w[((long long)n * kTaps + tap) * C + c] : 0.0f);
    } else if (e < nk + nd) {
        const long long f = e - nk;
        const int j = (int)(f & 7);
        const long long q = f >> 3;
        const int n = (int)(q % Cn), slab = (int)(q / Cn), tap = slab / O8, o = (slab % O8) * 8 + j;
        wd[f] = __float2bfloat16_rn(tap < kTaps && n < C && o < Cout ? w[((long long)o * kTaps + tap) * C + n] : 0.0f);
    }
}

int sm_count() {
    static const int n = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0 ? v : 152;
    }();
    return n;
}

int round_up(int n, int m) { return (n + m - 1) / m * m; }

// Entry lists: convolution rows (ncls 1; stride 1 or 2), its adjoint for
// stride 1 (mirrored offsets), or for stride 2 (parity classes).
void set_entry(Gather& g, int i, int cls, int id, int ez, int ey, int ex) {
    g.id[i] = id;
    g.off[i] = (ez * g.H + ey) * g.W + ex;
    const unsigned bit = 1u << (i - g.cbeg[cls]);
    const int e[3] = {ez, ey, ex};
    for (int a = 0; a < 3; ++a) {
        if (e[a] < 0) g.neg[cls][a] |= bit;
        if (e[a] > 0) g.pos[cls][a] |= bit;
    }
}

Gather gather_conv(int B, int D, int H, int W, int C8, int stride, bool adjoint) {
    Gather g{};
    g.B = B, g.D = D, g.H = H, g.W = W, g.C8 = C8;
    g.Dr = (D - 1) / stride + 1, g.Hr = (H - 1) / stride + 1, g.Wr = (W - 1) / stride + 1;
    g.scale = stride;
    g.ncls = 1;
    g.cbeg[1] = kTaps;
    g.rz[0] = g.Dr, g.ry[0] = g.Hr, g.rx[0] = g.Wr;
    const int m = adjoint ? -1 : 1;
    for (int t = 0; t < kTaps; ++t) set_entry(g, t, 0, t, m * (t / 9 - 1), m * (t / 3 % 3 - 1), m * (t % 3 - 1));
    g.tile0[1] = (int)(((long long)B * g.Dr * g.Hr * g.Wr + kRows - 1) / kRows);
    return g;
}

// rows: input voxels D x H x W; gathered: the stride-2 output grid.  Along an
// axis an even coordinate 2 i reads tap 1 of output i; an odd one, 2 i + 1,
// tap 0 of output i + 1 and tap 2 of output i.
Gather gather_adjoint2(int B, int D, int H, int W, int O8) {
    Gather g{};
    g.B = B, g.D = (D - 1) / 2 + 1, g.H = (H - 1) / 2 + 1, g.W = (W - 1) / 2 + 1, g.C8 = O8;
    g.Dr = D, g.Hr = H, g.Wr = W;
    g.scale = 1;
    g.ncls = 8;
    int i = 0;
    for (int c = 0; c < 8; ++c) {
        const int pz = c >> 2, py = (c >> 1) & 1, px = c & 1;
        g.rz[c] = (D - pz + 1) / 2, g.ry[c] = (H - py + 1) / 2, g.rx[c] = (W - px + 1) / 2;
        g.cbeg[c] = i;
        for (int t = 0; t < kTaps; ++t) {
            const int d[3] = {t / 9, t / 3 % 3, t % 3}, p[3] = {pz, py, px};
            bool on = true;
            for (int a = 0; a < 3; ++a) on = on && (p[a] ? d[a] != 1 : d[a] == 1);
            if (on) set_entry(g, i++, c, t, d[0] == 0, d[1] == 0, d[2] == 0);
        }
        const long long n = (long long)B * g.rz[c] * g.ry[c] * g.rx[c];
        g.tile0[c + 1] = g.tile0[c] + (int)((n + kRows - 1) / kRows);
    }
    g.cbeg[8] = i;
    return g;
}

// Accumulator columns (power of two, at least 32) and stages for tiles of bn
// columns: two blocks per SM while their stages fit, else one.
int acc_columns(int bn) { return bn <= 32 ? 32 : (bn <= 64 ? 64 : (bn <= 128 ? 128 : 256)); }
int stages_for(unsigned stage_bytes) {
    const int two = (int)(110u * 1024u / stage_bytes), one = (int)(220u * 1024u / stage_bytes);
    const int s = two >= kLag + 1 ? two : one;
    return s > kMaxStages ? kMaxStages : s;
}

// Tile width for N columns over mt row tiles: as wide as possible (the gather
// is repeated for every column tile) while the tiles still fill the GPU;
// small products (the deep levels) are cut into narrower ones.
int tile_cols(int Np, long long mt) {
    const int widest = Np < 256 ? Np : 256;
    int nt = (Np + widest - 1) / widest;
    while (mt * nt < sm_count() && round_up((Np + nt - 1) / nt, 16) > 16) ++nt;
    return round_up((Np + nt - 1) / nt, 16);
}

cudaError_t launch_conv(const void* A, const Gather& g, const void* wk, int N, float* Y, const float* bias, int relu,
                        unsigned* status, cudaStream_t s) {
    const int Np = round_up(N, 16), bn = tile_cols(Np, g.tile0[g.ncls]);
    const unsigned stage = kSlabs * kRows * 16 + kSlabs * bn * 16;
    const int stages = stages_for(stage), smem = (int)(stages * stage);
    const cudaError_t e = cudaFuncSetAttribute(k_conv, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024);
    if (e != cudaSuccess) return e;
    const long long tiles = (long long)g.tile0[g.ncls] * ((Np + bn - 1) / bn);
    const int slots = sm_count() * (smem <= 110 * 1024 && acc_columns(bn) <= 128 ? 2 : 1);
    const int vec = N % 4 == 0 && (reinterpret_cast<uintptr_t>(Y) & 15u) == 0;
    k_conv<<<(int)std::min<long long>(tiles, slots), kConvThreads, smem, s>>>(
        (const uint4*)A, g, (const uint4*)wk, Np, bn, acc_columns(bn), stages, Y, bias, N, relu, vec, status);
    return cudaGetLastError();
}

struct DwPlan {
    int mt, nt, bn, stages, smem, nchunks, per, splits;
};

DwPlan dw_plan(long long V, int C8, int Cout) {
    DwPlan p;
    p.mt = (kTaps * C8 + 15) / 16;
    const int Np = round_up(Cout, 16);
    p.nt = (Np + 255) / 256;
    p.bn = round_up((Np + p.nt - 1) / p.nt, 16);
    const unsigned stage = 16 * kDwVox * 16 + p.bn / 8 * kDwVox * 16;
    p.stages = stages_for(stage);
    p.smem = (int)(p.stages * stage);
    p.nchunks = (int)((V + kDwVox - 1) / kDwVox);
    const int slots = sm_count() * (p.smem <= 110 * 1024 ? 2 : 1);
    int want = slots / (p.mt * p.nt);
    want = want < 1 ? 1 : (want > p.nchunks ? p.nchunks : want);
    p.per = (p.nchunks + want - 1) / want;
    p.splits = (p.nchunks + p.per - 1) / p.per;
    return p;
}

int act_blocks(long long V) {
    const long long b = (V + 63) / 64;
    return (int)(b > 304 ? 304 : b);
}

bool bad_conv(int B, int D, int H, int W, int C, int Cout, int s) {
    if (B < 1 || D < 1 || H < 1 || W < 1 || C < 1 || Cout < 8 || Cout % 8 || (s != 1 && s != 2)) return true;
    return (long long)B * D * H * W > 0x7fffffffLL / ((C + 7) / 8 + Cout / 8);
}

bool misaligned(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) != 0; }

long long out_voxels(int B, int D, int H, int W, int s) {
    return (long long)B * ((D - 1) / s + 1) * ((H - 1) / s + 1) * ((W - 1) / s + 1);
}

}  // namespace
}  // namespace vefd_nn

using namespace vefd_nn;

extern "C" {

void vefd_nn_conv3d_sizes(int Cin, int Cout, long long* wk, long long* wd) {
    const int C8 = (Cin + 7) / 8, O8 = Cout / 8;
    if (wk) *wk = (long long)(kTaps * C8 + 1) * round_up(Cout, 16) * 8;
    if (wd) *wd = (long long)(kTaps * O8 + 1) * round_up(Cin, 16) * 8;
}

int vefd_nn_conv3d_pack(const float* w, int Cin, int Cout, void* wk, void* wd, void* stream) {
    if (!w || !wk || !wd || Cin < 1 || Cout < 8 || Cout % 8 || misaligned(wk) || misaligned(wd)) return VEFD_NN_ERR_ARG;
    long long nk, nd;
    vefd_nn_conv3d_sizes(Cin, Cout, &nk, &nd);
    k_conv_pack<<<(int)((nk + nd + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        w, Cout, Cin, (Cin + 7) / 8, round_up(Cout, 16), Cout / 8, round_up(Cin, 16), (__nv_bfloat16*)wk,
        (__nv_bfloat16*)wd);
    return cudaGetLastError() == cudaSuccess ? VEFD_NN_OK : VEFD_NN_ERR_CUDA;
}

int vefd_nn_conv3d_forward(const float* x, int B, int D, int H, int W, int Cin, int stride, const void* wk,
                           const float* bias, int Cout, int relu, void* xb, float* y, unsigned* status, void* stream) {
    if (!x || !wk || !xb || !y || !status || bad_conv(B, D, H, W, Cin, Cout, stride) || misaligned(wk) || misaligned(xb))
        return VEFD_NN_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int C8 = (Cin + 7) / 8;
    const long long V = (long long)B * D * H * W, n = V * C8;
    const int vec = Cin % 8 == 0 && !misaligned(x);
    k_pad_bf16<<<(int)std::min<long long>((n + 255) / 256, 152 * 16), 256, 0, s>>>(x, V, Cin, C8, vec, (uint4*)xb);
    const cudaError_t e = launch_conv(xb, gather_conv(B, D, H, W, C8, stride, false), wk, Cout, y, bias, relu, status, s);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? VEFD_NN_OK : VEFD_NN_ERR_CUDA;
}

long long vefd_nn_conv3d_backward_scratch(int B, int D, int H, int W, int Cin, int stride, int Cout) {
    if (bad_conv(B, D, H, W, Cin, Cout, stride)) return 0;
    const long long V = out_voxels(B, D, H, W, stride);
    const int C8 = (Cin + 7) / 8;
    const DwPlan p = dw_plan(V, C8, Cout);
    return V * Cout / 2 + (long long)p.splits * kTaps * C8 * 8 * Cout + (long long)act_blocks(V) * Cout;
}

int vefd_nn_conv3d_backward(const void* xb, const float* y, const float* dy, int B, int D, int H, int W, int Cin,
                            int stride, const void* wd, int Cout, int relu, float* scratch, float* dw, float* db,
                            int accumulate, float* dx, unsigned* status, void* stream) {
    if (!xb || !y || !dy || !wd || !scratch || !dw || !db || !dx || !status || bad_conv(B, D, H, W, Cin, Cout, stride))
        return VEFD_NN_ERR_ARG;
    if (misaligned(xb) || misaligned(y) || misaligned(dy) || misaligned(wd) || misaligned(scratch)) return VEFD_NN_ERR_ARG;
    const long long V = out_voxels(B, D, H, W, stride);
    if (V % 8) return VEFD_NN_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int C8 = (Cin + 7) / 8, O8 = Cout / 8, nb = act_blocks(V);
    const DwPlan p = dw_plan(V, C8, Cout);
    uint4* gb = (uint4*)scratch;
    float* parts = scratch + V * Cout / 2;
    float* dbpart = parts + (long long)p.splits * kTaps * C8 * 8 * Cout;
    const int rows = (int)((V + nb - 1) / nb);
    k_act_back_sum<<<nb, kActThreads, 0, s>>>(dy, y, V, O8, relu, rows, gb, dbpart);
    cudaError_t e = cudaFuncSetAttribute(k_conv_dw, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024);
    if (e != cudaSuccess) return VEFD_NN_ERR_CUDA;
    k_conv_dw<<<dim3(p.mt, p.nt, p.splits), kDwThreads, p.smem, s>>>(
        (const uint4*)xb, gather_conv(B, D, H, W, C8, stride, false), gb, Cout, p.bn, acc_columns(p.bn), p.stages,
        p.nchunks, p.per, parts, status);
    const int n = kTaps * C8 * 8 * Cout + Cout;
    k_dw_reduce<<<(n + 127) / 128, 128, 0, s>>>(parts, p.splits, Cin, C8 * 8, Cout, dbpart, nb, dw, db, accumulate);
    const Gather g = stride == 1 ? gather_conv(B, D, H, W, O8, 1, true) : gather_adjoint2(B, D, H, W, O8);
    e = launch_conv(gb, g, wd, Cin, dx, nullptr, 0, status, s);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? VEFD_NN_OK : VEFD_NN_ERR_CUDA;
}

}  // extern "C"

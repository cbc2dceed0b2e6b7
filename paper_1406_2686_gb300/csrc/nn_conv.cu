// 3x3x3 convolution layers of the warm-start network as implicit GEMMs on the
// tcgen05 tensor cores (channels-last activations, zero padding 1, stride 1 or 2).
//
// Nothing but a BF16 copy of the activations, xb[voxel][Cp] (Cp = channels
// rounded up to 8), is read: bulk tensor copies bring the voxels a tile's rows
// touch (the tile and a one-voxel halo, zeros beyond the grid) into shared
// memory once, as
//   [slab of 8 channels][plane z][row y][voxel x] of 16-byte pieces,
// and every one of the 27 taps is then an operand that lies there already:
// eight voxels along x are one core matrix of the no-swizzle layout (K-major for
// the rows of a product, MN-major for the voxel sum of the weight gradient), the
// row groups are one tile row apart, and a tap only moves the start address.
// For stride 2 the odd and the even voxels of a row are two tensors, staged one
// after the other, so that eight output voxels again read consecutive pieces.
// (Staging with 128 threads' 16-byte asynchronous copies instead was slower:
// 97 against 92 us for 48 -> 16 channels at 64^3, its weight gradient 82
// against 62 us.)
//   k_conv     rows = voxels, K = (tap, channel), N = output channels, bias and
//              ReLU in the epilogue: the forward pass, and with the gradient as
//              input the backward-data pass (stride 1: mirrored taps; stride 2:
//              the eight parities of the input voxels are eight accumulators
//              over the same staged gradient, each with its one to eight taps).
//   k_conv_dw  dW^T[(tap, channel)][o] = sum over voxels, one accumulator per tap.
// Sums over K run channel block by channel block (channel_blocks: one block up
// to 256 channels at stride 1 and 96 at stride 2), in it tap by tap and 16
// values at a time.  With one block of a multiple of 8 channels that is the
// order of the im2col product, and the bits are its bits; channels padded to a
// multiple of 8 and several blocks group the terms differently.
//
// Measured, 64^3 unless said: the prediction 330 us (explicit im2col matrices and
// their scalar kernels: 12263); 48 -> 16 channels forward and backward 171 us
// (6742), of it 43 us forward, 61 us weight gradient, 31 us data gradient, 36 us
// conversion, mask and sums; 232 -> 80 at 16^3 101 us (780).  Deep levels are one
// chain a tile: at 16^3 392 steps on one accumulator at 85 clocks, beside which
// setup (2k clocks), the halo's 9000 pieces (10k), and 49 chunks of weights count;
// 48 -> 16 at 64^3 by the tensor core's 39 clocks a step of 16 columns (22 us of
// the 43) and the staging of 16-byte pieces.  The layers of 8 and 16 channels at
// 64^3 take 22-24 us each, of which the tensor core needs 4 to 7: one or two items a
// block, so set-up, staging, steps and the epilogue's FP32 and BF16 stores (17 and 8
// MB) follow one another more than they overlap.  What made the chain
// shorter: weights of part of the columns by one box a chunk instead of 2 x chunk
// small copies (forward at 16^3 49.0 to 42.2 us together with halo planes that
// land in three groups), and waits of one poll (prediction 345 to 330 us).
#include <algorithm>
#include <cmath>

#include "nn_tc.cuh"
#include "vefd_nn.h"

namespace vefd_nn {
namespace {

constexpr int kTaps = 27;
constexpr int kConvThreads = 256;       // warps 0-3 epilogue, 4 and 6 matrix operations, 5 weights, 7 halo copies
constexpr int kBStages = 4;             // ring of weight chunks
constexpr int kTapPlanes = 3;           // groups of halo planes that land one after the other
constexpr int kMaxPairs = 512;          // K = 16 steps of a channel block
constexpr unsigned kSmemMax = 217u * 1024u;

// A pass over tiles of 8 x PY x T row voxels.  Row (z, y, x) sits at gathered
// voxel s * (z, y, x); the staged halo starts lo voxels from the tile's first
// one and spans hz x hy x hx (for s = 2: hx of each parity of x).
struct Halo {
    int B, D, H, W;     // gathered grid
    int C8;             // 16-byte pieces per gathered voxel
    int nblk, Cb;       // channel blocks staged one after the other, pieces of a block (one block: Cb = C8; else even)
    int slabs;          // staged slabs: Cb, or Cb + 1 for odd Cb (see pair_of)
    int s, lo;
    int PY, T;
    int hx, hy, hz;
    unsigned pitch_y, pitch_plane, pitch_par, pitch_slab;  // bytes
    int Rz, Ry, Rx;     // row grid the tiles cover
    int ntx, nty, ntz, ntiles;
    int odd_x;          // added to the x coordinate in the odd-voxel tensor (far out of range when it is empty)
};

struct TileAt {
    int b, z, y, x;  // first row voxel
};
__device__ __forceinline__ TileAt tile_at(const Halo& h, int t) {
    TileAt a;
    a.x = (t % h.ntx) * 8;
    t /= h.ntx;
    a.y = (t % h.nty) * h.PY;
    t /= h.nty;
    a.z = (t % h.ntz) * h.T;
    a.b = t / h.ntz;
    return a;
}

// Copies of one slab of the staged halo (from gathered plane gz on, channels
// c ..., boxes of the tensor maps): one tensor, or the odd and the even voxels.
__device__ __forceinline__ void stage_slab(const Halo& h, const CUtensorMap* tm0, const CUtensorMap* tm1, const TileAt& a,
                                           int gz, unsigned dst, int c, unsigned bar) {
    const int y = a.y * h.s + h.lo;
    if (h.s == 1) {
        tma_load_5d(dst, tm0, c, a.x + h.lo, y, gz, a.b, bar);
    } else {
        tma_load_5d(dst, tm1, c, a.x - 1 + h.odd_x, y, gz, a.b, bar);     // voxels 2 x - 1, 2 x + 1, ...
        tma_load_5d(dst + h.pitch_par, tm0, c, a.x, y, gz, a.b, bar);     // voxels 2 x, 2 x + 2, ...
    }
}

// Entries (taps) of a pass, grouped in runs; run r accumulates its entries
// [beg[r], beg[r + 1]) in accumulators r * T ... r * T + T - 1.
struct Entries {
    int nrun, beg[9];
    int off[kTaps];    // byte offset of the entry's first row in the staged halo (slab 0)
    int npairs;
};

// Operand A of every K = 16 step: the pieces q = 0, 1, ... of a run's (entry,
// slab) sequence two at a time.  Word 0 is the low word of the matrix
// descriptor (start and leading offset in 16-byte units, the start relative to
// the staged halo), word 1 the run and whether the step is its first.  For odd
// Cb a step may pair the last slab of one entry with the first of the next; the
// leading offset must be positive, so the last slab is staged a second time, in
// front (position 0, slab c at c + 1).  A run of an odd number of pieces ends
// with a zero weight slab (paired with staged data).
__device__ __forceinline__ uint2 pair_of(const Halo& h, const Entries& e, int k) {
    const int C = h.Cb;
    int r = 0, first = 0;
    for (;; ++r) {
        const int np = ((e.beg[r + 1] - e.beg[r]) * C + 1) / 2;
        if (k < first + np) break;
        first += np;
    }
    const int q = 2 * (k - first), n = (e.beg[r + 1] - e.beg[r]) * C;
    const bool odd = C & 1;
    const int i1 = e.beg[r] + q / C, c1 = q % C;
    const int p1 = odd ? (c1 == C - 1 ? 0 : c1 + 1) : c1;
    const unsigned a1 = e.off[i1] + (unsigned)p1 * h.pitch_slab;
    unsigned a2 = a1 + h.pitch_slab;
    if (q + 1 < n) {
        const int i2 = e.beg[r] + (q + 1) / C, c2 = (q + 1) % C;
        a2 = e.off[i2] + (unsigned)(odd ? c2 + 1 : c2) * h.pitch_slab;
    }
    return make_uint2((a1 >> 4) | (((a2 - a1) >> 4) << 16), (unsigned)r | (q == 0 ? 1u << 16 : 0u));
}

// Output voxel of row (z, y, x) in run r, -1 beyond the grid.  Parity runs
// (adjoint of stride 2): voxel 2 (z, y, x) + the run's parity bits.
__device__ __forceinline__ long long out_voxel(int nrun, int r, int b, int z, int y, int x, int Do, int Ho, int Wo) {
    if (nrun > 1) {
        z = 2 * z + (r >> 2);
        y = 2 * y + ((r >> 1) & 1);
        x = 2 * x + (r & 1);
    }
    if (z >= Do || y >= Ho || x >= Wo) return -1;
    return (((long long)b * Do + z) * Ho + y) * Wo + x;
}

constexpr unsigned kBHi = (128u >> 4) | (1u << 14);  // high word of the weights' matrix descriptor

__device__ __forceinline__ uint64_t desc64(unsigned lo, unsigned hi) { return (uint64_t)lo | ((uint64_t)hi << 32); }

// Steps [k0, k1) of a single run by one of the two issuing warps: its
// accumulators are the planes t = me, me + 2, ... < T.  Two steps an iteration
// with their table words loaded ahead; only the very first step starts the sums.
template <int T>
__device__ __forceinline__ void issue_steps(const uint2* pairs, int k0, int k1, unsigned me, unsigned base16, unsigned a_hi,
                                            unsigned step_t, unsigned b_lo, int bn, unsigned d, uint32_t idesc, bool started) {
    constexpr int U = T == 4 ? 2 : 1;  // accumulators of this warp
    const unsigned a0 = base16 + me * step_t, d0 = d + me * (unsigned)bn;
    const unsigned a1 = a0 + 2 * step_t, d1 = d0 + 2u * (unsigned)bn;
    unsigned acc = started ? 1u : 0u;
    uint4 next = *reinterpret_cast<const uint4*>(pairs + k0);
    int k = k0;
    for (; k + 1 < k1; k += 2) {
        const uint4 pr = next;
        next = *reinterpret_cast<const uint4*>(pairs + k + 2);
        const uint64_t b0 = desc64(b_lo, kBHi), b1 = desc64(b_lo + 2u * (unsigned)bn, kBHi);
        mma_f16_warp(d0, desc64(pr.x + a0, a_hi), b0, idesc, acc);
        if (U == 2) mma_f16_warp(d1, desc64(pr.x + a1, a_hi), b0, idesc, acc);
        mma_f16_warp(d0, desc64(pr.z + a0, a_hi), b1, idesc, 1u);
        if (U == 2) mma_f16_warp(d1, desc64(pr.z + a1, a_hi), b1, idesc, 1u);
        b_lo += 4u * (unsigned)bn;
        acc = 1u;
    }
    if (k < k1) {
        mma_f16_warp(d0, desc64(next.x + a0, a_hi), desc64(b_lo, kBHi), idesc, acc);
        if (U == 2) mma_f16_warp(d1, desc64(next.x + a1, a_hi), desc64(b_lo, kBHi), idesc, acc);
    }
}

// The same for the parity runs (T = 1): this warp's accumulators are the odd or
// the even runs.
__device__ __forceinline__ void issue_runs(const uint2* pairs, int k0, int k1, unsigned me, unsigned base16, unsigned a_hi,
                                           unsigned b_lo, int bn, unsigned d, uint32_t idesc, bool started) {
    for (int k = k0; k < k1; ++k, b_lo += 2u * (unsigned)bn) {
        const uint2 pr = pairs[k];
        const unsigned run = pr.y & 0xffu;
        if ((run & 1u) == me)
            mma_f16_warp(d + run * (unsigned)bn, desc64(pr.x + base16, a_hi), desc64(b_lo, kBHi), idesc,
                         (pr.y >> 16) && !started ? 0u : 1u);
    }
}

// Wait of a whole warp.  A phase that is complete already, the common case in
// front of a chunk, costs one poll; only a wait that is not looks at the abort flag.
__device__ __forceinline__ bool warp_wait(unsigned bar, unsigned parity, volatile int* abortp) {
    if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait(bar, parity) && !*abortp);
}

__device__ __forceinline__ uint4 pack8(const float* f) {
    __nv_bfloat162 h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]);
    return *reinterpret_cast<uint4*>(h);
}

// Blocks walk the (tile, column block) items blockIdx.x, + gridDim.x, ...
// Warp 7 copies each item's halo (channel block by channel block) into one of
// `nbuf` buffers, warp 5 streams the weights Wk[piece][Np][8 BF16] (pieces in
// the order of the K steps) through a ring; warps 4 and 6 issue the matrix operations, each
// those of every other accumulator, into one of `nset` accumulator sets; warps
// 0-3 drain the other.
// Every wait is bounded; a timeout sets the status bit and an abort flag that
// the other roles see at their next wait; each role then waits (bounded) for
// its own copies or matrix operations before tensor memory is freed.
__global__ void __launch_bounds__(kConvThreads, 2)
    k_conv(const __grid_constant__ CUtensorMap tm0, const __grid_constant__ CUtensorMap tm1,
           const __grid_constant__ CUtensorMap tmw, const __grid_constant__ Halo h, const __grid_constant__ Entries ent, const uint4* __restrict__ Wk, int Np, int bn,
           int nbuf, int nset, int cols, int chunk, int groups, float* __restrict__ Y, uint4* __restrict__ Yb, int Do, int Ho,
           int Wo, const float* __restrict__ bias, int N, int relu, int vec, unsigned* __restrict__ status) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) unsigned long long afull[2][kTapPlanes], aempty[2], bfull[kBStages], bempty[kBStages], acc_full[2],
        acc_empty[2], drain[2];
    __shared__ __align__(16) uint2 pairs[kMaxPairs + 2];
    __shared__ unsigned tmem_base;
    __shared__ int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned base = smem_addr(dsm);
    const unsigned a_bytes = (unsigned)h.slabs * h.pitch_slab, b_base = base + (unsigned)nbuf * a_bytes;
    const unsigned b_bytes = (unsigned)chunk * 2u * bn * 16u;
    const int nchunk = (ent.npairs + chunk - 1) / chunk;  // per channel block
    const int ntn = (Np + bn - 1) / bn, nitems = h.ntiles * ntn;
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            for (int g = 0; g < kTapPlanes; ++g) mbar_init_n(smem_addr(&afull[s][g]), 1);
            mbar_init_n(smem_addr(&aempty[s]), 2);
            mbar_init_n(smem_addr(&acc_full[s]), 2);
            mbar_init_n(smem_addr(&acc_empty[s]), 4);
            mbar_init_n(smem_addr(&drain[s]), 1);
        }
        for (int s = 0; s < kBStages; ++s) {
            mbar_init_n(smem_addr(&bfull[s]), 1);
            mbar_init_n(smem_addr(&bempty[s]), 2);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    if (warp == 4) tmem_alloc(&tmem_base, cols);
    for (int k = threadIdx.x; k < ent.npairs; k += kConvThreads) pairs[k] = pair_of(h, ent, k);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = tmem_base;
    volatile int* abortp = &abort_flag;
    bool failed = false;
    if (warp < 4) {
        // epilogue; tensor-memory lanes 32 q ... of this warp: 128 rows one per lane, 64 rows in the first 16 lanes
        const bool m64 = h.PY == 8;
        const int row = m64 ? warp * 16 + lane : warp * 32 + lane;
        const int nacc = ent.nrun * h.T;
        int j = 0;
        for (int t = blockIdx.x; t < nitems; t += gridDim.x, ++j) {
            const int set = j % nset;
            const TileAt a = tile_at(h, t / ntn);
            const int n0 = (t % ntn) * bn, bw = min(bn, Np - n0);
            const int ry = a.y + (row >> 3), rx = a.x + (row & 7);
            const bool ready = mbar_wait(smem_addr(&acc_full[set]), (unsigned)((j / nset) & 1)) && !*abortp;
            if (!__all_sync(0xffffffffu, ready)) {
                failed = true;
                break;
            }
            tc_fence_after();
            for (int k = 0; k < nacc; ++k) {
                const int r = k / h.T, rz = a.z + k % h.T;
                const bool in = (!m64 || lane < 16) && rz < h.Rz && ry < h.Ry && rx < h.Rx;
                const long long o = in ? out_voxel(ent.nrun, r, a.b, rz, ry, rx, Do, Ho, Wo) : -1;
                float* y = Y + (o < 0 ? 0 : o) * N;
                uint4* yb = Yb ? Yb + (o < 0 ? 0 : o) * (N / 8) : nullptr;
                for (int c0 = 0; c0 < bw && n0 + c0 < N; c0 += 16) {
                    uint32_t v[16];
                    tmem_ld16(tmem + ((unsigned)(warp * 32) << 16) + (unsigned)((set * nacc + k) * bn + c0), v);
                    if (o < 0) continue;
                    float f[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const int n = n0 + c0 + i;
                        f[i] = __uint_as_float(v[i]);
                        if (bias && n < N) f[i] += __ldg(bias + n);
                        if (relu) f[i] = fmaxf(f[i], 0.0f);
                    }
#pragma unroll
                    for (int i = 0; i < 16; i += 4) {
                        const int n = n0 + c0 + i;
                        if (vec) {
                            if (n < N) *reinterpret_cast<float4*>(y + n) = make_float4(f[i], f[i + 1], f[i + 2], f[i + 3]);
                        } else {
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                if (n + q < N) y[n + q] = f[i + q];
                        }
                    }
                    if (yb) {  // N a multiple of 8
#pragma unroll
                        for (int i = 0; i < 16; i += 8)
                            if (n0 + c0 + i < N) yb[(n0 + c0 + i) / 8] = pack8(f + i);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&acc_empty[set]));
        }
    } else if (warp == 5) {
        int ib = 0;
        for (int t = blockIdx.x; t < nitems && !failed; t += gridDim.x) {
            const int n0 = (t % ntn) * bn;
            for (int q = 0; q < nchunk * h.nblk; ++q, ++ib) {
                const int sb = ib % kBStages, blk = q / nchunk, c = q % nchunk;
                if (ib >= kBStages && !mbar_wait(smem_addr(&bempty[sb]), (unsigned)((ib / kBStages - 1) & 1))) failed = true;
                if (__any_sync(0xffffffffu, failed || *abortp)) {
                    failed = true;
                    break;
                }
                const unsigned bb = smem_addr(&bfull[sb]), dst = b_base + (unsigned)sb * b_bytes;
                const long long piece = ((long long)blk * ent.npairs + c * chunk) * 2;
                if (lane == 0) {
                    if (bn == Np) {
                        const unsigned bytes = 2u * (unsigned)min(chunk, ent.npairs - c * chunk) * (unsigned)bn * 16u;
                        mbar_expect(bb, bytes);
                        bulk_load(dst, Wk + piece * Np, bytes, bb);
                    } else {
                        // one box of chunk pieces x bn columns (zeros beyond the arrays count as copied)
                        mbar_expect(bb, b_bytes);
                        tma_load_2d(dst, &tmw, n0 * 2, (int)piece, bb);
                    }
                }
                __syncwarp();
            }
        }
        if (failed) *abortp = 1;
        // bounded: the copies in flight land before the block leaves
        for (int q = ib > kBStages ? ib - kBStages : 0; q < ib; ++q)
            mbar_wait(smem_addr(&bfull[q % kBStages]), (unsigned)((q / kBStages) & 1));
    } else if (warp == 7) {
        const unsigned tx = (unsigned)(h.slabs * h.s) * (unsigned)(h.hx * h.hy) * 16u;  // of one plane
        int ia = 0;
        for (int t = blockIdx.x; t < nitems && !failed; t += gridDim.x) {
            const TileAt a = tile_at(h, t / ntn);
            for (int blk = 0; blk < h.nblk; ++blk, ++ia) {
                const int s = ia % nbuf;
                if (ia >= nbuf && !mbar_wait(smem_addr(&aempty[s]), (unsigned)((ia / nbuf - 1) & 1))) failed = true;
                if (__any_sync(0xffffffffu, failed || *abortp)) {
                    failed = true;
                    break;
                }
                for (int g = 0; g < groups; ++g) {
                    const unsigned bar = smem_addr(&afull[s][g]);
                    const int z0 = g == 0 ? 0 : h.hz - groups + g, nz = g == 0 ? h.hz - groups + 1 : 1;
                    if (lane == 0) mbar_expect(bar, tx * (unsigned)nz);
                    __syncwarp();
                    const int boxes = groups == 1 ? 1 : nz;  // a box is the whole halo or one plane
                    for (int p = lane; p < h.slabs * boxes; p += 32) {
                        // slab q: piece q of the block, or with the copy in front (odd Cb) piece q - 1
                        const int q = p / boxes, z = z0 + p % boxes;
                        const int c = h.slabs == h.Cb ? blk * h.Cb + q : (q == 0 ? h.Cb : q) - 1;
                        stage_slab(h, &tm0, &tm1, a, a.z * h.s + h.lo + z,
                                   base + (unsigned)s * a_bytes + (unsigned)q * h.pitch_slab + (unsigned)z * h.pitch_plane,
                                   c * 8, bar);
                    }
                    __syncwarp();
                }
            }
        }
        if (failed) *abortp = 1;
        // bounded: the copies in flight land before the block leaves
        for (int q = ia > nbuf ? ia - nbuf : 0; q < ia; ++q)
            for (int g = 0; g < groups; ++g) mbar_wait(smem_addr(&afull[q % nbuf][g]), (unsigned)((q / nbuf) & 1));
    } else {
        const unsigned me = warp == 6;  // this warp's accumulators: run * T + t odd or even
        const unsigned a_hi = ((unsigned)h.s * h.pitch_y >> 4) | (1u << 14);
        const unsigned step_t = (unsigned)h.s * h.pitch_plane >> 4;
        const unsigned set_cols = (unsigned)(ent.nrun * h.T * bn);
        int ia = 0, ib = 0, j = 0;
        for (int t = blockIdx.x; t < nitems && !failed; t += gridDim.x, ++j) {
            const int set = j % nset, n0 = (t % ntn) * bn;
            const uint32_t idesc = instr_desc(h.PY * 8, min(bn, Np - n0));
            if (j >= nset)
                failed = __any_sync(0xffffffffu, !mbar_wait(smem_addr(&acc_empty[set]), (unsigned)((j / nset - 1) & 1)));
            tc_fence_after();
            for (int blk = 0; blk < h.nblk && !failed; ++blk, ++ia) {
                const int s = ia % nbuf;
                int landed = 0;  // plane groups waited for
                const unsigned base16 = (base + (unsigned)s * a_bytes) >> 4;
                for (int c = 0; c < nchunk && !failed; ++c, ++ib) {
                    const int sb = ib % kBStages;
                    failed = !warp_wait(smem_addr(&bfull[sb]), (unsigned)((ib / kBStages) & 1), abortp);
                    if (failed) break;
                    const int k0 = c * chunk, k1 = min(k0 + chunk, ent.npairs);
                    // the first step that reads tap plane g is 9 g Cb / 2
                    while (landed < groups && 2 * k1 > 9 * landed * h.Cb && !failed) {
                        failed = !warp_wait(smem_addr(&afull[s][landed]), (unsigned)((ia / nbuf) & 1), abortp);
                        ++landed;
                    }
                    if (failed) break;
                    tc_fence_after();
                    const unsigned b_lo = ((b_base + (unsigned)sb * b_bytes) >> 4) | ((unsigned)bn << 16);
                    const unsigned dset = tmem + (unsigned)set * set_cols;
                    if (ent.nrun > 1) issue_runs(pairs, k0, k1, me, base16, a_hi, b_lo, bn, dset, idesc, blk > 0);
                    else if (h.T == 4) issue_steps<4>(pairs, k0, k1, me, base16, a_hi, step_t, b_lo, bn, dset, idesc, blk + k0 > 0);
                    else if (h.T == 2) issue_steps<2>(pairs, k0, k1, me, base16, a_hi, step_t, b_lo, bn, dset, idesc, blk + k0 > 0);
                    else if (me == 0) issue_steps<1>(pairs, k0, k1, 0, base16, a_hi, step_t, b_lo, bn, dset, idesc, blk + k0 > 0);
                    mma_commit_warp(smem_addr(&bempty[sb]));
                }
                if (!failed) mma_commit_warp(smem_addr(&aempty[s]));
            }
            if (failed) break;
            mma_commit_warp(smem_addr(&acc_full[set]));  // arrives once the item's matrix operations have completed
        }
        if (failed) {
            *abortp = 1;
            // bounded: every matrix operation issued has completed before tensor memory is freed
            __syncwarp();
            mma_commit_warp(smem_addr(&drain[me]));
            mbar_wait(smem_addr(&drain[me]), 0u);
        }
    }
    __syncwarp();
    if (failed) *abortp = 1;
    if (failed && lane == 0) atomicOr(status, kStatusTimeout);
    tc_fence_before();
    __syncthreads();
    if (warp == 4) tmem_free(tmem, cols);
}

// parts[split][k][o] = sum over the split's voxels v of xb[neighbour of v by
// k's tap][k's channels] * gb[v][o], k = tap * 8 C8 + channel.  The rows of a
// product are (plane offset dz, channel slab) pairs, `mslabs` of the 3 C8 a block
// (64 or 128 rows, so that few channels still fill them); a block keeps one
// accumulator per tap (dy, dx) of its `ntap` and walks its tiles of 8 x PY
// voxels: per tile it stages the halo plane of every slab and the tile's
// gradients, [slab][row y][8 voxels], both MN-major operands, 16 voxels (two
// tile rows) a step.  Bound by the tensor core's 39 clocks a step.
constexpr int kDwStages = 4;  // at most

__global__ void __launch_bounds__(kConvThreads, 2)
    k_conv_dw(const __grid_constant__ CUtensorMap tm0, const __grid_constant__ CUtensorMap tm1,
              const __grid_constant__ CUtensorMap tmG, const __grid_constant__ Halo h, int Cout, int bn, int cols, int ntap,
              int mslabs, int stages, int tiles_per, float* __restrict__ parts, unsigned* __restrict__ status) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) unsigned long long full[kDwStages], empty[kDwStages], acc_full;
    __shared__ unsigned tmem_base;
    __shared__ int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned base = smem_addr(dsm);
    const unsigned a_bytes = (unsigned)mslabs * h.pitch_slab, g_slab = (unsigned)h.PY * 128u;
    const unsigned stage_bytes = a_bytes + (unsigned)(bn / 8) * g_slab;
    const int ngrp = 9 / ntap, grp = blockIdx.x % ngrp, mblk = blockIdx.x / ngrp;
    const int tap0 = grp * ntap;  // first (dy, dx)
    const int f0 = mblk * mslabs, nsl = min(mslabs, 3 * h.C8 - f0);  // (dz, slab) rows dz * C8 + slab
    const int n0 = blockIdx.y * bn, nb = min(bn, Cout - n0) / 8;
    const int t0 = blockIdx.z * tiles_per, nt = min(h.ntiles - t0, tiles_per);
    const int M = mslabs <= 8 ? 64 : 128;
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init_n(smem_addr(&full[s]), 1);
            mbar_init_n(smem_addr(&empty[s]), 2);
        }
        mbar_init_n(smem_addr(&acc_full), 2);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    if (warp == 4) tmem_alloc(&tmem_base, cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = tmem_base;
    volatile int* abortp = &abort_flag;
    bool failed = false;
    if (warp == 5) {
        const unsigned tx = (unsigned)(nsl * h.s) * (unsigned)(h.hx * h.hy) * 16u + (unsigned)nb * g_slab;
        int it = 0;
        for (; it < nt; ++it) {
            const int s = it % stages;
            if (it >= stages && !mbar_wait(smem_addr(&empty[s]), (unsigned)((it / stages - 1) & 1))) failed = true;
            if (__any_sync(0xffffffffu, failed || *abortp)) {
                failed = true;
                break;
            }
            const TileAt a = tile_at(h, t0 + it);
            const unsigned dst = base + (unsigned)s * stage_bytes, fb = smem_addr(&full[s]);
            if (lane == 0) mbar_expect(fb, tx);
            __syncwarp();
            for (int p = lane; p < nsl; p += 32) {
                const int f = f0 + p, dz = f / h.C8;
                stage_slab(h, &tm0, &tm1, a, a.z * h.s + h.lo + dz, dst + (unsigned)p * h.pitch_slab, (f - dz * h.C8) * 8, fb);
            }
            for (int o = lane; o < nb; o += 32)
                tma_load_5d(dst + a_bytes + (unsigned)o * g_slab, &tmG, n0 + o * 8, a.x, a.y, a.z, a.b, fb);
        }
        if (failed) *abortp = 1;
        // bounded: the copies in flight land before the block leaves
        for (int q = it > stages ? it - stages : 0; q < it; ++q)
            mbar_wait(smem_addr(&full[q % stages]), (unsigned)((q / stages) & 1));
    } else if (warp < 4) {
        const bool ready = !failed && mbar_wait(smem_addr(&acc_full), 0u) && !*abortp;
        if (__all_sync(0xffffffffu, ready)) {
            tc_fence_after();
            const int m = M == 64 ? warp * 16 + lane : warp * 32 + lane;
            const bool in = (M == 128 || lane < 16) && m < nsl * 8;
            const int f = f0 + (in ? m >> 3 : 0), dz = f / h.C8, c0 = (f - dz * h.C8) * 8 + (m & 7);
            for (int j = 0; j < ntap; ++j) {
                const long long k = (long long)(dz * 9 + tap0 + j) * h.C8 * 8 + c0;
                float* out = parts + ((long long)blockIdx.z * kTaps * h.C8 * 8 + (in ? k : 0)) * Cout + n0;
                for (int c = 0; c < bn && n0 + c < Cout; c += 16) {
                    uint32_t v[16];
                    tmem_ld16(tmem + ((unsigned)(warp * 32) << 16) + (unsigned)(j * bn + c), v);
                    if (!in) continue;
#pragma unroll
                    for (int i = 0; i < 16; i += 4)
                        if (n0 + c + i < Cout)
                            *reinterpret_cast<float4*>(out + c + i) =
                                make_float4(__uint_as_float(v[i]), __uint_as_float(v[i + 1]), __uint_as_float(v[i + 2]),
                                            __uint_as_float(v[i + 3]));
                }
            }
        } else {
            failed = true;
            *abortp = 1;
        }
    } else if (warp == 4 || warp == 6) {
        // warps 4 and 6 take every other tap
        const int me = warp == 6;
        const uint32_t idesc = instr_desc_mn(M, bn);
        const unsigned ky = (unsigned)h.s * h.pitch_y;  // voxel groups: one tile row apart
        for (int it = 0; it < nt; ++it) {
            const int s = it % stages;
            failed = !warp_wait(smem_addr(&full[s]), (unsigned)((it / stages) & 1), abortp);
            if (failed) break;
            tc_fence_after();
            const unsigned sa = base + (unsigned)s * stage_bytes, sb = sa + a_bytes;
            const uint64_t bd = smem_desc(sb, 128, g_slab);
            for (int j = me; j < ntap; j += 2) {
                const int dy = (tap0 + j) / 3, dx = (tap0 + j) % 3;
                // stride 2: dx = 0 and 2 read odd voxels (staged first), dx = 1 the even ones
                const unsigned a0 = sa + (unsigned)dy * h.pitch_y +
                                    (h.s == 1 ? (unsigned)dx * 16u : (dx == 1 ? h.pitch_par : (unsigned)(dx >> 1) * 16u));
                const uint64_t ad = smem_desc(a0, ky, h.pitch_slab);
                const unsigned d = tmem + (unsigned)(j * bn);
                mma_f16_warp(d, ad, bd, idesc, it > 0 ? 1u : 0u);
#pragma unroll 3
                for (int k = 1; k < h.PY / 2; ++k)
                    mma_f16_warp(d, ad + (uint64_t)((unsigned)k * (2 * ky >> 4)), bd + (uint64_t)(k * 16), idesc, 1u);
            }
            mma_commit_warp(smem_addr(&empty[s]));
        }
        if (failed) *abortp = 1;
        __syncwarp();
        mma_commit_warp(smem_addr(&acc_full));
        if (failed) mbar_wait(smem_addr(&acc_full), 0u);  // bounded: nothing in flight when tensor memory is freed
    }
    __syncwarp();
    if (failed && lane == 0) atomicOr(status, kStatusTimeout);
    tc_fence_before();
    __syncthreads();
    if (warp == 4) tmem_free(tmem, cols);
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
        xb[e] = pack8(f);
    }
}

// xb[v] = [u[v / 2] (nearest-neighbour upsampling by 2), s[v]]: the pieces of
// two BF16 grids, U8 and S8 a voxel; u is B x D/2 x H/2 x W/2, s and xb B x D x H x W.
__global__ void k_up_concat(const uint4* __restrict__ u, int U8, const uint4* __restrict__ s, int S8, int B, int D, int H, int W,
                            uint4* __restrict__ xb) {
    const unsigned C = U8 + S8, n = (unsigned)B * D * H * W * C;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const unsigned v = e / C, c = e - v * C;
        if (c >= (unsigned)U8) {
            xb[e] = s[(long long)v * S8 + c - U8];
        } else {
            const unsigned x = v % W, r = v / W, y = r % H, q = r / H, z = q % D, b = q / D;
            xb[e] = u[((((long long)b * (D / 2) + z / 2) * (H / 2) + y / 2) * (W / 2) + x / 2) * U8 + c];
        }
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
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (relu && !(o[j] > 0.0f)) f[j] = 0.0f;
                    acc[j] += f[j];
                }
                gb[e] = pack8(f);
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

// dw[o][tap C + c] (+)= sum_s parts[s][tap 8 C8 + c][o] (the first `dwblocks`
// blocks, a thread each), db[o] (+)= sum_b part[b][o] (a warp each: lanes take
// every 32nd part, then a fixed tree).
__global__ void __launch_bounds__(128)
    k_dw_reduce(const float* __restrict__ parts, int splits, int C, int Cp, int Cout, const float* __restrict__ dbpart,
                int nparts, int dwblocks, float* __restrict__ dw, float* __restrict__ db, int accumulate) {
    if ((int)blockIdx.x < dwblocks) {
        const int n = kTaps * Cp * Cout;
        const int e = blockIdx.x * blockDim.x + threadIdx.x;
        if (e >= n) return;
        const int o = e % Cout, k = e / Cout, tap = k / Cp, c = k % Cp;
        if (c >= C) return;
        float acc = 0.0f;
#pragma unroll 16
        for (int s = 0; s < splits; ++s) acc += parts[(long long)s * n + e];
        float* d = dw + ((long long)o * kTaps + tap) * C + c;
        *d = accumulate ? *d + acc : acc;
    } else {
        const int o = ((int)blockIdx.x - dwblocks) * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
        if (o >= Cout) return;
        float acc = 0.0f;
        for (int s = lane; s < nparts; s += 32) acc += dbpart[(long long)s * Cout + o];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, d);
        if (lane == 0) db[o] = accumulate ? db[o] + acc : acc;
    }
}

// Packed weights of a pass: pieces in the order of its K steps, channel block by
// channel block, run by run (tap by tap, the block's pieces of each), a run
// padded to an even count; piece [n < Np][8 BF16], zero where there is none.
// Forward: piece (tap, c8) holds w[n][tap C + 8 c8 + j].  Backward data: piece
// (tap, o8) holds w[8 o8 + j][tap C + n]; stride 1 visits mirrored taps, stride 2
// the taps of the eight parity runs.
struct PackRuns {
    int nrun, beg[9], tap[kTaps], slab0[9];  // slab0: first piece of a run inside a block, then the block's pieces
    int nblk, Cb, rows, cols;                // rows: output index n < rows; cols: channels summed over
    int np;                                  // n padded
    int sn, sc, st;                          // strides of w for n, the summed channel and the tap
};

__device__ __forceinline__ void pack_one(const float* __restrict__ w, const PackRuns& p, long long e,
                                         __nv_bfloat16* __restrict__ out) {
    const int j = (int)(e & 7);
    const long long q = e >> 3;
    const int n = (int)(q % p.np);
    int slab = (int)(q / p.np);
    const int blk = slab / p.slab0[p.nrun];
    slab -= blk * p.slab0[p.nrun];
    int r = 0;
    while (slab >= p.slab0[r + 1]) ++r;
    const int k = slab - p.slab0[r], i = p.beg[r] + k / p.Cb, c = (blk * p.Cb + k % p.Cb) * 8 + j;
    float v = 0.0f;
    if (i < p.beg[r + 1] && n < p.rows && c < p.cols)
        v = w[(long long)n * p.sn + (long long)c * p.sc + (long long)p.tap[i] * p.st];
    out[e] = __float2bfloat16_rn(v);
}

__global__ void k_conv_pack(const float* __restrict__ w, const __grid_constant__ PackRuns pk, long long nk,
                            __nv_bfloat16* __restrict__ wk, const __grid_constant__ PackRuns pd, long long nd,
                            __nv_bfloat16* __restrict__ wd) {
    const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (e < nk) pack_one(w, pk, e, wk);
    else if (e < nk + nd) pack_one(w, pd, e - nk, wd);
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

int acc_alloc(int cols) {
    int c = 32;
    while (c < cols) c *= 2;
    return c;
}

// Halo geometry of a pass: kind 0 convolution (or its stride-1 adjoint) over
// rows Rz x Ry x Rx at stride s, kind 1 the adjoint of stride 2 (rows: the
// gathered grid itself, each the corner of eight output voxels).
// Channel blocks: as many pieces as the smallest tile's halo can stage (4.8,
// 13.9 or 2.6 KB a piece); the usual layers are one block.
void channel_blocks(int kind, int s, int C8, int* nblk, int* Cb) {
    const int most = kind == 1 ? 36 : (s == 1 ? 32 : 12);
    *nblk = (C8 + most - 1) / most;
    *Cb = *nblk == 1 ? C8 : round_up((C8 + *nblk - 1) / *nblk, 2);
}

// Strides of the staged halo: boxes (all planes, or one each) land 128-byte aligned.
void set_pitches(Halo& h, bool plane_boxes = false) {
    h.pitch_y = h.hx * 16, h.pitch_plane = h.hy * h.pitch_y;
    if (plane_boxes) h.pitch_plane = round_up(h.pitch_plane, 128);
    h.pitch_par = round_up(h.hz * h.pitch_plane, 128);
    h.pitch_slab = h.s * h.pitch_par;
}

Halo halo_of(int kind, int B, int D, int H, int W, int C8, int s, int PY, int T) {
    Halo h{};
    h.B = B, h.D = D, h.H = H, h.W = W, h.C8 = C8;
    channel_blocks(kind, s, C8, &h.nblk, &h.Cb);
    h.slabs = (h.Cb & 1) ? h.Cb + 1 : h.Cb;
    h.s = s, h.PY = PY, h.T = T;
    if (kind == 0) {
        h.lo = -1;
        h.hx = s == 1 ? 10 : 9, h.hy = s * (PY - 1) + 3, h.hz = s * (T - 1) + 3;
        h.Rz = (D - 1) / s + 1, h.Ry = (H - 1) / s + 1, h.Rx = (W - 1) / s + 1;
    } else {
        h.lo = 0;
        h.hx = 9, h.hy = PY + 1, h.hz = T + 1;
        h.Rz = D, h.Ry = H, h.Rx = W;
    }
    set_pitches(h);
    h.ntx = (h.Rx + 7) / 8, h.nty = (h.Ry + PY - 1) / PY, h.ntz = (h.Rz + T - 1) / T;
    const long long n = (long long)B * h.ntx * h.nty * h.ntz;
    h.ntiles = n > 0x3fffffffLL ? 0 : (int)n;
    h.odd_x = W < 2 ? 1 << 20 : 0;
    return h;
}

// Entry at halo offset (z, y, x); for stride 2 x = 0 and 2 are odd voxels (staged first), 1 an even one.
void add_entry(Entries& e, const Halo& h, int i, int z, int y, int x) {
    const unsigned xo = h.s == 1 ? x * 16u : (x == 1 ? h.pitch_par : (x >> 1) * 16u);
    e.off[i] = (int)(z * h.pitch_plane + y * h.pitch_y + xo);
}

void count_pairs(Entries& e, int Cb) {
    e.npairs = 0;
    for (int r = 0; r < e.nrun; ++r) e.npairs += ((e.beg[r + 1] - e.beg[r]) * Cb + 1) / 2;
}

// Taps in the order of their pieces: the staged halo's (z, y, x) offsets.
Entries conv_entries(const Halo& h) {
    Entries e{};
    e.nrun = 1;
    e.beg[1] = kTaps;
    for (int t = 0; t < kTaps; ++t) add_entry(e, h, t, t / 9, t / 3 % 3, t % 3);
    count_pairs(e, h.Cb);
    return e;
}

// Adjoint of stride 2.  Along an axis an even input coordinate 2 i reads tap 1
// of output i; an odd one, 2 i + 1, tap 2 of output i and tap 0 of output i + 1.
// Run = parity (z, y, x); its entries by increasing offset.
PackRuns adjoint_runs() {
    PackRuns p{};
    p.nrun = 8;
    int i = 0;
    for (int c = 0; c < 8; ++c) {
        p.beg[c] = i;
        for (int k = 0; k < 8; ++k) {  // offsets (z, y, x) of the gathered output
            const int o[3] = {k >> 2, (k >> 1) & 1, k & 1}, par[3] = {c >> 2, (c >> 1) & 1, c & 1};
            int tap = 0;
            bool on = true;
            for (int a = 0; a < 3; ++a) {
                on = on && (par[a] || !o[a]);
                tap = 3 * tap + (par[a] ? (o[a] ? 0 : 2) : 1);
            }
            if (on) p.tap[i++] = tap;
        }
    }
    p.beg[8] = i;
    return p;
}

PackRuns plain_run(bool mirrored) {
    PackRuns p{};
    p.nrun = 1;
    p.beg[1] = kTaps;
    for (int t = 0; t < kTaps; ++t) p.tap[t] = mirrored ? kTaps - 1 - t : t;
    return p;
}

// The packed arrays of a layer w[Cout][27 Cin] (forward, or its data gradient)
// and their length in BF16 elements.
PackRuns pack_plan(bool adjoint, int Cin, int Cout, int stride, long long* elems) {
    const bool par = adjoint && stride == 2;
    PackRuns p = par ? adjoint_runs() : plain_run(adjoint);
    p.rows = adjoint ? Cin : Cout;
    p.cols = adjoint ? Cout : Cin;
    p.np = round_up(p.rows, 16);
    p.sn = adjoint ? 1 : kTaps * Cin;
    p.sc = adjoint ? kTaps * Cin : 1;
    p.st = Cin;
    channel_blocks(par, adjoint ? 1 : stride, (p.cols + 7) / 8, &p.nblk, &p.Cb);
    for (int r = 0; r < p.nrun; ++r) p.slab0[r + 1] = p.slab0[r] + ((p.beg[r + 1] - p.beg[r]) * p.Cb + 1) / 2 * 2;
    *elems = (long long)p.nblk * p.slab0[p.nrun] * p.np * 8;
    return p;
}

Entries adjoint_entries(const Halo& h) {
    Entries e{};
    e.nrun = 8;
    int i = 0;
    for (int c = 0; c < 8; ++c) {
        e.beg[c] = i;
        for (int k = 0; k < 8; ++k)
            if (((k >> 2) <= (c >> 2)) && (((k >> 1) & 1) <= ((c >> 1) & 1)) && ((k & 1) <= (c & 1)))
                add_entry(e, h, i++, k >> 2, (k >> 1) & 1, k & 1);
    }
    e.beg[8] = i;
    count_pairs(e, h.Cb);
    return e;
}

// Tensor map of a BF16 grid [B][D][H][W][8 C8], or of its voxels of one parity
// of x (step 2), with boxes of 8 channels x bx x by x bz voxels.
bool grid_map(CUtensorMap* out, const void* base, int B, int D, int H, int W, int C8, int step, int first, int bx, int by,
              int bz) {
    const EncodeTiled encode = tensor_map_encoder();
    if (!encode) return false;
    const int nx = (W - first + step - 1) / step;
    if (nx < 1) first = 0;  // no such voxel: any valid tensor, read out of range (Halo::odd_x)
    const cuuint64_t row = (cuuint64_t)C8 * 16;
    const cuuint64_t dims[5] = {(cuuint64_t)C8 * 8, (cuuint64_t)(nx < 1 ? 1 : nx), (cuuint64_t)H, (cuuint64_t)D, (cuuint64_t)B};
    const cuuint64_t strides[4] = {row * step, row * W, row * W * H, row * W * H * D};
    const cuuint32_t box[5] = {8, (cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz, 1}, one[5] = {1, 1, 1, 1, 1};
    return encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (char*)const_cast<void*>(base) + first * row, dims, strides, box,
                  one, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool halo_maps(CUtensorMap* tm0, CUtensorMap* tm1, const void* A, const Halo& h, int bz) {
    if (!grid_map(tm0, A, h.B, h.D, h.H, h.W, h.C8, h.s, 0, h.hx, h.hy, bz)) return false;
    *tm1 = *tm0;  // stride 1 has one tensor
    return h.s == 1 || grid_map(tm1, A, h.B, h.D, h.H, h.W, h.C8, h.s, h.s - 1, h.hx, h.hy, bz);
}

// Tensor map of packed weights [piece][Np][8 BF16] in 8-byte elements, with
// boxes of `pieces` pieces x bn columns.
bool weight_map(CUtensorMap* out, const void* wk, long long npieces, int Np, int bn, int pieces) {
    const EncodeTiled encode = tensor_map_encoder();
    if (!encode) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)Np * 2, (cuuint64_t)npieces}, strides[1] = {(cuuint64_t)Np * 16};
    const cuuint32_t box[2] = {(cuuint32_t)bn * 2, (cuuint32_t)pieces}, one[2] = {1, 1};
    return encode(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<void*>(wk), dims, strides, box, one,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct ConvPlan {
    int PY, T, bn, chunk, nbuf, nset, occ, groups;
    unsigned smem;
    bool ok;
};

// Tile of a pass: the choice with the least estimated time.  Per item, in SM
// clocks: the staged pieces at one a clock and their latency, the matrix
// operations at 39 a step (half a clock a column beyond 78) on the SM's tensor
// core and at 85 on each of a block's issuing warps, which take every other
// accumulator, 450 a chunk of weights, and 1500 between the items of a block;
// 6000 for launch and the first copies.  (Deep levels, a few hundred steps over
// a few tiles, are a chain of steps and chunks; the fine ones fill the SMs.)
ConvPlan search_plan(int kind, int B, int D, int H, int W, int C8, int s, int Np, int nrun, int npairs) {
    ConvPlan best{};
    double best_t = 0.0;
    for (int PY = 8; PY <= 16; PY += 8)
        for (int T = 1; T <= 4; T *= 2) {
            if (kind == 1 && T > 1) continue;
            const Halo h = halo_of(kind, B, D, H, W, C8, s, PY, T);
            if (!h.ntiles) continue;
            Halo hp = h;  // staged plane by plane
            set_pitches(hp, true);
            int last = 0;
            for (int nt = 1; nt <= (Np + 15) / 16; ++nt) {
                const int bn = round_up((Np + nt - 1) / nt, 16), set = nrun * T * bn;
                if (bn > (nt == 1 ? 256 : 128) || set > 512 || bn == last) continue;
                last = bn;
                for (int chunk = 2; chunk <= 32; chunk *= 2) {
                    ConvPlan p{PY, T, bn, chunk, 2, set <= 256 ? 2 : 1, 1, 1, 0, true};
                    const unsigned ring = kBStages * (unsigned)chunk * 2 * bn * 16;
                    const int cols = acc_alloc(p.nset * set);
                    const long long items = (long long)h.ntiles * ((Np + bn - 1) / bn);
                    auto fit = [&](const Halo& g) {
                        const unsigned a = g.slabs * g.pitch_slab;
                        p.nbuf = 2 * a + ring > kSmemMax ? 1 : 2;
                        p.smem = p.nbuf * a + ring;
                        p.occ = std::max(1, std::min(4, std::min((int)(kSmemMax / (p.smem + 5120)), 512 / cols)));
                    };
                    fit(hp);
                    if (kind == 0 && p.smem <= kSmemMax && items <= (long long)sm_count() * p.occ) p.groups = kTapPlanes;
                    else fit(h);
                    if (p.smem > kSmemMax) continue;
                    const long long slots = (long long)sm_count() * p.occ;
                    const double load = (double)h.nblk * (1.0 * h.hz * h.hy * h.hx * h.s * h.slabs + 1500.0);
                    const double steps = (double)npairs * h.nblk;
                    const double mma = steps * T * std::max(39.0, bn / 2.0);               // the SM's tensor core
                    const double issue = steps * (nrun > 1 ? 0.5 : (T + 1) / 2) * std::max(85.0, bn / 2.0) +
                                         450.0 * h.nblk * ((npairs + chunk - 1) / chunk);  // a block's warps
                    // an SM works through its share; a block's own items follow one another
                    const double share = (double)items / sm_count(), chain = (double)((items + slots - 1) / slots);
                    const double own = p.nbuf == 2 ? std::max(load, issue) : load + issue;
                    const double tm = std::max(std::ceil(share) * std::max(load, mma), chain * (own + 1500.0)) + load + 6000.0;
                    if (!best.ok || tm < best_t) {
                        best = p;
                        best_t = tm;
                    }
                }
            }
        }
    return best;
}

// The search takes longer on the host than a small layer on the device, so
// each thread keeps the plans of the last layer shapes it launched.
ConvPlan plan_conv(int kind, int B, int D, int H, int W, int C8, int s, int Np, int nrun, int npairs) {
    struct Slot {
        int key[8];
        ConvPlan plan;
    };
    constexpr int kSlots = 64;
    static thread_local Slot slots[kSlots];  // plan.ok == false: empty
    const int key[8] = {kind, B, D, H, W, C8, s, Np};
    unsigned at = 0;
    for (int v : key) at = (at * 31u + (unsigned)v) * 2654435761u;
    Slot& q = slots[at >> 26];
    if (!q.plan.ok || !std::equal(key, key + 8, q.key)) {
        q.plan = search_plan(kind, B, D, H, W, C8, s, Np, nrun, npairs);
        std::copy(key, key + 8, q.key);
    }
    return q.plan;
}

// kind as halo_of; N output channels, Y on the grid Do x Ho x Wo.
cudaError_t launch_conv(int kind, const void* A, int B, int D, int H, int W, int C8, int s, const void* wk, int N, float* Y,
                        void* Yb, int Do, int Ho, int Wo, const float* bias, int relu, unsigned* status, cudaStream_t st) {
    const int Np = round_up(N, 16), nrun = kind == 1 ? 8 : 1;
    Entries e = kind == 1 ? adjoint_entries(halo_of(1, B, D, H, W, C8, 1, 8, 1)) : conv_entries(halo_of(0, B, D, H, W, C8, s, 8, 1));
    if (e.npairs > kMaxPairs) return cudaErrorInvalidValue;
    const ConvPlan p = plan_conv(kind, B, D, H, W, C8, s, Np, nrun, e.npairs);
    if (!p.ok) return cudaErrorInvalidValue;
    Halo h = halo_of(kind, B, D, H, W, C8, s, p.PY, p.T);
    set_pitches(h, p.groups > 1);
    e = kind == 1 ? adjoint_entries(h) : conv_entries(h);
    const long long items = (long long)h.ntiles * ((Np + p.bn - 1) / p.bn);
    if (items > 0x3fffffffLL) return cudaErrorInvalidValue;
    const int grid = (int)std::min<long long>(items, (long long)sm_count() * p.occ);
    CUtensorMap tm0, tm1, tmw{};
    if (!halo_maps(&tm0, &tm1, A, h, p.groups == 1 ? h.hz : 1)) return cudaErrorInvalidValue;
    if (p.bn < Np && !weight_map(&tmw, wk, (long long)h.nblk * e.npairs * 2, Np, p.bn, p.chunk * 2)) return cudaErrorInvalidValue;
    const cudaError_t err = cudaFuncSetAttribute(k_conv, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (err != cudaSuccess) return err;
    const int vec = N % 4 == 0 && (reinterpret_cast<uintptr_t>(Y) & 15u) == 0;
    k_conv<<<grid, kConvThreads, p.smem, st>>>(tm0, tm1, tmw, h, e, (const uint4*)wk, Np, p.bn, p.nbuf, p.nset,
                                               acc_alloc(p.nset * nrun * p.T * p.bn), p.chunk, p.groups, Y, (uint4*)Yb, Do, Ho, Wo, bias, N, relu,
                                               vec, status);
    return cudaGetLastError();
}

struct DwPlan {
    int PY, bn, ntap, mslabs, mblks, nt, stages, ntiles, per, splits;
    unsigned smem;
};

// Halo of the weight gradient: one plane at a time.
Halo dw_halo(int B, int D, int H, int W, int C8, int s, int PY) {
    Halo h = halo_of(0, B, D, H, W, C8, s, PY, 1);
    h.hz = 1;
    set_pitches(h);
    return h;
}

// Weight gradient: as many taps per block as tensor memory holds (they share
// the staged planes), rows in equal blocks of at most 16 slabs; split over the
// tiles until the blocks fill the SMs.
DwPlan dw_plan(int B, int D, int H, int W, int C8, int s, int Cout) {
    DwPlan p{};
    const int Np = round_up(Cout, 16);
    p.nt = (Np + 159) / 160;
    p.bn = round_up((Np + p.nt - 1) / p.nt, 16);
    p.ntap = 9 * p.bn <= 512 ? 9 : 3;
    p.mblks = (3 * C8 + 15) / 16;
    p.mslabs = (3 * C8 + p.mblks - 1) / p.mblks;
    for (p.PY = (H - 1) / s + 1 > 8 ? 16 : 8;; p.PY = 8) {
        const Halo h = dw_halo(B, D, H, W, C8, s, p.PY);
        const unsigned stage = p.mslabs * h.pitch_slab + p.bn / 8 * (unsigned)p.PY * 128;
        // rows beyond the staged slabs read on into what follows: the last stage needs this slack
        const unsigned slack = ((p.mslabs <= 8 ? 8 : 16) - p.mslabs) * h.pitch_slab;
        p.stages = std::min(kDwStages, (int)((kSmemMax - slack) / stage));
        p.smem = p.stages * stage + slack;
        p.ntiles = h.ntiles;
        if (p.stages >= 2 || p.PY == 8) break;
    }
    const int cols = acc_alloc(p.ntap * p.bn);
    const int occ = std::max(1, std::min((int)(kSmemMax / (p.smem + 2048)), 512 / cols));
    const int blocks = 9 / p.ntap * p.mblks * p.nt;
    const int want = std::max(1, std::min(sm_count() * occ / blocks, p.ntiles));
    p.per = (p.ntiles + want - 1) / want;
    p.splits = (p.ntiles + p.per - 1) / p.per;
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

int vefd_nn_conv3d_sizes(int Cin, int Cout, int stride, long long* wk, long long* wd) {
    if (!wk || !wd || Cin < 1 || Cout < 8 || Cout % 8 || (stride != 1 && stride != 2)) return VEFD_NN_ERR_ARG;
    pack_plan(false, Cin, Cout, stride, wk);
    pack_plan(true, Cin, Cout, stride, wd);
    return VEFD_NN_OK;
}

int vefd_nn_conv3d_pack(const float* w, int Cin, int Cout, int stride, void* wk, void* wd, void* stream) {
    if (!w || !wk || !wd || misaligned(wk) || misaligned(wd) || Cin < 1 || Cout < 8 || Cout % 8 ||
        (stride != 1 && stride != 2))
        return VEFD_NN_ERR_ARG;
    long long nk, nd;
    const PackRuns pk = pack_plan(false, Cin, Cout, stride, &nk), pd = pack_plan(true, Cin, Cout, stride, &nd);
    k_conv_pack<<<(unsigned)((nk + nd + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        w, pk, nk, (__nv_bfloat16*)wk, pd, nd, (__nv_bfloat16*)wd);
    return cudaGetLastError() == cudaSuccess ? VEFD_NN_OK : VEFD_NN_ERR_CUDA;
}

int vefd_nn_up_concat(const void* u, int Cu, const void* s, int Cs, int B, int D, int H, int W, void* xb, void* stream) {
    if (!u || !s || !xb || Cu < 8 || Cs < 8 || Cu % 8 || Cs % 8 || B < 1 || D < 2 || H < 2 || W < 2 || D % 2 || H % 2 || W % 2)
        return VEFD_NN_ERR_ARG;
    if (misaligned(u) || misaligned(s) || misaligned(xb)) return VEFD_NN_ERR_ARG;
    const long long n = (long long)B * D * H * W * (Cu + Cs) / 8;
    if (n > 0x7fffffffLL) return VEFD_NN_ERR_ARG;
    k_up_concat<<<(int)std::min<long long>((n + 255) / 256, 152 * 16), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        (const uint4*)u, Cu / 8, (const uint4*)s, Cs / 8, B, D, H, W, (uint4*)xb);
    return cudaGetLastError() == cudaSuccess ? VEFD_NN_OK : VEFD_NN_ERR_CUDA;
}

int vefd_nn_conv3d_forward(const float* x, int B, int D, int H, int W, int Cin, int stride, const void* wk,
                           const float* bias, int Cout, int relu, void* xb, float* y, void* yb, unsigned* status,
                           void* stream) {
    if (!wk || !xb || !y || !status || bad_conv(B, D, H, W, Cin, Cout, stride) || misaligned(wk) || misaligned(xb) ||
        misaligned(yb))
        return VEFD_NN_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int C8 = (Cin + 7) / 8;
    const long long V = (long long)B * D * H * W, n = V * C8;
    const int vec = Cin % 8 == 0 && !misaligned(x);
    if (x)
        k_pad_bf16<<<(int)std::min<long long>((n + 255) / 256, 152 * 16), 256, 0, s>>>(x, V, Cin, C8, vec, (uint4*)xb);
    const cudaError_t e = launch_conv(0, xb, B, D, H, W, C8, stride, wk, Cout, y, yb, (D - 1) / stride + 1, (H - 1) / stride + 1,
                                      (W - 1) / stride + 1, bias, relu, status, s);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? VEFD_NN_OK : VEFD_NN_ERR_CUDA;
}

long long vefd_nn_conv3d_backward_scratch(int B, int D, int H, int W, int Cin, int stride, int Cout) {
    if (bad_conv(B, D, H, W, Cin, Cout, stride)) return 0;
    const long long V = out_voxels(B, D, H, W, stride);
    const int C8 = (Cin + 7) / 8;
    const DwPlan p = dw_plan(B, D, H, W, C8, stride, Cout);
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
    const DwPlan p = dw_plan(B, D, H, W, C8, stride, Cout);
    if (p.stages < 2) return VEFD_NN_ERR_ARG;
    uint4* gb = (uint4*)scratch;
    float* parts = scratch + V * Cout / 2;
    float* dbpart = parts + (long long)p.splits * kTaps * C8 * 8 * Cout;
    const int rows = (int)((V + nb - 1) / nb);
    k_act_back_sum<<<nb, kActThreads, 0, s>>>(dy, y, V, O8, relu, rows, gb, dbpart);
    cudaError_t e = cudaFuncSetAttribute(k_conv_dw, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return VEFD_NN_ERR_CUDA;
    const Halo h = dw_halo(B, D, H, W, C8, stride, p.PY);
    CUtensorMap tm0, tm1, tmG;
    if (!halo_maps(&tm0, &tm1, xb, h, 1) || !grid_map(&tmG, gb, B, h.Rz, h.Ry, h.Rx, O8, 1, 0, 8, p.PY, 1))
        return VEFD_NN_ERR_CUDA;
    k_conv_dw<<<dim3(9 / p.ntap * p.mblks, p.nt, p.splits), kConvThreads, p.smem, s>>>(
        tm0, tm1, tmG, h, Cout, p.bn, acc_alloc(p.ntap * p.bn), p.ntap, p.mslabs, p.stages, p.per, parts, status);
    const int dwblocks = (kTaps * C8 * 8 * Cout + 127) / 128;
    k_dw_reduce<<<dwblocks + (Cout + 3) / 4, 128, 0, s>>>(parts, p.splits, Cin, C8 * 8, Cout, dbpart, nb, dwblocks, dw, db,
                                                          accumulate);
    const int Do = (D - 1) / stride + 1, Ho = (H - 1) / stride + 1, Wo = (W - 1) / stride + 1;
    e = launch_conv(stride == 1 ? 0 : 1, gb, B, Do, Ho, Wo, O8, 1, wd, Cin, dx, nullptr, D, H, W, nullptr, 0, status, s);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? VEFD_NN_OK : VEFD_NN_ERR_CUDA;
}

}  // extern "C"

// A x and A^T r without stored records, from a table of legs (the on-the-fly form's workspace, or TAB mode without
// records).  Every tap of a pair shares one table phase, so with the pairs of an A-scan grouped by first tap n0
//     S[n0][col] = sum of the pairs' bilinear corner weights on table column col times x,
//     y[n0 + 1 + m] += sum_col S[n0][col] T[col][m],       col = plane * (Q + 1) + phase,
// for one tile of 128 values of n0 after another.
//
// Pairs: among rows that cross the same layers (a segment: GeomParams::seg_row) the delay grows with depth, so each
// (column, segment) of the image holds a tile's pixels in one run of rows; a cursor per (column, segment) moves on
// from tile to tile, so each pair is evaluated about once, and none past the record's end.  Just below an interface
// the delay of steep pairs grows by less per row than its rounding error (1e-5 of it at most, under one sample), so
// every bound of a run leaves one sample for pairs out of order.  A tile reaches only one or two segments of a column,
// so several warps take every nsub-th row of a run each (one thread per run left most threads waiting at the barrier
// for runs of up to 40 rows: 3.3 ms instead of 2.6, before the two forms shared the walk).  Nothing is sorted,
// compacted or staged.
//
// S is summed in 64-bit fixed point in shared memory (two 32-bit atomics per corner, the carry taken from the
// first one's old value), at a scale that the largest |x| and the tile's largest weight and number of pairs keep from
// overflow: exact, so the result does not depend on the order of the additions and every output bit is reproducible.
// A tile none of whose sums has kFlMinBits bits at that scale (x there is far below its largest) is walked again at the
// scale of its largest |w x|: the grid stays finer than FP32 beside the tile's own sums.  The product
// with the table is FP32 on the CUDA cores: it is a short convolution per column, which a thread does for four
// outputs and a share of the columns, and it keeps FP32's accuracy, which two FP16 parts on the tensor cores
// would not (3e-7 against 1.5e-7 from FP64).
//
// 256x512, 64 x 16 A-scans of 2048 samples (41 M pairs, FP32), legs included: 2.65 ms against 10.7 ms of
// forward_kernel, which gathers every tap of every pair.  The product takes 0.95 ms of it (its FP32 rate and
// the shared-memory loads that feed it), the walk over the pairs the rest (latency of the legs and the atomics).
#include <algorithm>
#include <cmath>
#include <vector>

#include "device_common.cuh"

namespace mbir {

constexpr int kFlTile = 128;                     // values of n0 per tile
constexpr int kFlThreads = 1024;
constexpr int kFlMaxTiles = 512;                 // tiles of an A-scan (set-up's shared memory)
constexpr int kFlMinBits = 26;                   // of a tile's largest sum on its fixed-point grid

// Shared memory: S as low and high words (columns of 128), then the edge taps' words, the share sums, carries,
// row flags and cursors.
struct FlLayout {
    int ng, ncg;             // groups of four outputs; shares of the columns
    size_t off_hi, off_edge, off_part, off_carry, off_bad, off_cur, smem;
};
__host__ __device__ inline FlLayout fl_layout(const GeomParams& P, int kw)
{
    FlLayout L;
    L.ng = (kFlTile + P.Tw - 1 + 3) / 4;
    L.ncg = kFlThreads / L.ng;
    L.off_hi = (size_t)kw * kFlTile * 4;
    L.off_edge = 2 * L.off_hi;
    L.off_part = L.off_edge + 2 * kFlTile * 4;
    L.off_carry = L.off_part + (size_t)L.ncg * L.ng * 16;
    L.off_bad = L.off_carry + 2 * kFlTile * 4;
    L.off_cur = L.off_bad + (kFlTile + 4) * 4;
    L.smem = L.off_cur + (((size_t)P.W * P.n_seg * 8 + 15) & ~(size_t)15);
    return L;
}

__device__ __forceinline__ float fl_float(float v) { return v; }
__device__ __forceinline__ float fl_float(__nv_bfloat16 v) { return __bfloat162float(v); }

// *out = bits of the largest finite |x| (zero before)
template <typename T>
__global__ void fl_xmax_kernel(long long N, const T* __restrict__ x, unsigned int* __restrict__ out)
{
    unsigned int m = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        const unsigned int b = __float_as_uint(fl_float(x[i])) & 0x7fffffffu;
        if (b < 0x7f800000u) m = max(m, b);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m) atomicMax(out, m);
}

// v 2^e (e split in two: 2^e itself may be out of range)
__device__ __forceinline__ float fl_scale(float v, int e)
{
    const int e1 = e >> 1;
    return v * __int_as_float((e1 + 127) << 23) * __int_as_float((e - e1 + 127) << 23);
}

// The word at `at` and its high word (`hi` words further) += q
__device__ __forceinline__ void fl_add(unsigned int* at, size_t hi, long long q)
{
    const unsigned int l = (unsigned int)q;
    unsigned int h = (unsigned int)(q >> 32);
    const unsigned int old = atomicAdd(at, l);
    h += old + l < old ? 1u : 0u;
    if (h) atomicAdd(at + hi, h);
}

__device__ __forceinline__ long long fl_word(unsigned int lo, unsigned int hi)
{
    return (long long)((unsigned long long)hi << 32 | lo);
}

__device__ __forceinline__ Leg fl_leg(float4 v) { return Leg{v.x, v.y, v.z, v.w}; }

// The cursors at tile t0: the first row of each (segment, column) whose pair starts in that tile or later, or one
// sample before it.  A cursor is row << 16 | the first tile that its pair or a later one can start in (0: not looked
// at); nxt, for the next tile, starts past each run's end.
template <int NT>
__device__ __forceinline__ void fl_cursors(const GeomParams& P, const DevPtrs& D, const int* htx, const int* hrx, int t0,
                                           unsigned int* cur, unsigned int* nxt)
{
    for (int j = threadIdx.x; j < P.W * P.n_seg; j += NT) {
        const int sg = j / P.W, col = j - sg * P.W;
        int a = P.seg_row[sg], b = P.seg_row[sg + 1];
        if (t0 == 0) b = a;
        const int ht = __ldg(htx + col), hr = __ldg(hrx + col);
        while (a < b) {
            const int mid = (a + b) >> 1;
            const float4* lr = D.legs + (size_t)mid * P.nh;
            if (make_pair(P, fl_leg(__ldg(lr + ht)), fl_leg(__ldg(lr + hr)), 1.0f).n0 < t0 * kFlTile - 1) a = mid + 1;
            else b = mid;
        }
        cur[j] = (unsigned int)a << 16;
        nxt[j] = (unsigned int)P.seg_row[sg + 1] << 16;
    }
}

// Calls pair(row, column, pair, n0 - tile's start, x) for every pair of the tile t (of non-zero weight or not), and
// sets nxt to the runs' next rows.  A warp takes 32 columns and every nsub-th row of each segment's run, with enough
// warps per run for every warp of the block to take part.
template <int NT, typename F>
__device__ __forceinline__ void fl_walk(const GeomParams& P, const DevPtrs& D, const int* htx, const int* hrx,
                                        const float* __restrict__ x, int t, const unsigned int* cur, unsigned int* nxt,
                                        F&& pair)
{
    const int ngrp = (P.W + 31) / 32, nsub = min(16, max(1, NT / 32 / ngrp)), units = ngrp * nsub;
    const int lim = min(kFlTile, P.M - 1 - t * kFlTile);           // past the tile's, and the record's, last n0
    for (int u = threadIdx.x >> 5; u < units; u += NT / 32) {
        const int sub = u / ngrp, col = (u - sub * ngrp) * 32 + (threadIdx.x & 31);
        if (col >= P.W) continue;
        const int ht = __ldg(htx + col), hr = __ldg(hrx + col);
        for (int sg = 0; sg < P.n_seg; ++sg) {
            const int j = sg * P.W + col, end = P.seg_row[sg + 1];
            const unsigned int at = cur[j];
            if ((int)(at & 0xffffu) > t) {                         // the run starts in a later tile
                if (sub == 0) atomicMin(nxt + j, at);
                continue;
            }
            int row = (int)(at >> 16) + sub;
            if (row >= end) continue;
            const float4* lr = D.legs + (size_t)row * P.nh;
            float4 a = __ldg(lr + ht), b = __ldg(lr + hr);
            for (;;) {
                // the next row's legs load while this one's pair is evaluated
                lr += (size_t)nsub * P.nh;
                float4 an = a, bn = b;
                const float xv = x ? __ldg(x + (size_t)row * P.W + col) : 0.0f;
                if (row + nsub < end) {
                    an = __ldg(lr + ht);
                    bn = __ldg(lr + hr);
                }
                const Pair pr = make_pair(P, fl_leg(a), fl_leg(b), __ldg(&D.rows[row].tau));
                const int n0r = pr.n0 - t * kFlTile;
                if (n0r > lim) {                                   // the rows below start in later tiles
                    atomicMin(nxt + j, (unsigned int)row << 16 | (unsigned int)((min(pr.n0, P.M) - 1) / kFlTile));
                    break;
                }
                if (n0r == lim) atomicMin(nxt + j, (unsigned int)row << 16 | (unsigned int)t);
                if ((unsigned)n0r < (unsigned)lim) pair(row, col, pr, n0r, xv);
                row += nsub;
                if (row >= end) break;
                a = an;
                b = bn;
            }
        }
    }
}

// The walked tile's cursors for the tile after the next
template <int NT>
__device__ __forceinline__ void fl_advance(const GeomParams& P, unsigned int*& cur, unsigned int*& nxt)
{
    for (int j = threadIdx.x; j < P.W * P.n_seg; j += NT) cur[j] = (unsigned int)P.seg_row[j / P.W + 1] << 16;
    unsigned int* const was = cur;
    cur = nxt;
    nxt = was;
}

// Block (A-scan, chunk of tiles): tiles [ta, tb), and the one before for the taps that reach past it.
__global__ void __launch_bounds__(kFlThreads, 1)
    forward_legs_kernel(GeomParams P, DevPtrs D, const float* __restrict__ ftab, const uint2* __restrict__ crange,
                        const float* __restrict__ x, const unsigned int* __restrict__ xmax, int ebits,
                        int kwmax, int per, float* __restrict__ y_f32, __nv_bfloat16* __restrict__ y_bf16,
                        int out_stride)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const FlLayout L = fl_layout(P, kwmax);
    unsigned int* lo = reinterpret_cast<unsigned int*>(smem);
    unsigned int* edge = reinterpret_cast<unsigned int*>(smem + L.off_edge);
    float* part = reinterpret_cast<float*>(smem + L.off_part);
    float* carry = reinterpret_cast<float*>(smem + L.off_carry);
    int* bad = reinterpret_cast<int*>(smem + L.off_bad);                 // rows with a non-finite x; [128]: any
    unsigned int* smax = reinterpret_cast<unsigned int*>(bad + kFlTile + 1);    // bits of the tile's largest |S|, |w x|
    // cursors of this tile and of the next, per (layer, column)
    unsigned int* cur = reinterpret_cast<unsigned int*>(smem + L.off_cur);
    unsigned int* nxt = cur + (size_t)P.W * P.n_seg;
    const size_t hiw = L.off_hi / 4;
    const int tid = threadIdx.x, k = blockIdx.x;
    const int ntile = (P.M + kFlTile - 1) / kFlTile;
    const int ta = blockIdx.y * per, tb = min(ta + per, ntile), t0 = max(ta - 1, 0);
    const int R = P.Q + 1, dR = P.G > 1 ? R : 0;
    const int* htx = D.hidx + (size_t)__ldg(D.txpos + k / P.n_rx) * P.W;
    const int* hrx = D.hidx + (size_t)__ldg(D.rxpos + k) * P.W;
    int ex = 0;                                                          // |x| < 2^ex
    frexpf(__uint_as_float(__ldg(xmax)), &ex);

    auto store = [&](int n, float v) {
        if (y_f32) y_f32[(size_t)k * out_stride + n] = v;
        else y_bf16[(size_t)k * out_stride + n] = __float2bfloat16_rn(v);
    };
    for (size_t i = tid; i < L.off_part / 4; i += kFlThreads) lo[i] = 0u;
    if (tid < 2 * kFlTile) carry[tid] = 0.0f;
    if (tid <= kFlTile + 2) bad[tid] = 0;
    if (ta == 0 && tid == 0) store(0, 0.0f);
    if (tb == ntile)
        for (int n = P.M + tid; n < out_stride; n += kFlThreads) store(n, 0.0f);
    fl_cursors<kFlThreads>(P, D, htx, hrx, t0, cur, nxt);
    __syncthreads();

    const int cg = tid / L.ng, og = tid - cg * L.ng;
    int par = 0;
    for (int t = t0; t < tb; ++t) {
        const int ts = t * kFlTile;
        const uint2 cr = __ldg(crange + (size_t)k * ntile + t);
        const int c_lo = (int)(cr.x & 0xffffu), kw = (int)(cr.x >> 16) - c_lo;
        // fixed-point scale: weights below 2^(cr.y >> 16), |x| below 2^ex and the tile's pairs of them stay below 2^61
        // (2^62 with the rounding of the products)
        const int nbits = (int)(cr.y & 0xffffu);
        int se = min(nbits - ((int)cr.y >> 16) - ex, 250);
        bool rescaled = false;
        for (bool again = kw > 0; again;) {
            // ---- the tile's pairs into S
            bool any = false;
            fl_walk<kFlThreads>(P, D, htx, hrx, x, t, cur, nxt, [&](int row, int col, const Pair& pr, int n0r, float xv) {
                const float wx = pr.w * xv;
                if (!(wx != 0.0f)) return;
                if (!(fabsf(wx) <= 3.4028235e38f)) {
                    bad[n0r] = 1;
                    bad[kFlTile] = 1;
                    return;
                }
                any = true;
                const float p1 = pr.psi, p0 = 1.0f - pr.psi;
                unsigned int* s = lo + (size_t)(pr.gi * R + pr.r - c_lo) * kFlTile + n0r;
                const float wa = wx * pr.w0, wb = wx * pr.w1;
                fl_add(s, hiw, __float2ll_rn(fl_scale(wa * p0, se)));
                fl_add(s + kFlTile, hiw, __float2ll_rn(fl_scale(wb * p0, se)));
                if (dR) {
                    fl_add(s + dR * kFlTile, hiw, __float2ll_rn(fl_scale(wa * p1, se)));
                    fl_add(s + (dR + 1) * kFlTile, hiw, __float2ll_rn(fl_scale(wb * p1, se)));
                }
                if (pr.flag0) {
                    // tau = t0 exactly: the last tap of the upper phase lies outside the window
                    const float* tl = ftab + (size_t)(pr.gi * R + pr.r + 1) * P.Tw4 + P.Tw - 1;
                    const float ev = wb * (p0 * __ldg(tl) + p1 * __ldg(tl + dR * P.Tw4));
                    fl_add(edge + n0r, kFlTile, __float2ll_rn(fl_scale(ev, se - ebits)));
                }
            });
            any = __syncthreads_or(any);
            // ---- S as FP32 in place of its low words
            uint4* l4 = reinterpret_cast<uint4*>(lo);
            uint4* h4 = reinterpret_cast<uint4*>(lo + hiw);
            float sm = 0.0f;
            for (int i = tid; i < kw * (kFlTile / 4); i += kFlThreads) {
                const uint4 l = l4[i], h = h4[i];
                h4[i] = make_uint4(0u, 0u, 0u, 0u);
                const float4 v = make_float4(__ll2float_rn(fl_word(l.x, h.x)), __ll2float_rn(fl_word(l.y, h.y)),
                                             __ll2float_rn(fl_word(l.z, h.z)), __ll2float_rn(fl_word(l.w, h.w)));
                sm = fmaxf(fmaxf(sm, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
                l4[i] = make_uint4(__float_as_uint(fl_scale(v.x, -se)), __float_as_uint(fl_scale(v.y, -se)),
                                   __float_as_uint(fl_scale(v.z, -se)), __float_as_uint(fl_scale(v.w, -se)));
            }
            unsigned int m = __reduce_max_sync(0xffffffffu, __float_as_uint(sm));
            if ((tid & 31) == 0 && m) atomicMax(smax, m);
            __syncthreads();
            again = any && !rescaled && __uint_as_float(*smax) < (float)(1u << kFlMinBits);
            if (again) {
                // too coarse a grid, unless the sums are small by cancellation: the tile's largest |w x|
                m = 0;
                fl_walk<kFlThreads>(P, D, htx, hrx, x, t, cur, nxt, [&](int, int, const Pair& pr, int, float xv) {
                    const unsigned int b = __float_as_uint(pr.w * xv) & 0x7fffffffu;
                    if (b < 0x7f800000u) m = max(m, b);
                });
                m = __reduce_max_sync(0xffffffffu, m);
                if ((tid & 31) == 0 && m) atomicMax(smax + 1, m);
                __syncthreads();
                int em = 0;
                frexpf(__uint_as_float(smax[1]), &em);
                rescaled = true;
                again = smax[1] != 0 && em + se < kFlMinBits;
                if (again) {
                    se = nbits - em;
                    for (int i = tid; i < kw * (kFlTile / 4); i += kFlThreads) l4[i] = make_uint4(0u, 0u, 0u, 0u);
                    if (tid < 2 * kFlTile) edge[tid] = 0u;
                    __syncthreads();
                }
            }
        }
        if (kw > 0) {
            // ---- outputs 4 og .. 4 og + 3 of this thread's columns: sum_m S[o - m] T[m], four taps at a time
            // against the blocks of four values of S at and below the output
            if (cg < L.ncg) {
                float y0 = 0.f, y1 = 0.f, y2 = 0.f, y3 = 0.f;
                const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
                const int ntb = P.Tw4 / 4;
                for (int c = cg; c < kw; c += L.ncg) {
                    const float4* S = reinterpret_cast<const float4*>(lo + (size_t)c * kFlTile);
                    const float4* T = reinterpret_cast<const float4*>(ftab + (size_t)(c_lo + c) * P.Tw4);
                    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
                    float4 h = og < kFlTile / 4 ? S[og] : zero;
#pragma unroll 4
                    for (int mb = 0; mb < ntb; ++mb) {
                        const int l = og - mb - 1;
                        const float4 b = (unsigned)l < (unsigned)(kFlTile / 4) ? S[l] : zero;
                        const float4 w = __ldg(T + mb);
                        a0 = fmaf(h.x, w.x, fmaf(b.w, w.y, fmaf(b.z, w.z, fmaf(b.y, w.w, a0))));
                        a1 = fmaf(h.y, w.x, fmaf(h.x, w.y, fmaf(b.w, w.z, fmaf(b.z, w.w, a1))));
                        a2 = fmaf(h.z, w.x, fmaf(h.y, w.y, fmaf(h.x, w.z, fmaf(b.w, w.w, a2))));
                        a3 = fmaf(h.w, w.x, fmaf(h.z, w.y, fmaf(h.y, w.z, fmaf(h.x, w.w, a3))));
                        h = b;
                    }
                    y0 += a0;
                    y1 += a1;
                    y2 += a2;
                    y3 += a3;
                }
                reinterpret_cast<float4*>(part)[cg * L.ng + og] = make_float4(y0, y1, y2, y3);
            }
            __syncthreads();
        }
        // ---- the shares' sums, the previous tile's carry and the edge taps -> y; taps past this tile carry on
        if (tid < 2 * kFlTile) {
            float v = 0.0f;
            if (kw > 0 && tid < 4 * L.ng) {
                for (int c = 0; c < L.ncg; ++c) v += part[c * L.ng * 4 + tid];
                const int r = tid - (P.Tw - 1);
                if (r >= 0 && r < kFlTile)
                    v -= fl_scale(__ll2float_rn(fl_word(edge[r], edge[kFlTile + r])), ebits - se);
                if (bad[kFlTile])
                    for (int q = max(r, 0); q <= min(tid, kFlTile - 1); ++q)
                        if (bad[q]) v = __uint_as_float(0x7fc00000u);
            }
            if (tid < kFlTile) {
                const int n = ts + 1 + tid;
                v += carry[par * kFlTile + tid];
                if (t >= ta && n < P.M) store(n, v);
            } else {
                carry[(par ^ 1) * kFlTile + tid - kFlTile] = v;
            }
        }
        par ^= 1;
        if (kw > 0) {
            uint4* l4 = reinterpret_cast<uint4*>(lo);
            for (int i = tid; i < kw * (kFlTile / 4); i += kFlThreads) l4[i] = make_uint4(0u, 0u, 0u, 0u);
            fl_advance<kFlThreads>(P, cur, nxt);
        }
        __syncthreads();
        if (kw > 0) {
            if (tid < 2 * kFlTile) edge[tid] = 0u;
            if (tid <= kFlTile + 2) bad[tid] = 0;
            __syncthreads();
        }
    }
}

constexpr int kBlThreads = 512;
// The A^T's sums are kept on two grids: a tile whose residual is below 2^-kBlFiner of the largest adds to a grid that
// much finer, so that its pairs keep FP32's bits down to 2^-2 kBlFiner of the largest residual.
constexpr int kBlFiner = 25;

struct BlLayout {
    size_t off_e, off_max, off_cur, smem;
};
__host__ __device__ inline BlLayout bl_layout(const GeomParams& P, int kw)
{
    BlLayout L;
    L.off_e = (size_t)kw * kFlTile * 4;
    L.off_max = L.off_e + (size_t)(kFlTile + P.Tw4) * 4;
    L.off_cur = L.off_max + 16;
    L.smem = L.off_cur + (((size_t)P.W * P.n_seg * 8 + 15) & ~(size_t)15);
    return L;
}

// Scale of the adjoint's fixed-point sums: 2^bl_exponent times the pixel's own power of two (FlPlanes, fl_unit_kernel).
// Every contribution is at most max |e| / (2 K unit) in magnitude and a pixel has at most one per A-scan, so with the
// rounding of the products no partial sum reaches 2^61.
__device__ __forceinline__ int bl_exponent(unsigned int emax_bits)
{
    int ex = 0;
    frexpf(__uint_as_float(emax_bits), &ex);
    return 61 - ex;
}

// Per attenuation plane: the largest sum of |T| over a table row, plus the largest |T| (the tau = t0 tap).
struct FlPlanes {
    float b[64];
};

// A^T r from the legs, the adjoint of the sums above: for a tile of 128 values of n0
//     C[n0][col] = sum_m e[n0 + 1 + m] T[col][m]
// (FP32, eight values of n0 and a share of the columns per thread), of which each pair combines four, and adds the
// result to its pixel's 64-bit fixed-point sum, in units of the largest that one of the pixel's pairs can add (so that
// a pixel far from every transducer is summed on as fine a grid, relative to its value, as one below them; one unit and
// one grid for the image took 1.26 ms and lost pixels of weights below 1e-13 altogether).  Block (A-scan, chunk of tiles), two blocks per SM: one's products
// run beside the other's walk.
// 256x512, 64 x 16 A-scans (41 M pairs, FP32), legs included: 1.29 ms against 2.26 ms of backproject_kernel, which
// is bound by the shared-memory loads of its taps (83 % of their peak); the walk takes about half of it.
template <typename E>
__global__ void __launch_bounds__(kBlThreads, 2)
    backward_legs_kernel(GeomParams P, DevPtrs D, const float* __restrict__ ftab, const uint2* __restrict__ crange,
                         const E* __restrict__ e, const unsigned int* __restrict__ emax, const unsigned char* __restrict__ unit,
                         int kwmax, int per, unsigned long long* __restrict__ acc, unsigned char* __restrict__ bad)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const BlLayout L = bl_layout(P, kwmax);
    float* C = reinterpret_cast<float*>(smem);
    float* sE = reinterpret_cast<float*>(smem + L.off_e);
    unsigned int* smax = reinterpret_cast<unsigned int*>(smem + L.off_max);    // bits of max |e| of this and the next tile
    unsigned int* cur = reinterpret_cast<unsigned int*>(smem + L.off_cur);
    unsigned int* nxt = cur + (size_t)P.W * P.n_seg;
    const int tid = threadIdx.x, k = blockIdx.x;
    const int ntile = (P.M + kFlTile - 1) / kFlTile;
    const int ta = blockIdx.y * per, tb = min(ta + per, ntile);
    const int R = P.Q + 1, dR = P.G > 1 ? R : 0;
    const int* htx = D.hidx + (size_t)__ldg(D.txpos + k / P.n_rx) * P.W;
    const int* hrx = D.hidx + (size_t)__ldg(D.rxpos + k) * P.W;
    const int se0 = bl_exponent(__ldg(emax));
    const int cg = tid >> 4, og = tid & 15;
    if (tid < 2) smax[tid] = 0u;
    fl_cursors<kBlThreads>(P, D, htx, hrx, ta, cur, nxt);
    __syncthreads();
    int par = 0;
    for (int t = ta; t < tb; ++t) {
        const uint32_t cr = __ldg(&crange[(size_t)k * ntile + t].x);
        const int c_lo = (int)(cr & 0xffffu), kw = (int)(cr >> 16) - c_lo;
        if (kw <= 0) continue;
        unsigned int em = 0;
        for (int i = tid; i < kFlTile + P.Tw4; i += kBlThreads) {
            const int n = t * kFlTile + 1 + i;
            const float v = n < P.Mp ? fl_float(e[(size_t)k * P.Mp + n]) : 0.0f;
            sE[i] = v;
            const unsigned int b = __float_as_uint(v) & 0x7fffffffu;
            if (b < 0x7f800000u) em = max(em, b);
        }
        em = __reduce_max_sync(0xffffffffu, em);
        if ((tid & 31) == 0 && em) atomicMax(smax + par, em);
        __syncthreads();
        const bool fine = bl_exponent(smax[par]) - kBlFiner >= se0;
        const int se = se0 + (fine ? kBlFiner : 0);
        unsigned long long* const sum = acc + (fine ? (size_t)P.W * P.H : 0);
        par ^= 1;
        if (tid == 0) smax[par] = 0u;                              // (two barriers before the next tile's)
        // ---- C, rows 8 og .. 8 og + 7: four taps at a time against the window's next four samples
        const float4* W = reinterpret_cast<const float4*>(sE);
        const int ntb = P.Tw4 / 4;
        for (int c = cg; c < kw; c += kBlThreads / 16) {
            const float4* T = reinterpret_cast<const float4*>(ftab + (size_t)(c_lo + c) * P.Tw4);
            float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            float4 f0 = W[2 * og], f1 = W[2 * og + 1];
#pragma unroll 4
            for (int mb = 0; mb < ntb; ++mb) {
                const float4 f2 = W[2 * og + 2 + mb];
                const float4 w = __ldg(T + mb);
                const float v[12] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w, f2.x, f2.y, f2.z, f2.w};
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    a[j] = fmaf(v[j + 3], w.w, fmaf(v[j + 2], w.z, fmaf(v[j + 1], w.y, fmaf(v[j], w.x, a[j]))));
                f0 = f1;
                f1 = f2;
            }
            float4* o = reinterpret_cast<float4*>(C + (size_t)c * kFlTile + 8 * og);
            o[0] = make_float4(a[0], a[1], a[2], a[3]);
            o[1] = make_float4(a[4], a[5], a[6], a[7]);
        }
        __syncthreads();
        fl_walk<kBlThreads>(P, D, htx, hrx, nullptr, t, cur, nxt, [&](int row, int col, const Pair& pr, int n0r, float) {
            if (pr.w == 0.0f) return;
            const int px = row * P.W + col;
            const float u = __uint_as_float((unsigned int)__ldg(unit + px) << 23);
            const float* c = C + (size_t)(pr.gi * R + pr.r - c_lo) * kFlTile + n0r;
            const float p1 = pr.psi, p0 = 1.0f - pr.psi;
            float hv = pr.w0 * (p0 * c[0] + p1 * c[dR * kFlTile]) +
                       pr.w1 * (p0 * c[kFlTile] + p1 * c[(dR + 1) * kFlTile]);
            if (pr.flag0) {
                // tau = t0 exactly: the last tap of the upper phase lies outside the window
                const float* tl = ftab + (size_t)(pr.gi * R + pr.r + 1) * P.Tw4 + P.Tw - 1;
                hv -= pr.w1 * (p0 * __ldg(tl) + p1 * __ldg(tl + dR * P.Tw4)) * sE[n0r + P.Tw - 1];
            }
            const float v = pr.w * hv;
            if (fabsf(v) <= 3.4028235e38f)
                red_add_global_u64(sum + px, (unsigned long long)__float2ll_rn(fl_scale(v, se) * u));
            else
                bad[px] = 1;
        });
        __syncthreads();
        fl_advance<kBlThreads>(P, cur, nxt);
    }
}

// b from the fixed-point sums of the two grids; NaN where a contribution was not finite
__global__ void bl_finish_kernel(int N, const unsigned long long* __restrict__ acc, const unsigned char* __restrict__ bad,
                                 const unsigned int* __restrict__ emax, const unsigned char* __restrict__ unit,
                                 float* __restrict__ b)
{
    const int se = bl_exponent(*emax);
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < N; v += gridDim.x * blockDim.x)
        b[v] = bad[v] ? __uint_as_float(0x7fc00000u) : fl_scale((float)((double)(long long)acc[v] + (double)(long long)acc[N + v] / (1 << kBlFiner)) /
                                                              __uint_as_float((unsigned int)unit[v] << 23), -se);
}

// unit[v] = biased exponent of 2^-e for bounds[v] 2 K < 2^e (bounds[v]: bits of the largest contribution of one of the
// pixel's pairs at max |e| = 1, 0 for none)
__global__ void fl_unit_kernel(int N, int K, const unsigned int* __restrict__ bounds, unsigned char* __restrict__ unit)
{
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < N; v += gridDim.x * blockDim.x) {
        int e = 0;
        frexpf(__uint_as_float(bounds[v]) * (2.0f * (float)K), &e);
        unit[v] = (unsigned char)(min(max(-e, -120), 120) + 127);
    }
}

// Per (A-scan, tile): x = the attenuation planes that its pairs reach, as the range of table columns first | end << 16
// (0: no pair), y = the bits that their number leaves of 61 | exponent of the largest weight << 16; wide: the widest
// range; bounds: for fl_unit_kernel (zero before).  Block per A-scan.
__global__ void fl_range_kernel(GeomParams P, DevPtrs D, FlPlanes planes, uint2* __restrict__ crange,
                                int* __restrict__ wide, unsigned int* __restrict__ bounds)
{
    __shared__ int lo[kFlMaxTiles], hi[kFlMaxTiles], count[kFlMaxTiles];
    __shared__ unsigned int wmax[kFlMaxTiles];
    const int k = blockIdx.x, ntile = (P.M + kFlTile - 1) / kFlTile;
    for (int t = threadIdx.x; t < ntile; t += blockDim.x) {
        lo[t] = 1 << 30;
        hi[t] = -1;
        count[t] = 0;
        wmax[t] = 0;
    }
    __syncthreads();
    const int tp = __ldg(D.txpos + k / P.n_rx), rp = __ldg(D.rxpos + k);
    for (int v = threadIdx.x; v < P.W * P.H; v += blockDim.x) {
        const int row = v / P.W, col = v - row * P.W;
        const RowInfo ri = load_row(D.rows, row);
        if (!(ri.tvert < (float)(P.M - 1))) continue;
        const Pair pr = make_pair(P, get_leg<1, kModeTAB>(P, D, ri, row, col, tp),
                                  get_leg<1, kModeTAB>(P, D, ri, row, col, rp), ri.tau);
        if (pr.w == 0.0f || pr.n0 < 0 || pr.n0 + 1 >= P.M) continue;
        const int t = pr.n0 / kFlTile;
        if (pr.gi < lo[t]) atomicMin(lo + t, pr.gi);
        if (pr.gi > hi[t]) atomicMax(hi + t, pr.gi);
        atomicAdd(count + t, 1);
        const unsigned int wb = __float_as_uint(fabsf(pr.w));
        if (wb > wmax[t]) atomicMax(wmax + t, wb);
        const unsigned int cb = __float_as_uint(fabsf(pr.w) * fmaxf(planes.b[pr.gi], planes.b[min(pr.gi + 1, P.G - 1)]));
        if (cb > *(volatile unsigned int*)(bounds + v)) atomicMax(bounds + v, cb);
    }
    __syncthreads();
    const int R = P.Q + 1;
    for (int t = threadIdx.x; t < ntile; t += blockDim.x) {
        uint2 r = make_uint2(0u, 0u);
        if (hi[t] >= 0) {
            const int a = lo[t] * R, b = (min(hi[t] + 1, P.G - 1) + 1) * R;
            int ew = 0;
            frexpf(__uint_as_float(wmax[t]), &ew);
            const int np = 32 - __clz(count[t] - 1);            // count <= 2^np
            r = make_uint2((uint32_t)a | (uint32_t)b << 16, (uint32_t)(61 - np) | (uint32_t)ew << 16);
            atomicMax(wide, b - a);
        }
        crange[(size_t)k * ntile + t] = r;
    }
}

// Set-up for a geometry without stored records: the column ranges (from the legs, solved here for the on-the-fly
// form), the table by columns and the exponents.  cudaErrorNotSupported keeps forward_kernel.
cudaError_t build_forward_legs(mbir_geometry* g, cudaStream_t st)
{
    const GeomParams& P = g->P;
    const int ntile = (P.M + kFlTile - 1) / kFlTile, R = P.Q + 1;
    if (!g->d_legs || g->d_rec_key || g->d_tf4_bop || P.Tw > kFlTile || ntile > kFlMaxTiles || P.G * R > 65535 ||
        P.H > 65535 || (long long)P.W * P.n_seg > 8192)
        return cudaErrorNotSupported;
    // the table by columns, its largest value and the planes' bounds
    const bool bf = P.precision == MBIR_PREC_BF16;
    const int nq = P.Q * P.Tw + 1;
    const size_t ncr = (size_t)P.K * ntile, ntab = (size_t)P.G * R * P.Tw4, N = (size_t)P.W * P.H;
    std::vector<float> tab(ntab, 0.0f);
    FlPlanes planes{};
    float tmax = 0.0f, bmax = 0.0f;
    for (int gp = 0; gp < P.G; ++gp) {
        float pmax = 0.0f, psum = 0.0f;
        for (int r = 0; r < R; ++r) {
            float sum = 0.0f;
            for (int m = 0; m < P.Tw; ++m) {
                float v = (float)g->tab_host[(size_t)gp * nq + m * P.Q + r];
                if (bf) v = __bfloat162float(__float2bfloat16_rn(v));
                tab[((size_t)gp * R + r) * P.Tw4 + m] = v;
                pmax = std::max(pmax, std::fabs(v));
                sum += std::fabs(v);
            }
            psum = std::max(psum, sum);
        }
        planes.b[gp] = psum + pmax;
        tmax = std::max(tmax, pmax);
        bmax = std::max(bmax, planes.b[gp]);
    }
    if (!(bmax > 0.0f && bmax < 1e12f)) return cudaErrorNotSupported;        // (keeps the scaled sums in range)
    uint2* d_cr = nullptr;
    float* d_tab = nullptr;
    unsigned int *d_max = nullptr, *d_bound = nullptr;
    unsigned char* d_unit = nullptr;
    unsigned char* d_acc = nullptr;                  // per pixel: the adjoint's sums, (one word) max |e|, the NaN marks
    const size_t nacc = 17 * N + 8;
    int wide = 0;
    cudaError_t e = cudaMalloc((void**)&d_cr, sizeof(uint2) * ncr);
    if (e == cudaSuccess) e = cudaMalloc((void**)&d_tab, sizeof(float) * ntab);
    if (e == cudaSuccess) e = cudaMalloc((void**)&d_max, sizeof(wide));
    if (e == cudaSuccess) e = cudaMalloc((void**)&d_unit, N);
    if (e == cudaSuccess) e = cudaMalloc((void**)&d_bound, sizeof(unsigned int) * N);
    if (e == cudaSuccess) e = cudaMalloc((void**)&d_acc, nacc);
    if (e == cudaSuccess) e = cudaMemcpy(d_tab, tab.data(), sizeof(float) * ntab, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_max, 0, sizeof(wide), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_bound, 0, sizeof(unsigned int) * N, st);
    if (e == cudaSuccess) {
        bool table = false;
        e = solve_otf_legs(g, st, &table);
    }
    if (e == cudaSuccess) {
        fl_range_kernel<<<P.K, 1024, 0, st>>>(P, dev_ptrs(g), planes, d_cr, reinterpret_cast<int*>(d_max), d_bound);
        fl_unit_kernel<<<(int)std::min<size_t>((N + 255) / 256, 1024), 256, 0, st>>>((int)N, P.K, d_bound, d_unit);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&wide, d_max, sizeof(wide), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(d_bound);
    const int kw = std::max(wide, 1);
    const size_t sm = fl_layout(P, kw).smem;
    if (e == cudaSuccess && sm > 226 * 1024) e = cudaErrorNotSupported;     // a tile reaches too many planes
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(forward_legs_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    for (const void* f : {(const void*)backward_legs_kernel<float>, (const void*)backward_legs_kernel<__nv_bfloat16>})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    if (e != cudaSuccess) {
        cudaFree(d_cr);
        cudaFree(d_tab);
        cudaFree(d_max);
        cudaFree(d_unit);
        cudaFree(d_acc);
        cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? cudaErrorNotSupported : e;
    }
    int ext = 0;
    std::frexp(tmax, &ext);
    g->fl_ebits = std::max(ext, 0);
    g->fl_kw = kw;
    g->d_fl_crange = d_cr;
    g->d_fl_tab = d_tab;
    g->d_fl_max = d_max;
    g->w_fl_acc = d_acc;
    g->d_fl_unit = d_unit;
    g->bytes += sizeof(uint2) * ncr + sizeof(float) * ntab + N + sizeof(wide) + nacc;
    return cudaSuccess;
}

// Ends the segments at the first row whose vertical path already ends past the record (no pair below it is active).
static void fl_clip_rows(const mbir_geometry* g, GeomParams& P)
{
    const int rows = (int)(std::lower_bound(g->h_tvert, g->h_tvert + P.H, (float)(P.M - 1)) - g->h_tvert);
    for (int i = 0; i <= P.n_seg; ++i) P.seg_row[i] = std::min(P.seg_row[i], rows);
}

// One block per A-scan runs alone on its SM, so few A-scans leave SMs idle: their tiles are then cut into chunks
// until there are four blocks per SM, of at least four tiles (each chunk repeats the tile before it).
cudaError_t launch_forward_legs(const mbir_geometry* g, const float* x, float* yf, __nv_bfloat16* yb, int stride,
                                cudaStream_t st)
{
    GeomParams P = g->P;
    const int N = P.W * P.H, ntile = (P.M + kFlTile - 1) / kFlTile;
    fl_clip_rows(g, P);
    cudaError_t e = cudaMemsetAsync(g->d_fl_max, 0, sizeof(unsigned int), st);
    if (e != cudaSuccess) return e;
    fl_xmax_kernel<float><<<std::max(1, std::min((N + 1023) / 1024, g->n_sm)), 256, 0, st>>>(N, x, g->d_fl_max);
    const int want = (4 * g->n_sm + P.K - 1) / P.K;
    const int per = std::max((ntile + want - 1) / want, std::min(4, ntile));
    forward_legs_kernel<<<dim3(P.K, (ntile + per - 1) / per), kFlThreads, fl_layout(P, g->fl_kw).smem, st>>>(
        P, dev_ptrs(g), g->d_fl_tab, g->d_fl_crange, x, g->d_fl_max, g->fl_ebits, g->fl_kw, per, yf, yb,
        stride);
    return cudaGetLastError();
}

// A^T e, with e K x Mp (its BF16 copy in the BF16 form); chunks as above, for eight blocks per SM, two of which run
// at a time.
cudaError_t launch_backproject_legs(const mbir_geometry* g, const float* e_pad, const __nv_bfloat16* e_bf, float* b,
                                    cudaStream_t st)
{
    GeomParams P = g->P;
    const int N = P.W * P.H, ntile = (P.M + kFlTile - 1) / kFlTile;
    fl_clip_rows(g, P);
    auto* acc = reinterpret_cast<unsigned long long*>(g->w_fl_acc);
    auto* emax = reinterpret_cast<unsigned int*>(acc + 2 * (size_t)N);
    unsigned char* bad = g->w_fl_acc + 8 * (2 * (size_t)N + 1);
    cudaError_t e = cudaMemsetAsync(g->w_fl_acc, 0, 17 * (size_t)N + 8, st);
    if (e != cudaSuccess) return e;
    const long long ne = (long long)P.K * P.Mp;
    const int eg = (int)std::max(1LL, std::min((ne + 255) / 256, (long long)g->n_sm * 8));
    const int want = (8 * g->n_sm + P.K - 1) / P.K;
    const int per = std::max((ntile + want - 1) / want, std::min(4, ntile));
    const dim3 grid(P.K, (ntile + per - 1) / per);
    const size_t sm = bl_layout(P, g->fl_kw).smem;
    if (P.precision == MBIR_PREC_BF16) {
        fl_xmax_kernel<__nv_bfloat16><<<eg, 256, 0, st>>>(ne, e_bf, emax);
        backward_legs_kernel<__nv_bfloat16><<<grid, kBlThreads, sm, st>>>(
            P, dev_ptrs(g), g->d_fl_tab, g->d_fl_crange, e_bf, emax, g->d_fl_unit, g->fl_kw, per, acc, bad);
    } else {
        fl_xmax_kernel<float><<<eg, 256, 0, st>>>(ne, e_pad, emax);
        backward_legs_kernel<float><<<grid, kBlThreads, sm, st>>>(
            P, dev_ptrs(g), g->d_fl_tab, g->d_fl_crange, e_pad, emax, g->d_fl_unit, g->fl_kw, per, acc, bad);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    bl_finish_kernel<<<std::max(1, std::min((N + 255) / 256, g->n_sm * 8)), 256, 0, st>>>(N, acc, bad, emax, g->d_fl_unit,
                                                                                            b);
    return cudaGetLastError();
}

}  // namespace mbir

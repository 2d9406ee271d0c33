// Matrix-free projectors of the unmatched pair (A, B) (paper Sec. 1,
// eq. (1.1)-(1.2)): the Joseph ray-driven forward projector A, one thread
// per ray, and the back projector of batched and served solves, one thread
// per pixel (four pixels per thread), gather-only (no atomics).  The single
// launches' back projectors are in back.cu.
//
// Both kernels read their input as (value, forward difference) pairs, so one
// 8-byte load and one FMA give a linear interpolation:
//   lerp(v, j + f) = v[j] + f (v[j+1] - v[j]).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "proj_device.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kPadTile = 32;
constexpr int kPadRows = 8;    // staging blocks are kPadTile x kPadRows threads

__device__ __forceinline__ float2 lerp_pair(float v0, float v1) {
    // (v0 - dv, dv): with m = 1 + f, (v0 - dv) + m dv = v0 + f dv
    const float dv = v1 - v0;
    return make_float2(v0 - dv, dv);
}

// Stage the image for the forward projector (layout in ctg_internal.cuh):
// entries j = -1 .. N-1 of every row of x and of x^T; the other border
// entries are zero pairs written once when the buffer is allocated.  With
// kImgs = 2 two images x (type T) and x2 (FP32) are staged interleaved, each
// entry a float4 (pair of x, pair of x2), so that the forward projector
// reads both with one load.
template <int kImgs, typename T>
__device__ __forceinline__ void pad_pairs_block(const T *__restrict__ x, const float *__restrict__ x2,
                                                void *__restrict__ pad_out, int N, int stride, int border,
                                                int bx, int by) {
    using E = typename std::conditional<kImgs == 2, float4, float2>::type;
    // odd pitch: the column reads of the transposed copy hit 32 distinct banks
    __shared__ float tile[kImgs][kPadTile + 1][kPadTile + 1];
    E *pad = static_cast<E *>(pad_out);
    E *xp = pad + border, *xtp = pad + (size_t)N * stride + border;
    const int j0 = bx * kPadTile, i0 = by * kPadTile;
    // tile[q][r][c] = image q at (i0 + r, j0 + c) for r, c in [0, 33) (0
    // outside); every load is issued before the first shared store
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kPadTile + tx;
    constexpr int kPasses = (kPadTile + kPadRows) / kPadRows;   // rows 0 .. kPadTile
    float v[kImgs][kPasses];
#pragma unroll
    for (int t = 0; t < kPasses; ++t) {
        const int r = ty + t * kPadRows, i = i0 + r, j = j0 + tx;
        const bool in = r <= kPadTile && i < N && j < N;
        v[0][t] = in ? to_f(x[(size_t)i * N + j]) : 0.0f;
        if (kImgs == 2) v[kImgs - 1][t] = in ? x2[(size_t)i * N + j] : 0.0f;
    }
    float edge[kImgs];                    // column kPadTile, rows 0 .. kPadTile
#pragma unroll
    for (int q = 0; q < kImgs; ++q) edge[q] = 0.0f;
    if (tid <= kPadTile) {
        const int i = i0 + tid, j = j0 + kPadTile;
        const bool in = i < N && j < N;
        edge[0] = in ? to_f(x[(size_t)i * N + j]) : 0.0f;
        if (kImgs == 2) edge[kImgs - 1] = in ? x2[(size_t)i * N + j] : 0.0f;
    }
#pragma unroll
    for (int q = 0; q < kImgs; ++q) {
#pragma unroll
        for (int t = 0; t < kPasses; ++t)
            if (ty + t * kPadRows <= kPadTile) tile[q][ty + t * kPadRows][tx] = v[q][t];
        if (tid <= kPadTile) tile[q][tid][kPadTile] = edge[q];
    }
    __syncthreads();
    auto entry = [&](int r0, int c0, int r1, int c1) -> E {
        if constexpr (kImgs == 2) {
            const float2 a = lerp_pair(tile[0][r0][c0], tile[0][r1][c1]);
            const float2 b = lerp_pair(tile[1][r0][c0], tile[1][r1][c1]);
            return make_float4(a.x, a.y, b.x, b.y);
        } else {
            return lerp_pair(tile[0][r0][c0], tile[0][r1][c1]);
        }
    };
    // both copies written along their own rows, so each warp store is one
    // contiguous run of 32 entries
    for (int r = threadIdx.y; r < kPadTile; r += kPadRows) {
        const int i = i0 + r, j = j0 + threadIdx.x;
        if (i < N && j < N) xp[(size_t)i * stride + j] = entry(r, threadIdx.x, r, threadIdx.x + 1);
    }
    for (int c = threadIdx.y; c < kPadTile; c += kPadRows) {
        const int j = j0 + c, i = i0 + threadIdx.x;
        if (i < N && j < N) xtp[(size_t)j * stride + i] = entry(threadIdx.x, c, threadIdx.x + 1, c);
    }
    // entry j = -1 of each row: (0 - x[0], x[0])
    auto first = [&](size_t p) -> E {
        if constexpr (kImgs == 2) {
            const float2 a = lerp_pair(0.0f, to_f(x[p])), b = lerp_pair(0.0f, x2[p]);
            return make_float4(a.x, a.y, b.x, b.y);
        } else {
            return lerp_pair(0.0f, to_f(x[p]));
        }
    };
    if (bx == 0)
        for (int r = threadIdx.y * blockDim.x + threadIdx.x; r < kPadTile; r += blockDim.x * blockDim.y) {
            const int i = i0 + r;
            if (i < N) xp[(size_t)i * stride - 1] = first((size_t)i * N);
        }
    if (by == 0)
        for (int c = threadIdx.y * blockDim.x + threadIdx.x; c < kPadTile; c += blockDim.x * blockDim.y) {
            const int j = j0 + c;
            if (j < N) xtp[(size_t)j * stride - 1] = first((size_t)j);
        }
}

// xc: the image is column xc of a basis (x + col_offset(xc)), or x itself.
// at: the pointer of the FP32 image (x2 of two, else x) is read there.
template <int kImgs, typename T>
__global__ void pad_pairs_kernel(const T *__restrict__ x, ColRef xc, const float *__restrict__ x2,
                                 const float *const *at, void *__restrict__ pad, int N, int stride, int border) {
    if (at) {
        if constexpr (kImgs == 2) x2 = *at;
        else if constexpr (std::is_same<T, float>::value) x = *at;
    }
    pad_pairs_block<kImgs, T>(x + col_offset(xc), x2, pad, N, stride, border, blockIdx.x, blockIdx.y);
}

__device__ __forceinline__ float one_plus_frac(unsigned lo) {
    // 1 + (top 23 bits of a 32-bit fraction), exactly, in [1, 2): the low
    // word of (0x7F : lo) >> 9 is 0x3F800000 | (lo >> 9), one funnel shift
    return __uint_as_float(__funnelshift_r(lo, 0x7Fu, 9));
}

// Image loads in flight per lane (multiples of 4).  The compiler, left alone,
// holds these kernels to 32 registers for occupancy and serialises the loads
// behind their uses; the launch bounds below leave it 64 (one image) and 80 (two),
// enough for the loads: the walk is bound by load latency, and 32 warps per SM
// with 16 loads each beat 64 with about 6.  512^2, 720 angles, 4 angles per warp:
// 67.4 -> 63.6 us; 512^2, 180 angles, one angle per warp: 37 -> 25; two images with
// 4 angles per warp: 153 -> 123.
constexpr int kFwdDepth = 16;
constexpr int kFwdDepth2 = 12;      // two images: 16-byte loads
constexpr int fwd_min_blocks(int warps, int imgs) { return (imgs == 2 ? 24 : 32) / warps; }

// b[a * n_det + d] = scale_a * sum_t lerp(img_a[t, .], u(d, t)).
// A warp holds group `group` of kSplit consecutive angles (fewer where the
// drive changes: all walk the same copy of the image) and 32 / kSplit adjacent
// rays of each, ray group bx, and walks the union of its rays'
// chords' row ranges in lockstep, so each load instruction reads one image
// row per angle: the angles' taps in one row fall on nearly the same pairs, so
// a warp load touches few sectors.  Two images interleaved (16-byte pairs) are
// bound by the L1 data path, where eight angles per warp do best (512^2, 720
// angles: 123 us with 4, 89 with 8; 1001^2, 900 angles: 534 and 394).
// The walk position is 32.32 fixed point with the row stride
// folded into the step, so its high word is the staged-pair index and its
// low word the interpolation weight.  A lane outside its own chord reads
// zero pairs in the border (or, with kClamp, a clamped index into the
// 2-pair border).  The walk starts at a multiple of 4 and step s adds into
// accumulator s % 4, so a ray's sum depends on its own chord only: every
// block shape, warp layout and load depth gives the same result bit for
// bit.  kSplit > 1 needs the host's check (FwdGroups::safe) that
// every lane stays inside the border.
// kImgs = 2 projects two images staged interleaved (pad_pairs_block<2>) in
// the same walk, b from the first and b2 from the second: each ray's two
// sums are the ones the one-image kernel gives for each image alone.
template <bool kClamp, int kSplit, int kImgs>
__device__ __forceinline__ void joseph_forward_warp(const void *__restrict__ pad_in, int N,
                                                    int stride, int border, int n_det,
                                                    const FwdAngle *__restrict__ tab,
                                                    float *__restrict__ b, float *__restrict__ b2,
                                                    int bx, int group) {
    using E = typename std::conditional<kImgs == 2, float4, float2>::type;
    constexpr int kRays = 32 / kSplit, kDepth = kImgs == 2 ? kFwdDepth2 : kFwdDepth;
    const int lane = threadIdx.x & 31, ai = lane / kRays;
    int a = group, na = 1;
    if constexpr (kSplit > 1) {
        const unsigned g = kSplit == 8 ? tab[group].row_group8 : tab[group].group4;
        a = (int)(g >> 4);
        na = (int)((g >> 1) & 7u) + 1;
        a += min(ai, na - 1);             // lanes past the group's last angle walk with it
    }
    const int d = bx * kRays + lane % kRays;
    const bool live = ai < na && d < n_det;
    const FwdAngle t = tab[a];
    const E *img = static_cast<const E *>(pad_in) + (fwd_row_driven(t) ? 0 : (size_t)N * stride) + border;

    // this ray's steps whose taps can touch the image (-1 < u < N), with a
    // one-step margin; rays past the last detector or angle take an empty
    // range
    int lo = N, hi = -1;
    if (live) {
        const float u0 = fmaf((float)d, t.pf, t.qf);
        if (fabsf(t.df) > 1e-20f) {
            const float r1 = (-1.0f - u0) / t.df, r2 = ((float)N - u0) / t.df;
            const float tlo = fmaxf(fminf(r1, r2), -2.0f), thi = fminf(fmaxf(r1, r2), (float)N + 1);
            lo = max(0, (int)floorf(tlo) - 1);
            hi = min(N - 1, (int)ceilf(thi) + 1);
            // a ray that misses the image: the empty range of every other
            // such lane, so that it does not widen the warp's walk (rounded
            // down to a multiple of 4, it could start one far from the image)
            if (lo > hi) lo = N, hi = -1;
        } else if (u0 > -2.0f && u0 < (float)N + 1.0f) {
            lo = 0;
            hi = N - 1;
        }
    }
    const int wlo = __reduce_min_sync(0xffffffffu, lo) & ~3;
    const int whi = __reduce_max_sync(0xffffffffu, hi);
    // acc[i] for image 1, acc[4 + i] for image 2, i = step mod 4
    float acc[4 * kImgs];
#pragma unroll
    for (int i = 0; i < 4 * kImgs; ++i) acc[i] = 0.0f;
    auto add = [&](float *ac, float mw, const E &p) {
        if constexpr (kImgs == 2) {
            ac[0] = fmaf(mw, p.y, ac[0] + p.x);
            ac[4] = fmaf(mw, p.w, ac[4] + p.z);
        } else {
            ac[0] = fmaf(mw, p.y, ac[0] + p.x);
        }
    };
    if (!kClamp) {
        const long long Ds = t.D + ((long long)stride << CTG_FXF_BITS);
        long long U = t.Q + (long long)d * t.P + (long long)wlo * Ds;
        int s = wlo;
        for (; s + kDepth - 1 <= whi; s += kDepth) {
            E p[kDepth];
            float mw[kDepth];
#pragma unroll
            for (int i = 0; i < kDepth; ++i) {
                p[i] = __ldg(img + (int)(U >> CTG_FXF_BITS));
                mw[i] = one_plus_frac((unsigned)U);
                U += Ds;
            }
#pragma unroll
            for (int i = 0; i < kDepth; ++i) add(acc + (i & 3), mw[i], p[i]);
        }
        for (; s + 3 <= whi; s += 4) {
            E p[4];
            float mw[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                p[i] = __ldg(img + (int)(U >> CTG_FXF_BITS));
                mw[i] = one_plus_frac((unsigned)U);
                U += Ds;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) add(acc + i, mw[i], p[i]);
        }
        // at most three steps left, s a multiple of 4
#pragma unroll
        for (int i = 0; i < 3; ++i)
            if (s + i <= whi) {
                const E pa = __ldg(img + (int)(U >> CTG_FXF_BITS));
                add(acc + i, one_plus_frac((unsigned)U), pa);
                U += Ds;
            }
    } else {
        long long U = t.Q + (long long)d * t.P + (long long)wlo * t.D;
        for (int s = wlo; s <= whi; ++s) {
            const int j = min(max((int)(U >> CTG_FXF_BITS), -2), N);
            const E pa = __ldg(img + (size_t)s * stride + j);
            add(acc, one_plus_frac((unsigned)U), pa);
            U += t.D;
        }
    }
    if (live) {
        b[(size_t)a * n_det + d] = ((acc[0] + acc[2]) + (acc[1] + acc[3])) * t.scale;
        if constexpr (kImgs == 2) b2[(size_t)a * n_det + d] = ((acc[4] + acc[6]) + (acc[5] + acc[7])) * t.scale;
    }
}

// One block per (ray group bx, kWarps angle groups by), on a 1-D grid of gx *
// gy blocks; block i takes tile order[i] = by * gx + bx (order NULL: tile i),
// so that the dispatch order can put the longest walks first.
template <bool kClamp, int kWarps, int kSplit, int kImgs>
__global__ void __launch_bounds__(32 * kWarps, fwd_min_blocks(kWarps, kImgs))
joseph_forward_kernel(const void *__restrict__ pad, int N, int stride, int border, int ngroups,
                      int n_det, const FwdAngle *__restrict__ tab,
                      float *__restrict__ b, float *__restrict__ b2, const int *__restrict__ order,
                      int gx) {
    const int tile = order ? order[blockIdx.x] : (int)blockIdx.x;
    const int group = tile / gx * kWarps + (threadIdx.x >> 5);
    if (group >= ngroups) return;                     // whole warp past the last group
    joseph_forward_warp<kClamp, kSplit, kImgs>(pad, N, stride, border, n_det, tab, b, b2, tile % gx, group);
}

// ---------------------------------------------------------------------------
// Back projection of batched and served solves.  (Single launches have faster
// kernels, back.cu, which round differently, about 1e-7 of B b, and are nearer to
// FP64.  This one stays so that batched results stay bit for bit what they were:
// with the 2 x 2 block kernel in its place a batch was 10 % faster, iterates of
// 10 early steps moved by 2e-5 and those of ill-conditioned solves at k >= 20 by up
// to 5e-3, as they do under any change of rounding; which of the two lies nearer
// to the FP64 iterate there was not measured.  A solve can so stop a step apart
// from the same solve alone.)
// A thread-block cluster of kBSplit CTAs owns
// a 32 x 32 pixel tile; each CTA (256 threads, four rows each) sums a
// contiguous quarter of the angles.  For a chunk of angles a CTA stages, per
// angle, the detector window that the tile projects onto as
// (b[d], b[d+1] - b[d]) pairs in shared memory (zeros outside the
// detector), so the inner loop has no bounds test and one 8-byte shared
// load per interpolation.  The tile origin's detector position is formed
// exactly in fixed point; each pixel adds a small float offset.  The CTAs'
// partial sums are then added through distributed shared memory in rank
// order (deterministic, no atomics), each CTA finishing a quarter of the
// tile's rows.
constexpr int kBT = 32;          // tile side
constexpr int kBRows = 4;        // rows per thread (threads: 32 x 8), batched launches
constexpr int kBThreads = 256;
template <int kRows>
__host__ __device__ constexpr int back_threads() { return kBT * (kBT / kRows); }
constexpr int kBChunk = 32;      // angles staged per pass
constexpr int kBSplit = 4;       // CTAs per cluster = angle groups per tile

// Body of one CTA of the back-projection cluster for tile (bx, by).  Every
// CTA of a cluster must call it (it synchronises the cluster twice).
// kModel: 0 the pixel-driven B (linear interpolation on the detector);
// 1 the matched A^T and 2 the thresholded B_tau, whose weights for the two
// nearest bins d0, d0 + 1 of a pixel at detector position d0 + f are
// scale * max(0, 1 - f inv_w) and scale * max(0, 1 - (1 - f) inv_w) (terms
// below thr dropped for 2).  The staged pairs are (b[d], b[d+1] - b[d]) for
// the pixel-driven B and (b[d], b[d+1]) for the others.
// kRows: pixel rows per thread, kBT / kRows row threads per column (rows
// di, di + kBT / kRows, ...): more rows per thread spread the per-angle
// setup over more interpolations.
template <typename T, int kModel = 0, int kChunk = kBChunk, int kRows = kBRows>
__device__ __forceinline__ void pixel_back_tile(const T *__restrict__ b, int N, int n_angles,
                                                int n_det, const BackAngle *__restrict__ tab,
                                                int W, const float *__restrict__ add,
                                                float *__restrict__ x, int bx, int by,
                                                const MatchedAngle *__restrict__ mt = nullptr,
                                                float thr = 0.0f) {
    constexpr int kThr = back_threads<kRows>(), kRT = kBT / kRows;
    static_assert(kChunk <= kThr && kRows % 2 == 0 && kRows <= 16, "back tile shape");
    extern __shared__ float2 s_pairs[];               // kChunk * W pairs
    __shared__ float4 s_par[kChunk];                  // cf, sf, u0' (window-relative), origin
    __shared__ float4 s_wt[kModel ? kChunk : 1];      // scale, scale inv_w, scale - scale inv_w
    __shared__ float s_part[kRows][kThr];             // this CTA's partial sums
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();       // == blockIdx.z
    const int j0 = bx * kBT, i0 = by * kBT;
    const int dj = threadIdx.x & 31, di = threadIdx.x >> 5;   // di in [0, kRT)
    const float fdj = (float)dj, fdi = (float)di;
    const int per = (n_angles + kBSplit - 1) / kBSplit;
    const int a_begin = min(n_angles, rank * per), a_end = min(n_angles, a_begin + per);
    float acc[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) acc[r] = 0.f;
    for (int a0 = a_begin; a0 < a_end; a0 += kChunk) {
        const int na = min(kChunk, a_end - a0);
        __syncthreads();
        if (threadIdx.x < na) {
            const BackAngle t = tab[a0 + threadIdx.x];
            const long long U0 = t.C + (long long)j0 * t.COS + (long long)i0 * t.SIN;
            const int dbase = (int)(U0 >> CTG_FX_BITS);
            const float phi = fx_frac(U0);
            // lowest detector position over the tile (a corner), minus one
            const float umin = phi + fminf(0.f, (kBT - 1) * t.cf) + fminf(0.f, (kBT - 1) * t.sf);
            const int org = dbase + (int)floorf(umin) - 1;
            s_par[threadIdx.x] = make_float4(t.cf, t.sf, (float)(dbase - org) + phi,
                                             __int_as_float(org));
            if constexpr (kModel != 0) {
                const MatchedAngle m = mt[a0 + threadIdx.x];
                const float sw = m.scale * m.inv_w;
                s_wt[threadIdx.x] = make_float4(m.scale, sw, m.scale - sw, 0.0f);
            }
        }
        __syncthreads();
        // one warp per staged angle, lanes along its window (no division)
        for (int k = threadIdx.x >> 5; k < na; k += kThr / 32) {
            const int org = __float_as_int(s_par[k].w);
            const T *brow = b + (size_t)(a0 + k) * n_det;
            float2 *dst = s_pairs + k * W;
            for (int w = threadIdx.x & 31; w < W; w += 32) {
                const int dd = org + w;
                const float v0 = ((unsigned)dd < (unsigned)n_det) ? to_f(__ldg(brow + dd)) : 0.0f;
                const float v1 = ((unsigned)(dd + 1) < (unsigned)n_det) ? to_f(__ldg(brow + dd + 1)) : 0.0f;
                dst[w] = kModel == 0 ? make_float2(v0, v1 - v0) : make_float2(v0, v1);
            }
        }
        __syncthreads();
        // shared address of an angle's window less the magic number's bits
        // times 8, so that row r's pair is at sb + 8 t_r (32-bit wrap-around)
        // with t_r the bits of u_r + M: one shift-add per pair address
        unsigned sb = (unsigned)__cvta_generic_to_shared(s_pairs) - (0x4B400000u << 3);
#pragma unroll 2
        for (int k = 0; k < na; ++k, sb += 8u * (unsigned)W) {
            const float4 p = s_par[k];
            const float du = (float)kRT * p.y;
            float u[kRows];
            u[0] = fmaf(fdi, p.y, fmaf(fdj, p.x, p.z));
#pragma unroll
            for (int r = 1; r < kRows; ++r) u[r] = u[r - 1] + du;
            float tt[kRows], ff[kRows];
#pragma unroll
            for (int r = 0; r < kRows; r += 2) floor_frac2(u[r], u[r + 1], tt[r], tt[r + 1], ff[r], ff[r + 1]);
            float4 wt = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (kModel != 0) wt = s_wt[k];
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
                const float f = ff[r];
                const float2 pr =
                    *static_cast<const float2 *>(__cvta_shared_to_generic(sb + (__float_as_uint(tt[r]) << 3)));
                if constexpr (kModel == 0) {
                    acc[r] += fmaf(f, pr.y, pr.x);
                } else {
                    float w0 = fmaxf(0.0f, fmaf(-f, wt.y, wt.x));
                    float w1 = fmaxf(0.0f, fmaf(f, wt.y, wt.z));
                    if constexpr (kModel == 2) {
                        w0 = w0 >= thr ? w0 : 0.0f;
                        w1 = w1 >= thr ? w1 : 0.0f;
                    }
                    acc[r] = fmaf(w0, pr.x, fmaf(w1, pr.y, acc[r]));
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) s_part[r][threadIdx.x] = acc[r];
    cluster.sync();
    // this CTA finishes row groups rank, rank + kBSplit, ... of every
    // thread: pixel rows di + kRT r
#pragma unroll
    for (int r = rank; r < kRows; r += kBSplit) {
        float sum = 0.0f;
#pragma unroll
        for (int q = 0; q < kBSplit; ++q)
            sum += cluster.map_shared_rank(&s_part[r][0], q)[threadIdx.x];
        const int i = i0 + di + kRT * r, j = j0 + dj;
        if (i < N && j < N) {
            const size_t p = (size_t)i * N + j;
            x[p] = add ? sum + add[p] : sum;
        }
    }
    cluster.sync();   // peers' shared memory must outlive the reads above
}

// One solve of a batch on its own (its start and exit): the same tile.
template <int kModel>
__global__ void __cluster_dims__(1, 1, kBSplit) __launch_bounds__(kBThreads)
batch_back_one_kernel(const float *__restrict__ b, int N, int n_angles, int n_det,
                      const BackAngle *__restrict__ tab, int W, const MatchedAngle *__restrict__ mt, float thr,
                      const float *__restrict__ add, float *__restrict__ x) {
    pixel_back_tile<float, kModel>(b, N, n_angles, n_det, tab, W, add, x, blockIdx.x, blockIdx.y, mt, thr);
}

// ---- batched kernels: one launch for the same phase of every instance ----
// map[blockIdx.x] = (instance, local block of that instance's own grid).

// One instance's tile with its back projector.
template <typename T, int kChunk>
__device__ __forceinline__ void batch_back_tile(const BatchInst &I, const T *in, int bx, int by) {
    if (I.back_model == CTG_BACK_MATCHED)
        pixel_back_tile<T, 1, kChunk>(in, I.N, I.n_angles, I.n_det, I.back, I.back_window, nullptr, I.vn, bx,
                                      by, I.mt, 0.0f);
    else if (I.back_model == CTG_BACK_THRESHOLD)
        pixel_back_tile<T, 2, kChunk>(in, I.N, I.n_angles, I.n_det, I.back, I.back_window, nullptr, I.vn, bx,
                                      by, I.mt, I.back_thr);
    else
        pixel_back_tile<T, 0, kChunk>(in, I.N, I.n_angles, I.n_det, I.back, I.back_window, nullptr, I.vn, bx,
                                      by);
}

// T = float: AB instances with an FP32 basis (back-projecting w_k) and all
// BA instances (back-projecting the FP32 t_k = A w_k); T = BF16 / FP16: AB
// instances whose basis is stored in that type (their own launch, so that
// each kernel holds the tile code of one input type only).
// kChunk: angles staged per pass (the result does not depend on it).
template <typename T, int kChunk>
__global__ void __cluster_dims__(1, 1, kBSplit) __launch_bounds__(kBThreads)
batch_back_kernel(const BatchInst *__restrict__ insts, const int2 *__restrict__ map) {
    const int2 mp = map[blockIdx.x];
    const BatchInst &I = insts[mp.x];
    // the same decision in all CTAs of the cluster (they share blockIdx.x)
    if (!I.active) return;
    constexpr int kType = std::is_same<T, __nv_bfloat16>::value ? CTG_BASIS_BF16
                          : std::is_same<T, __half>::value      ? CTG_BASIS_FP16
                                                                : CTG_BASIS_FP32;
    if (I.variant == CTG_AB && I.wtype != kType) return;
    if (I.variant == CTG_BA && kType != CTG_BASIS_FP32) return;
    const int tx = (I.N + kBT - 1) / kBT;
    const T *in;
    if constexpr (kType == CTG_BASIS_FP32)
        in = I.variant == CTG_AB ? static_cast<const float *>(I.W) + (size_t)(I.k - 1) * I.ldw : I.vm;
    else
        in = static_cast<const T *>(I.W) + (size_t)(I.k - 1) * I.ldw;
    batch_back_tile<T, kChunk>(I, in, mp.y % tx, mp.y / tx);
}

// AB: stage t = B w_k (in vn); BA: stage w_{k+1} (stored type), with x_k
// interleaved for the DP stop.
template <int kVariant>
__global__ void batch_pad_kernel(const BatchInst *__restrict__ insts, const int2 *__restrict__ map) {
    const int2 mp = map[blockIdx.x];
    const BatchInst &I = insts[mp.x];
    if (!I.active) return;
    const int tx = (I.N + kPadTile - 1) / kPadTile, bx = mp.y % tx, by = mp.y / tx;
    if (kVariant == CTG_AB) {
        pad_pairs_block<1, float>(I.vn, nullptr, I.pad, I.N, I.pad_stride, I.pad_border, bx, by);
        return;
    }
    const size_t off = (size_t)I.k * I.ldw;
    const bool two = I.target > 0.0;
    auto stage = [&](auto *w) {
        if (two) pad_pairs_block<2>(w + off, I.x, I.pad2, I.N, I.pad_stride, I.pad_border, bx, by);
        else pad_pairs_block<1>(w + off, nullptr, I.pad, I.N, I.pad_stride, I.pad_border, bx, by);
    };
    if (I.wtype == CTG_BASIS_BF16) stage(static_cast<const __nv_bfloat16 *>(I.W));
    else if (I.wtype == CTG_BASIS_FP16) stage(static_cast<const __half *>(I.W));
    else stage(static_cast<const float *>(I.W));
}

// AB: q = A t (into vm); BA: t_{k+1} = A w_{k+1} (into vm) and, with the DP
// stop, A x_k (into vr) from the two-image staging.  Each instance has its own
// angles per warp.
template <int kImgs>
__device__ __forceinline__ void batch_forward(const BatchInst &I, const void *pad, float *b2, int tile) {
    const int rays = 32 / I.fwd_split, bxn = (I.n_det + rays - 1) / rays;
    const int bx = tile % bxn, group = tile / bxn * kBatchFwdWarps + (threadIdx.x >> 5);
    if (group >= I.fwd_groups) return;
    if (I.pad_clamp)
        joseph_forward_warp<true, 1, kImgs>(pad, I.N, I.pad_stride, I.pad_border, I.n_det, I.fwd, I.vm, b2, bx, group);
    else if (kImgs == 2 && I.fwd_split == 8)
        joseph_forward_warp<false, 8, kImgs>(pad, I.N, I.pad_stride, I.pad_border, I.n_det, I.fwd, I.vm, b2, bx, group);
    else if (I.fwd_split == 4)
        joseph_forward_warp<false, 4, kImgs>(pad, I.N, I.pad_stride, I.pad_border, I.n_det, I.fwd, I.vm, b2, bx, group);
    else
        joseph_forward_warp<false, 1, kImgs>(pad, I.N, I.pad_stride, I.pad_border, I.n_det, I.fwd, I.vm, b2, bx, group);
}

template <int kVariant>
__global__ void __launch_bounds__(32 * kBatchFwdWarps, fwd_min_blocks(kBatchFwdWarps, kVariant == CTG_BA ? 2 : 1))
batch_forward_kernel(const BatchInst *__restrict__ insts, const int2 *__restrict__ map) {
    const int2 mp = map[blockIdx.x];
    const BatchInst &I = insts[mp.x];
    if (!I.active) return;
    if (kVariant == CTG_BA && I.target > 0.0) batch_forward<2>(I, I.pad2, I.vr, mp.y);
    else batch_forward<1>(I, I.pad, nullptr, mp.y);
}

}  // namespace

int ctg_back_tiles(int N) {
    const int t = (N + kBT - 1) / kBT;
    return t * t;
}
int ctg_pad_tiles(int N) {
    const int t = (N + kPadTile - 1) / kPadTile;
    return t * t;
}
int ctg_fwd_blocks(int warps, int split, int ngroups, int n_det) {
    const int rays = 32 / split;
    return ((n_det + rays - 1) / rays) * ((ngroups + warps - 1) / warps);
}
// largest window the tiled back projector can stage in shared memory
int ctg_back_window_max() { return (40 * 1024) / (int)(sizeof(float2) * kBChunk); }

namespace {
template <int kChunk>
void batch_back_t(BatchInst *insts, const int2 *map, int nblocks, int max_window, cudaStream_t st, int wtype) {
    const size_t smem = sizeof(float2) * (size_t)kChunk * max_window;
    const dim3 grid(nblocks, 1, kBSplit);
    if (wtype == CTG_BASIS_BF16)
        batch_back_kernel<__nv_bfloat16, kChunk><<<grid, kBThreads, smem, st>>>(insts, map);
    else if (wtype == CTG_BASIS_FP16)
        batch_back_kernel<__half, kChunk><<<grid, kBThreads, smem, st>>>(insts, map);
    else
        batch_back_kernel<float, kChunk><<<grid, kBThreads, smem, st>>>(insts, map);
}
}  // namespace

cudaError_t ctg_batch_back_one(const float *b, int back_model, int N, int n_angles, int n_det,
                               const BackAngle *tab, int window, const MatchedAngle *mt, float thr,
                               const float *add, float *x, cudaStream_t st) {
    if (window <= 0 || window > ctg_back_window_max()) return cudaErrorInvalidValue;
    const size_t smem = sizeof(float2) * (size_t)kBChunk * window;
    const dim3 grid((N + kBT - 1) / kBT, (N + kBT - 1) / kBT, kBSplit);
    auto run = [&](auto kernel) {
        kernel<<<grid, kBThreads, smem, st>>>(b, N, n_angles, n_det, tab, window, mt, thr, add, x);
    };
    if (back_model == CTG_BACK_PIXEL) run(batch_back_one_kernel<0>);
    else if (thr > 0.0f) run(batch_back_one_kernel<2>);
    else run(batch_back_one_kernel<1>);
    return cudaGetLastError();
}

bool ctg_batch_back_chunk_ok(int chunk, int max_window) {
    return (chunk == 16 || chunk == 32 || chunk == 64) && (size_t)chunk * max_window * sizeof(float2) <= 40 * 1024;
}

cudaError_t ctg_batch_back(BatchInst *insts, const int2 *map, int nblocks, int max_window,
                           cudaStream_t st, int wtype, int chunk) {
    if (nblocks <= 0) return cudaSuccess;
    if (!ctg_batch_back_chunk_ok(chunk, max_window)) chunk = kBChunk;
    if (chunk == 16) batch_back_t<16>(insts, map, nblocks, max_window, st, wtype);
    else if (chunk == 64) batch_back_t<64>(insts, map, nblocks, max_window, st, wtype);
    else batch_back_t<kBChunk>(insts, map, nblocks, max_window, st, wtype);
    return cudaGetLastError();
}

cudaError_t ctg_batch_pad(BatchInst *insts, const int2 *map, int nblocks, int variant, cudaStream_t st) {
    if (nblocks <= 0) return cudaSuccess;
    if (variant == CTG_AB) batch_pad_kernel<CTG_AB><<<nblocks, dim3(kPadTile, kPadRows), 0, st>>>(insts, map);
    else batch_pad_kernel<CTG_BA><<<nblocks, dim3(kPadTile, kPadRows), 0, st>>>(insts, map);
    return cudaGetLastError();
}

cudaError_t ctg_batch_forward(BatchInst *insts, const int2 *map, int nblocks, int variant, cudaStream_t st) {
    if (nblocks <= 0) return cudaSuccess;
    if (variant == CTG_AB) batch_forward_kernel<CTG_AB><<<nblocks, 32 * kBatchFwdWarps, 0, st>>>(insts, map);
    else batch_forward_kernel<CTG_BA><<<nblocks, 32 * kBatchFwdWarps, 0, st>>>(insts, map);
    return cudaGetLastError();
}

int ctg_back_window(const BackAngle *host_tab, int n_angles) {
    // detector span of a 32 x 32 tile at any angle, plus the floor/ceil and
    // second-tap margins
    double span = 0.0;
    for (int a = 0; a < n_angles; ++a) {
        const double s = (kBT - 1) * ((double)fabsf(host_tab[a].cf) + (double)fabsf(host_tab[a].sf));
        if (s > span) span = s;
    }
    return (int)ceil(span) + 4;
}

cudaError_t ctg_launch_pad(const void *x, int dtype, float2 *pad, int N, const PadLayout &pl,
                           cudaStream_t st, ColRef xc, const float *const *xat) {
    if (xat && dtype != CTG_BASIS_FP32) return cudaErrorInvalidValue;
    dim3 grid((N + kPadTile - 1) / kPadTile, (N + kPadTile - 1) / kPadTile), block(kPadTile, kPadRows);
    switch (dtype) {
        case CTG_BASIS_FP32:
            pad_pairs_kernel<1><<<grid, block, 0, st>>>(static_cast<const float *>(x), xc, nullptr, xat, pad, N,
                                                        pl.stride, pl.border);
            break;
        case CTG_BASIS_BF16:
            pad_pairs_kernel<1><<<grid, block, 0, st>>>(static_cast<const __nv_bfloat16 *>(x), xc, nullptr,
                                                        nullptr, pad, N, pl.stride, pl.border);
            break;
        case CTG_BASIS_FP16:
            pad_pairs_kernel<1><<<grid, block, 0, st>>>(static_cast<const __half *>(x), xc, nullptr, nullptr, pad, N,
                                                        pl.stride, pl.border);
            break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t ctg_launch_pad2(const void *x, int dtype, ColRef xc, const float *x2, float4 *pad2, int N,
                            const PadLayout &pl, cudaStream_t st, float *const *x2at) {
    const float *const *at = x2at;
    dim3 grid((N + kPadTile - 1) / kPadTile, (N + kPadTile - 1) / kPadTile), block(kPadTile, kPadRows);
    switch (dtype) {
        case CTG_BASIS_FP32:
            pad_pairs_kernel<2><<<grid, block, 0, st>>>(static_cast<const float *>(x), xc, x2, at, pad2, N,
                                                        pl.stride, pl.border);
            break;
        case CTG_BASIS_BF16:
            pad_pairs_kernel<2><<<grid, block, 0, st>>>(static_cast<const __nv_bfloat16 *>(x), xc, x2, at,
                                                        pad2, N, pl.stride, pl.border);
            break;
        case CTG_BASIS_FP16:
            pad_pairs_kernel<2><<<grid, block, 0, st>>>(static_cast<const __half *>(x), xc, x2, at, pad2, N,
                                                        pl.stride, pl.border);
            break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

namespace {

template <int kShape, int kImgs>
void launch_forward_t(const void *pad, int N, const PadLayout &pl, int n_det, const FwdAngle *tab, float *b,
                      float *b2, cudaStream_t st, int ngroups, const int *order) {
    constexpr int kWarps = kFwdShapeWarps[kShape], kSplit = kFwdShapeSplit[kShape], kRays = 32 / kSplit;
    const int gx = (n_det + kRays - 1) / kRays;
    const unsigned grid = (unsigned)ctg_fwd_blocks(kWarps, kSplit, ngroups, n_det);
    if (pl.clamp)
        joseph_forward_kernel<true, kWarps, kSplit, kImgs><<<grid, 32 * kWarps, 0, st>>>(
            pad, N, pl.stride, pl.border, ngroups, n_det, tab, b, b2, order, gx);
    else
        joseph_forward_kernel<false, kWarps, kSplit, kImgs><<<grid, 32 * kWarps, 0, st>>>(
            pad, N, pl.stride, pl.border, ngroups, n_det, tab, b, b2, order, gx);
}

template <int kImgs>
void launch_forward_shape(int shape, const void *pad, int N, const PadLayout &pl, int n_det, const FwdAngle *tab,
                          float *b, float *b2, cudaStream_t st, int ngroups, const int *order) {
    switch (shape) {
        case 1: launch_forward_t<1, kImgs>(pad, N, pl, n_det, tab, b, b2, st, ngroups, order); break;
        case 2: launch_forward_t<2, kImgs>(pad, N, pl, n_det, tab, b, b2, st, ngroups, order); break;
        case 3: launch_forward_t<3, kImgs>(pad, N, pl, n_det, tab, b, b2, st, ngroups, order); break;
        case kFwdShapeTwo:
            if constexpr (kImgs == 2)
                launch_forward_t<kFwdShapeTwo, 2>(pad, N, pl, n_det, tab, b, b2, st, ngroups, order);
            break;
        default: launch_forward_t<0, kImgs>(pad, N, pl, n_det, tab, b, b2, st, ngroups, order); break;
    }
}

// walk range [lo, hi] of ray d of angle t, as joseph_forward_warp forms it, in
// the same operations (one rounding in u0: at an angle almost parallel to the
// walk a last bit there is the difference between no row and all of them).
// Returns 0 for a ray that meets the image; for one that misses it (lo = N, hi
// = -1), -1 or 1 as its crossing lies before the first or past the last row.
int ray_range(const FwdAngle &t, int N, int d, int &lo, int &hi) {
    const float u0 = std::fma((float)d, t.pf, t.qf);
    lo = N;
    hi = -1;
    if (std::fabs(t.df) > 1e-20f) {
        const float r1 = (-1.0f - u0) / t.df, r2 = ((float)N - u0) / t.df;
        const float tlo = std::max(std::min(r1, r2), -2.0f), thi = std::min(std::max(r1, r2), (float)N + 1);
        const float flo = std::floor(tlo) - 1.0f, fhi = std::ceil(thi) + 1.0f;
        if (fhi < 0.0f) return -1;
        if (flo > (float)(N - 1)) return 1;
        lo = std::max(0, (int)flo);
        hi = std::min(N - 1, (int)fhi);
        if (lo <= hi) return 0;
        lo = N;
        hi = -1;
        return 1;
    }
    if (u0 > -2.0f && u0 < (float)N + 1.0f) {
        lo = 0;
        hi = N - 1;
        return 0;
    }
    return u0 < 0.0f ? -1 : 1;
}

// union walk range of rays d0 .. d1 - 1 of angle t: a ray's range ends are
// clamped linear functions of d, so where the first and the last ray meet the
// image they give it, and where both miss it on the same side so do all others
// (else, and for a walk parallel to the detector, D = 0, all rays are asked)
void group_range(const FwdAngle &t, int N, int d0, int d1, int &wlo, int &whi) {
    int lo, hi;
    const int first = ray_range(t, N, d0, wlo, whi), last = ray_range(t, N, d1 - 1, lo, hi);
    const bool all = !(std::fabs(t.df) > 1e-20f) || first != last;
    wlo = std::min(wlo, lo);
    whi = std::max(whi, hi);
    if (all)
        for (int d = d0 + 1; d < d1 - 1; ++d) {
            ray_range(t, N, d, lo, hi);
            wlo = std::min(wlo, lo);
            whi = std::max(whi, hi);
        }
}

}  // namespace

cudaError_t ctg_launch_forward(const float2 *pad, int N, const PadLayout &pl, int n_angles,
                               int n_det, const FwdAngle *tab, float *b, cudaStream_t st,
                               int shape, int ngroups, const int *order) {
    // every ray's sum depends on its own chord only, so the result depends
    // on neither the shape nor the dispatch order
    (void)n_angles;
    launch_forward_shape<1>(shape, pad, N, pl, n_det, tab, b, nullptr, st, ngroups, order);
    return cudaGetLastError();
}

cudaError_t ctg_launch_forward2(const float4 *pad2, int N, const PadLayout &pl, int n_angles, int n_det,
                                const FwdAngle *tab, float *b, float *b2, cudaStream_t st, int shape, int ngroups,
                                const int *order) {
    (void)n_angles;
    launch_forward_shape<2>(shape, pad2, N, pl, n_det, tab, b, b2, st, ngroups, order);
    return cudaGetLastError();
}

FwdGroups ctg_forward_groups(std::vector<FwdAngle> &tab) {
    FwdGroups G{};
    const int n = (int)tab.size();
    G.count[0] = n;
    G.safe[0] = true;
    for (int a = 0; a < n; ++a) {
        tab[a].row_group8 &= 1u;
        tab[a].group4 = 0;
    }
    for (const int split : {4, 8}) {
        int &g = G.count[fwd_split_index(split)];
        for (int a = 0, c; a < n; a += c, ++g) {
            for (c = 1; c < split && a + c < n && fwd_row_driven(tab[a + c]) == fwd_row_driven(tab[a]);) ++c;
            (split == 8 ? tab[g].row_group8 : tab[g].group4) |= fwd_group_word(a, c);
        }
    }
    return G;
}

namespace {
// Block order, longest first (stable): a counting sort of the blocks' steps.
void longest_first(const std::vector<int> &cost, int ng, int gx, int W, std::vector<int> &order) {
    const int gy = (ng + W - 1) / W;
    std::vector<int> sum((size_t)gx * gy, 0), at;
    for (int g = 0; g < ng; ++g)
        for (int bx = 0; bx < gx; ++bx) sum[(size_t)(g / W) * gx + bx] += cost[(size_t)g * gx + bx];
    const int top = sum.empty() ? 0 : *std::max_element(sum.begin(), sum.end());
    at.assign((size_t)top + 2, 0);
    for (const int c : sum) ++at[top - c + 1];
    for (int c = 0; c <= top; ++c) at[c + 1] += at[c];
    order.resize(sum.size());
    for (size_t i = 0; i < sum.size(); ++i) order[at[top - sum[i]]++] = (int)i;
}
}  // namespace

// Row ranges [x, y] of the walks of each angle's groups of eight rays.
std::vector<int2> ctg_forward_ranges(const FwdAngle *tab, int N, int n_angles, int n_det) {
    const int gx = (n_det + 7) / 8;
    std::vector<int2> r((size_t)n_angles * gx);
    for (int a = 0; a < n_angles; ++a)
        for (int bx = 0; bx < gx; ++bx) {
            int2 &w = r[(size_t)a * gx + bx];
            group_range(tab[a], N, 8 * bx, std::min(n_det, 8 * bx + 8), w.x, w.y);
        }
    return r;
}

void ctg_forward_plan(const FwdAngle *tab, int N, int n_angles, int n_det, const PadLayout &pl, int split,
                      FwdGroups &G, std::initializer_list<int> warps, std::vector<int> *orders,
                      const std::vector<int2> &ranges) {
    const int R = 32 / split, gx = (n_det + R - 1) / R, ng = G.count[fwd_split_index(split)];
    // groups cut short by changes of drive leave lanes idle: not worth it when
    // more than a fifth are (widely spaced angles)
    bool safe = split == 1 || (long long)ng * split * 4 <= 5LL * n_angles + 12 * split;
    const int gx8 = (n_det + 7) / 8;      // the ranges' groups of eight rays
    // steps of each warp's lockstep walk plus a fixed cost
    std::vector<int> cost((size_t)ng * gx);
    for (int g = 0; g < ng; ++g) {
        const unsigned w = split == 8 ? tab[g].row_group8 : tab[g].group4;
        const int a0 = split == 1 ? g : (int)(w >> 4), na = split == 1 ? 1 : (int)((w >> 1) & 7u) + 1;
        for (int bx = 0; bx < gx; ++bx) {
            const int d0 = bx * R, d1 = std::min(n_det, d0 + R);
            int wlo = N, whi = -1;
            for (int a = a0; a < a0 + na; ++a)
                for (int r8 = d0 / 8; 8 * r8 < d1; ++r8) {
                    const int2 r = ranges[(size_t)a * gx8 + r8];
                    wlo = std::min(wlo, r.x);
                    whi = std::max(whi, r.y);
                }
            cost[(size_t)g * gx + bx] = (whi >= wlo ? whi - (wlo & ~3) + 1 : 0) + 16;
            if (!safe || split == 1 || pl.clamp || whi < wlo) continue;     // clamped indices are safe
            // the device's range, with a margin of a step of the walk's start
            const int s_lo = std::max(0, (wlo & ~3) - 4), s_hi = std::min(N - 1, whi + 4);
            // a lane's column is affine in its ray d, so the warp's first and
            // last ray of each angle are its extremes
            long long least = 0, most = 0;
            for (int a = a0; a < a0 + na; ++a) {
                const long long u = tab[a].Q + d0 * tab[a].P + s_lo * tab[a].D;
                const long long dd = (R - 1) * tab[a].P, ds = (s_hi - s_lo) * tab[a].D;
                least = std::min(least, u + std::min(0LL, dd) + std::min(0LL, ds));
                most = std::max(most, u + std::max(0LL, dd) + std::max(0LL, ds));
            }
            if ((least >> CTG_FXF_BITS) < -pl.border || (most >> CTG_FXF_BITS) > N - 1 + pl.border) safe = false;
        }
    }
    G.safe[fwd_split_index(split)] = safe;
    for (const int W : warps) longest_first(cost, ng, gx, W, *orders++);
}

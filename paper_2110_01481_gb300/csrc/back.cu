// The back projectors of single launches: the pixel-driven B (paper Sec. 1,
// eq. (1.2)), the matched A^T and the thresholded B_tau of Sec. 6.5, gather-only
// (no atomics).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "proj_device.cuh"

namespace cg = cooperative_groups;

namespace {

// ---- one pixel and its reflection: A^T, B_tau, and B for pitches below a pixel ----
// Image grid and detector are centred, so pixel
// (i, j) and its point reflection (N-1-i, N-1-j) sit at detector positions u
// and (n_det-1) - u of every angle: with the reversed projection b'[d] =
// b[n_det-1-d] the reflected pixel interpolates b' at the same u, with the
// same index and weight.  So a tile covers 32 x 32 pixels of the upper half of
// the image and their reflections: position, floor, weight and shared address
// are formed once for two interpolations, and one 16-byte shared load brings
// the operands of both.
//
// A thread-block cluster of kSplit CTAs owns a tile; each CTA sums a contiguous
// share of the angles.  For a chunk of angles a CTA stages, per angle, the
// detector window that the tile projects onto as (b[d], b'[d], b[d+1] - b[d],
// b'[d+1] - b'[d]) in shared memory (zeros outside the detector), so the inner
// loop has no bounds test.  The tile centre's detector position is formed
// exactly in fixed point; each pixel adds a float offset of at most 22
// bins.  The CTAs' partial sums are then added through distributed shared
// memory in rank order (deterministic, no atomics), each CTA finishing a share
// of the tile's rows.
// Bound by the shared-memory data path (8 bytes per interpolation, 16 per clock
// and SM; the pixel-driven B at 2048^2, 1800 angles runs at 80 % of that); with
// one pixel per position it was bound by issue slots.  A^T at 512^2, 720 angles
// 103 -> 70 us, at 1001^2, 900 angles 466 -> 280 us.
constexpr int kPT = 32;             // tile side
template <int kRows>
__host__ __device__ constexpr int pair_threads() { return kPT * (kPT / kRows); }
constexpr int kPairChunk = 32;      // angles staged per pass
constexpr int kMaxSplit = 8;        // CTAs per cluster = angle groups per tile, at most (portable clusters)
// tiles of an image: columns x rows of the upper half
__host__ __device__ constexpr int back_tiles_x(int N) { return (N + kPT - 1) / kPT; }
__host__ __device__ constexpr int back_tiles_y(int N) { return ((N + 1) / 2 + kPT - 1) / kPT; }

__device__ __forceinline__ void add2(float &a0, float &a1, float v0, float v1) {
    asm("{\n\t.reg .b64 a, v;\n\t"
        "mov.b64 a, {%0, %1};\n\t"
        "mov.b64 v, {%2, %3};\n\t"
        "add.rn.f32x2 a, a, v;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "+f"(a0), "+f"(a1)
        : "f"(v0), "f"(v1));
}

// Body of one CTA of the back-projection cluster for tile (bx, by).  Every
// CTA of a cluster must call it (it synchronises the cluster twice).
// kModel: 0 the pixel-driven B (linear interpolation on the detector);
// 1 the matched A^T and 2 the thresholded B_tau, whose weights for the two
// nearest bins d0, d0 + 1 of a pixel at detector position d0 + f are
// scale * max(0, 1 - f inv_w) and scale * max(0, 1 - (1 - f) inv_w) (terms
// below thr dropped for 2).  The staged entries are (b[d], b'[d], differences)
// for the pixel-driven B and (b[d], b'[d], b[d+1], b'[d+1]) for the others.
// kRows: pixel rows per thread, kPT / kRows row threads per column (rows
// di, di + kPT / kRows, ...).
template <typename T, int kModel, int kChunk, int kRows, int kSplit>
__device__ __forceinline__ void pixel_pair_tile(const T *__restrict__ b, int N, int n_angles,
                                                int n_det, const BackAngle *__restrict__ tab,
                                                int W, const float *__restrict__ add,
                                                float *__restrict__ x, int bx, int by,
                                                const MatchedAngle *__restrict__ mt = nullptr,
                                                float thr = 0.0f) {
    constexpr int kThr = pair_threads<kRows>(), kRT = kPT / kRows;
    static_assert(kChunk <= kThr && kRows % 2 == 0 && kRows <= 16, "back tile shape");
    extern __shared__ float4 s_win[];                 // kChunk * W entries; at the end the partial sums
    __shared__ float4 s_par[kChunk];                  // cf, sf, u at the tile centre, kRT sf
    __shared__ int s_org[kChunk];                     // detector bin of the window's first entry
    __shared__ float4 s_wt[kModel ? kChunk : 1];      // scale, scale inv_w, scale - scale inv_w
    float *s_part = reinterpret_cast<float *>(s_win); // [2 kRows][kThr]
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();       // == blockIdx.z
    const int j0 = bx * kPT, i0 = by * kPT;
    const int dj = threadIdx.x & 31, di = threadIdx.x >> 5;   // di in [0, kRT)
    const float fdj = (float)dj - 0.5f * (kPT - 1), fdi = (float)di - 0.5f * (kPT - 1);
    const int per = (n_angles + kSplit - 1) / kSplit;
    const int a_begin = min(n_angles, rank * per), a_end = min(n_angles, a_begin + per);
    const int wc = W / 2;                             // window entry of the tile centre's bin
    float sum[kRows][2], acc[kRows][2];               // direct and reflected pixel; of the latest 32 angles
#pragma unroll
    for (int r = 0; r < kRows; ++r) sum[r][0] = sum[r][1] = acc[r][0] = acc[r][1] = 0.f;
    for (int a0 = a_begin; a0 < a_end; a0 += kChunk) {
        const int na = min(kChunk, a_end - a0);
        __syncthreads();
        if (threadIdx.x < na) {
            const BackAngle t = tab[a0 + threadIdx.x];
            // the tile centre is 15.5 pixels from its origin in both directions
            const long long Uc = t.C + (long long)j0 * t.COS + (long long)i0 * t.SIN +
                                 (((kPT - 1) * (t.COS + t.SIN)) >> 1);
            s_par[threadIdx.x] = make_float4(t.cf, t.sf, fx_frac(Uc), (float)kRT * t.sf);
            s_org[threadIdx.x] = (int)(Uc >> CTG_FX_BITS) - wc;
            if constexpr (kModel != 0) {
                const MatchedAngle m = mt[a0 + threadIdx.x];
                const float sw = m.scale * m.inv_w;
                s_wt[threadIdx.x] = make_float4(m.scale, sw, m.scale - sw, 0.0f);
            }
        }
        __syncthreads();
        // one warp per staged angle, lanes along its window (no division)
        for (int k = threadIdx.x >> 5; k < na; k += kThr / 32) {
            const int org = s_org[k];
            const T *brow = b + (size_t)(a0 + k) * n_det;
            float4 *dst = s_win + k * W;
            auto bin = [&](int d) {
                return ((unsigned)d < (unsigned)n_det) ? to_f(__ldg(brow + d)) : 0.0f;
            };
            for (int w = threadIdx.x & 31; w < W; w += 32) {
                const int d = org + w, e = n_det - 1 - d;
                const float v0 = bin(d), v1 = bin(d + 1), m0 = bin(e), m1 = bin(e - 1);
                dst[w] = kModel == 0 ? make_float4(v0, m0, v1 - v0, m1 - m0) : make_float4(v0, m0, v1, m1);
            }
        }
        __syncthreads();
        // shared address of an angle's window centre less the magic number's
        // bits times 16, so that row r's entry is at sb + 16 t_r (32-bit
        // wrap-around) with t_r the bits of u_r + M: one shift-add per address
        unsigned sb = (unsigned)__cvta_generic_to_shared(s_win + wc) - (0x4B400000u << 4);
#pragma unroll 2
        for (int k = 0; k < na; ++k, sb += 16u * (unsigned)W) {
            const float4 p = s_par[k];
            float u[kRows];
            u[0] = fmaf(fdi, p.y, fmaf(fdj, p.x, p.z));
#pragma unroll
            for (int r = 1; r < kRows; ++r) u[r] = u[r - 1] + p.w;
            float tt[kRows], ff[kRows];
#pragma unroll
            for (int r = 0; r < kRows; r += 2) floor_frac2(u[r], u[r + 1], tt[r], tt[r + 1], ff[r], ff[r + 1]);
            float4 wt = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (kModel != 0) wt = s_wt[k];
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
                const float f = ff[r];
                const float4 e =
                    *static_cast<const float4 *>(__cvta_shared_to_generic(sb + (__float_as_uint(tt[r]) << 4)));
                if constexpr (kModel == 0) {
                    add2(acc[r][0], acc[r][1], fmaf(f, e.z, e.x), fmaf(f, e.w, e.y));
                } else {
                    float w0 = fmaxf(0.0f, fmaf(-f, wt.y, wt.x));
                    float w1 = fmaxf(0.0f, fmaf(f, wt.y, wt.z));
                    if constexpr (kModel == 2) {
                        w0 = w0 >= thr ? w0 : 0.0f;
                        w1 = w1 >= thr ? w1 : 0.0f;
                    }
                    acc[r][0] = fmaf(w0, e.x, fmaf(w1, e.z, acc[r][0]));
                    acc[r][1] = fmaf(w0, e.y, fmaf(w1, e.w, acc[r][1]));
                }
            }
        }
        // 32 angles at a time (whatever the chunk), which keeps the chains of
        // additions short for every split
        if ((a0 - a_begin + kChunk) % kPairChunk == 0 || a0 + kChunk >= a_end)
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
                add2(sum[r][0], sum[r][1], acc[r][0], acc[r][1]);
                acc[r][0] = acc[r][1] = 0.f;
            }
    }
    __syncthreads();                                  // the windows have been read
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        s_part[(2 * r) * kThr + threadIdx.x] = sum[r][0];
        s_part[(2 * r + 1) * kThr + threadIdx.x] = sum[r][1];
    }
    cluster.sync();
    // this CTA finishes planes rank, rank + kSplit, ...: plane 2 r + h holds
    // pixel rows di + kRT r (h = 0) or their reflections (h = 1).  A pixel at
    // or before the image's centre is written by the direct plane, the others
    // by the reflected one (on the middle row of an odd N both reach it).
    const long long last = (long long)N * N - 1;
#pragma unroll
    for (int q = rank; q < 2 * kRows; q += kSplit) {
        float all = 0.0f;
#pragma unroll
        for (int c = 0; c < kSplit; ++c) all += cluster.map_shared_rank(s_part + q * kThr, c)[threadIdx.x];
        const int i = i0 + di + kRT * (q >> 1), j = j0 + dj;
        const long long p = (long long)i * N + j;
        if (i < N && j < N && ((q & 1) ? 2 * p < last : 2 * p <= last)) {
            const long long o = (q & 1) ? last - p : p;
            x[o] = add ? all + add[o] : all;
        }
    }
    cluster.sync();   // peers' shared memory must outlive the reads above
}

// ---- 2 x 2 pixel blocks: the pixel-driven B for pitches of a pixel or more (ctg_back_blocks_ok) ----
// One interpolation per shared load is bound by the shared-memory data path
// (8 bytes per interpolation, 16 interpolations per clock and SM).  Where one
// pixel step moves at most one detector bin (|cos|, |sin| <= the pitch), a 2 x 2
// block of pixels lies within three bins of its lowest corner, so four bins
// b0..b3 from floor(v) on serve all four pixels (and four reversed ones their
// reflections): 4 bytes per interpolation, and one floor and one address for
// eight.  A pixel at t bins from bin j takes b[j-1], b[j], b[j+1] with the weights
// max(0, -t), 1 - |t| and max(0, t) for |t| <= 1, so with the corner's fraction f
// and oB, oC the block's steps along its columns and rows: the corner takes b0
// and b1 with 1 - f and f, the next column and the next row lie at f + oB - 1 and
// f + oC - 1 from b1, and the far corner at f + oB + oC - 2 from b2 where oB + oC
// >= 1 (kUnit; at every angle for a pitch of a pixel, ctg_back_blocks_unit), else
// it takes all four bins.  A bin that a pixel does not interpolate has the weight
// zero exactly, so a large value leaves nothing in its neighbours.  (First and
// second differences from b0, shared by the four pixels, are 2 % faster, but carry
// the rounding of every bin of the four: a bin of 1e6 in unit noise left 0.6 in
// pixels beside its reach at 64^2, 90 angles and 1.1 at 512^2, now 3e-5 and 1.4e-4,
// what the noise alone leaves.)
// An angle with sin < 0 is taken as its opposite (the reversed projection), so
// the lowest corner is the left column for cos >= 0 and the right one for cos
// < 0; the sums go to the pixels when that changes, and every kBlkFlush chunks
// (which also keeps the chains of additions short: at 512^2, 720 angles the error
// against FP64 is 6.6e-8 on smooth data and 1.1e-6 on white noise, 0.6 times that
// of one pixel per position from the tile's corner).
// The raw bins are staged by 4-byte cp.async (rows have any alignment) one chunk
// ahead.  Now bound by issue slots (5.2 issued instructions per interpolation)
// and, at 512^2 with its 512 blocks, by latency at few warps (55 % of the slots
// and 61 % of the shared path there, 103 registers): 512^2, 720 angles 73.5
// -> 51.3 us (3.7 T interpolations/s), 2048^2, 1800 angles 2,383 -> 1,437 us (5.3
// T/s); 50.4 and 1,414 us with the differences.
constexpr int kBlkWarps = 4, kBlkThreads = 32 * kBlkWarps;
constexpr int kBlkChunk = 16;         // angles per stage, two stages in flight
constexpr int kBlkFlush = 4;          // (1 in the smaller clusters: few angles, so few chains to average over)
// Window of a 32 x th tile: at a pitch of a pixel or more a block's lowest corner
// lies within half the tile's diagonal of the centre (21.92 bins for 32 rows, 35.11
// for 64) plus a phase below one, and reads the three bins after its own.  A finer
// pitch whose angles all lie near a diagonal also has steps of at most one bin, but
// up to 1.41 times the reach: ctg_back_blocks_ok asks for both.
constexpr int blk_centre(int th) { return th <= 32 ? 24 : 37; }
constexpr int blk_window(int th) { return th <= 32 ? 52 : 78; }

// acc += a * (s, s)
__device__ __forceinline__ void fma2s(float2 &acc, float2 a, float s) {
    asm("{\n\t.reg .b64 c, a, s;\n\t"
        "mov.b64 c, {%0, %1};\n\t"
        "mov.b64 a, {%2, %3};\n\t"
        "mov.b64 s, {%4, %4};\n\t"
        "fma.rn.f32x2 c, a, s, c;\n\t"
        "mov.b64 {%0, %1}, c;\n\t}"
        : "+f"(acc.x), "+f"(acc.y)
        : "f"(a.x), "f"(a.y), "f"(s));
}
// acc += the interpolation at t from the middle one of three bins, |t| <= 1
__device__ __forceinline__ void three_bins(float2 &acc, float2 lo, float2 mid, float2 hi, float t) {
    fma2s(acc, lo, fmaxf(-t, 0.0f));
    fma2s(acc, mid, 1.0f - fabsf(t));
    fma2s(acc, hi, fmaxf(t, 0.0f));
}

// The CTA's pixel sums for angles [a_begin, a_end) one interpolation at a time,
// from global memory: taken when the block sums hold a value that is not
// finite, because a weight of zero would carry an infinite or NaN bin to
// neighbours that do not interpolate it.
template <typename T>
__device__ __noinline__ void pixel_back_plain(const T *__restrict__ b, int n_det, const BackAngle *__restrict__ tab,
                                              int a_begin, int a_end, int j0, int i0, int rows, float *s_px) {
    for (int e = threadIdx.x; e < 2 * rows * kPT; e += blockDim.x) {
        const int h = e / (rows * kPT), i = i0 + (e / kPT) % rows, j = j0 + e % kPT;
        float acc = 0.0f;
        for (int a = a_begin; a < a_end; ++a) {
            const BackAngle t = tab[a];
            const long long U = t.C + (long long)j * t.COS + (long long)i * t.SIN;
            const int d = (int)(U >> CTG_FX_BITS), d0 = h ? n_det - 1 - d : d, d1 = h ? d0 - 1 : d0 + 1;
            const float v0 = (unsigned)d0 < (unsigned)n_det ? to_f(__ldg(b + (size_t)a * n_det + d0)) : 0.0f;
            const float v1 = (unsigned)d1 < (unsigned)n_det ? to_f(__ldg(b + (size_t)a * n_det + d1)) : 0.0f;
            acc += fmaf(fx_frac(U), v1 - v0, v0);
        }
        s_px[e] = acc;
    }
}

// Body of one CTA of the cluster for the 32 x (16 kNB) tile (bx, by) of the
// upper half; each of the 128 threads owns kNB blocks 16 rows apart.  Every CTA
// of a cluster must call it.
template <typename T, int kNB, int kSplit, bool kUnit>
__device__ __forceinline__ void pixel_back_blocks(const T *__restrict__ b, int N, int n_angles, int n_det,
                                                  const BackAngle *__restrict__ tab,
                                                  const float *__restrict__ add, float *__restrict__ x, int bx,
                                                  int by) {
    constexpr int kThr = kBlkThreads, kStep = 4 * kBlkWarps, kTH = kStep * kNB;   // rows between blocks; tile height
    constexpr int kWin = blk_window(kTH), kCentre = blk_centre(kTH);
    constexpr int kFlush = kSplit == kMaxSplit ? kBlkFlush : 1;
    extern __shared__ float4 s_dyn[];
    float2 *s_win = reinterpret_cast<float2 *>(s_dyn);            // [2][kBlkChunk][kWin] (b, b')
    float *s_px = reinterpret_cast<float *>(s_win + 2 * kBlkChunk * kWin);   // [2][kTH][32] sums of the pixels
    static_assert(kNB % 2 == 0 && kTH <= 64, "block tile shape");
    // per angle: phase at the tile centre, oB, oC, oB - 1; oC - 1, oB + oC - 1, oB + oC - 2
    __shared__ float4 s_par[4][kBlkChunk][2];
    __shared__ int2 s_org[4][kBlkChunk];                          // first bin, flip
    __shared__ unsigned s_right[4];                               // angles whose lowest corner is on the right
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j0 = bx * kPT, i0 = by * kTH;
    // a quarter warp holds 4 x 2 blocks, a warp 8 x 4 (16 x 8 pixels): the
    // bins of a half warp's loads span at most 16 entries, no bank conflicts
    const int cb = 8 * (warp & 1) + (lane & 3) + 4 * ((lane >> 3) & 1);
    const int rb = 4 * (warp >> 1) + ((lane >> 2) & 1) + 2 * (lane >> 4);
    const float fdj = 2.0f * cb - 0.5f * (kPT - 1), fdi = 2.0f * rb - 0.5f * (kTH - 1);
    const int per = (n_angles + kSplit - 1) / kSplit;
    const int a_begin = min(n_angles, rank * per), a_end = min(n_angles, a_begin + per);
    const int nchunks = (a_end - a_begin + kBlkChunk - 1) / kBlkChunk;
    for (int e = tid; e < 2 * kTH * kPT / 4; e += kThr)
        reinterpret_cast<float4 *>(s_px)[e] = make_float4(0.f, 0.f, 0.f, 0.f);

    auto params = [&](int c) {
        if (warp != 0) return;
        const int k = lane, a = a_begin + c * kBlkChunk + k;
        bool right = false;
        if (k < kBlkChunk && a < a_end) {
            const BackAngle t = tab[a];
            long long Uc = t.C + (long long)j0 * t.COS + (long long)i0 * t.SIN +
                           (((kPT - 1) * t.COS + (kTH - 1) * t.SIN) >> 1);
            float cf = t.cf, sf = t.sf;
            const int flip = t.SIN < 0;
            if (flip) {
                Uc = ((long long)(n_det - 1) << CTG_FX_BITS) - Uc;
                cf = -cf;
                sf = -sf;
            }
            right = cf < 0.0f;
            const float oB = fabsf(cf);
            s_par[c & 3][k][0] = make_float4(fx_frac(Uc), oB, sf, oB - 1.0f);
            s_par[c & 3][k][1] = make_float4(sf - 1.0f, oB + (sf - 1.0f), (oB - 1.0f) + (sf - 1.0f), 0.0f);
            s_org[c & 3][k] = make_int2((int)(Uc >> CTG_FX_BITS) - kCentre, flip);
        }
        const unsigned m = __ballot_sync(0xffffffffu, right);
        if (lane == 0) s_right[c & 3] = m;
    };
    auto stage = [&](int c) {
        const int a0 = a_begin + c * kBlkChunk, na = min(kBlkChunk, a_end - a0);
        for (int k = warp; k < na; k += kBlkWarps) {
            const int2 o = s_org[c & 3][k];
            const T *row = b + (size_t)(a0 + k) * n_det;
            float2 *dst = s_win + ((c & 1) * kBlkChunk + k) * kWin;
            for (int w = lane; w < kWin; w += 32) {
                const int d = o.x + w, e = n_det - 1 - d;
                const bool in = (unsigned)d < (unsigned)n_det;     // e is in range exactly when d is
                const T *p0 = row + (in ? (o.y ? e : d) : 0), *p1 = row + (in ? (o.y ? d : e) : 0);
                if constexpr (std::is_same<T, float>::value) {
                    const unsigned s0 = (unsigned)__cvta_generic_to_shared(dst + w);
                    const int sz = in ? 4 : 0;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(s0), "l"(p0), "r"(sz));
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(s0 + 4), "l"(p1), "r"(sz));
                } else {
                    dst[w] = in ? make_float2(to_f(__ldg(p0)), to_f(__ldg(p1))) : make_float2(0.f, 0.f);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    float2 A[kNB], B[kNB], C[kNB], E[kNB];             // lowest corner, next column, next row, far corner
    auto clear = [&] {
#pragma unroll
        for (int q = 0; q < kNB; ++q) A[q] = B[q] = C[q] = E[q] = make_float2(0.f, 0.f);
    };
    auto flush = [&](bool right) {
#pragma unroll
        for (int q = 0; q < kNB; ++q) {
            const int row = 2 * rb + kStep * q, col = 2 * cb;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                auto at = [&](const float2 &v) { return h ? v.y : v.x; };
                const float a = at(A[q]), bb = at(B[q]), cc = at(C[q]), ee = at(E[q]);
                float2 *p0 = reinterpret_cast<float2 *>(s_px + (h * kTH + row) * kPT + col);
                float2 *p1 = reinterpret_cast<float2 *>(s_px + (h * kTH + row + 1) * kPT + col);
                float2 t0 = *p0, t1 = *p1;
                t0.x += right ? bb : a;
                t0.y += right ? a : bb;
                t1.x += right ? ee : cc;
                t1.y += right ? cc : ee;
                *p0 = t0;
                *p1 = t1;
            }
        }
        clear();
    };
    clear();
    bool right = false;
    float sdj = fdj;                        // u = phase + oB sdj + oC fdi at the block's lowest corner
    params(0);
    __syncthreads();
    stage(0);
    for (int c = 0; c < nchunks; ++c) {
        if (c + 1 < nchunks) params(c + 1); // (slower warps may still read those of c - 1 and c)
        __syncthreads();                    // params of c + 1 written; the windows of c - 1 have been read
        if (c + 1 < nchunks) {
            stage(c + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();                    // the windows of c have landed
        const int na = min(kBlkChunk, a_end - a_begin - c * kBlkChunk);
        const float4 (*par)[2] = s_par[c & 3];
        // shared address of the window's centre less the magic number's bits
        // times 8 (32-bit wrap-around), as in pixel_pair_tile
        unsigned sb = (unsigned)__cvta_generic_to_shared(s_win + (c & 1) * kBlkChunk * kWin + kCentre) -
                      (0x4B400000u << 3);
        // runs of angles with the lowest corner on the same side
        const unsigned rights = s_right[c & 3];
        for (int k = 0; k < na;) {
            const bool r = (rights >> k) & 1;
            const unsigned change = (r ? ~rights : rights) >> k;
            const int end = change ? min(na, k + __ffs(change) - 1) : na;
            if (r != right) {
                flush(right);
                right = r;
                sdj = r ? -(fdj + 1.0f) : fdj;
            }
#pragma unroll 4
            for (; k < end; ++k, sb += 8u * kWin) {
                const float4 p = par[k][0], o = par[k][1];
                const float u0 = fmaf(p.z, fdi, fmaf(p.y, sdj, p.x));
                float tt[kNB], ff[kNB];
#pragma unroll
                for (int q = 0; q < kNB; q += 2)
                    floor_frac2(fmaf(p.z, (float)(kStep * q), u0), fmaf(p.z, (float)(kStep * (q + 1)), u0), tt[q],
                                tt[q + 1], ff[q], ff[q + 1]);
#pragma unroll
                for (int q = 0; q < kNB; ++q) {
                    const unsigned at = sb + (__float_as_uint(tt[q]) << 3);
                    const float2 *e = static_cast<const float2 *>(__cvta_shared_to_generic(at));
                    const float2 b0 = e[0], b1 = e[1], b2 = e[2], b3 = e[3];
                    const float f = ff[q];
                    fma2s(A[q], b0, 1.0f - f);
                    fma2s(A[q], b1, f);
                    const float tB = f + p.w, tC = f + o.x, tE = f + o.z;
                    three_bins(B[q], b0, b1, b2, tB);
                    three_bins(C[q], b0, b1, b2, tC);
                    if constexpr (kUnit) {
                        three_bins(E[q], b1, b2, b3, tE);
                    } else {
                        const float t = f + o.y;            // from b1, tE from b2
                        fma2s(E[q], b0, fmaxf(-t, 0.0f));
                        fma2s(E[q], b1, __saturatef(1.0f - fabsf(t)));
                        fma2s(E[q], b2, __saturatef(1.0f - fabsf(tE)));
                        fma2s(E[q], b3, fmaxf(tE, 0.0f));
                    }
                }
            }
        }
        if (c % kFlush == kFlush - 1) flush(right);
    }
    flush(right);
    {
        bool bad = false;
#pragma unroll
        for (int q = 0; q < kNB; ++q)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float2 v = *reinterpret_cast<const float2 *>(
                    s_px + ((r >> 1) * kTH + 2 * rb + kStep * q + (r & 1)) * kPT + 2 * cb);
                bad = bad || !(fabsf(v.x) <= 3.402823466e38f) || !(fabsf(v.y) <= 3.402823466e38f);
            }
        if (__syncthreads_or(bad)) pixel_back_plain<T>(b, n_det, tab, a_begin, a_end, j0, i0, kTH, s_px);
    }
    cluster.sync();
    // this CTA finishes a share of the 2 x (kTH x 32) sums: h = 0 the tile's
    // pixels, h = 1 their reflections.  A pixel at or before the image's centre
    // is written by h = 0, the others by h = 1 (on the middle row of an odd N
    // both reach it).
    const long long last = (long long)N * N - 1;
    constexpr int kShare = 2 * kTH * kPT / kSplit;
    for (int e = rank * kShare + tid; e < (rank + 1) * kShare; e += kThr) {
        float sum = 0.0f;
#pragma unroll
        for (int q = 0; q < kSplit; ++q) sum += cluster.map_shared_rank(s_px, q)[e];
        const int h = e / (kTH * kPT), i = i0 + (e / kPT) % kTH, j = j0 + e % kPT;
        const long long p = (long long)i * N + j;
        if (i < N && j < N && (h ? 2 * p < last : 2 * p <= last)) {
            const long long o = h ? last - p : p;
            x[o] = add ? sum + add[o] : sum;
        }
    }
    cluster.sync();   // peers' shared memory must outlive the reads above
}
constexpr size_t blk_smem(int nb) {
    return sizeof(float2) * 2 * kBlkChunk * blk_window(16 * nb) + sizeof(float) * 2 * 16 * nb * kPT;
}
constexpr int blk_tiles_y(int N, int nb) { return ((N + 1) / 2 + 16 * nb - 1) / (16 * nb); }

template <typename T, int kNB, int kSplit, bool kUnit>
__global__ void __cluster_dims__(1, 1, kSplit) __launch_bounds__(kBlkThreads, kNB == 4 ? 4 : 7)
pixel_back_blocks_kernel(const T *__restrict__ b, ColRef bc, int N, int n_angles, int n_det,
                         const BackAngle *__restrict__ tab, const float *__restrict__ add, float *__restrict__ x,
                         const SolveIo *__restrict__ io) {
    if (io) add = io->x0, x = io->x;
    pixel_back_blocks<T, kNB, kSplit, kUnit>(b + col_offset(bc), N, n_angles, n_det, tab, add, x, blockIdx.x, blockIdx.y);
}

// bc: the input is column bc of a basis (b + col_offset(bc)), or b itself.
// kModel: the pixel-driven B (0), A^T (1) or B_tau (2).
template <typename T, int kModel, int kChunk, int kRows, int kSplit>
__global__ void __cluster_dims__(1, 1, kSplit) __launch_bounds__(pair_threads<kRows>())
pixel_pair_kernel(const T *__restrict__ b, ColRef bc, int N, int n_angles, int n_det,
                  const BackAngle *__restrict__ tab, int W, const MatchedAngle *__restrict__ mt, float thr,
                  const float *__restrict__ add, float *__restrict__ x, const SolveIo *__restrict__ io) {
    if (io) add = io->x0, x = io->x;
    pixel_pair_tile<T, kModel, kChunk, kRows, kSplit>(b + col_offset(bc), N, n_angles, n_det, tab, W, add, x,
                                                      blockIdx.x, blockIdx.y, mt, thr);
}

// Generic pixel-driven back projection (any detector pitch): 32 x 8 tiles,
// taps read through L1 with bounds tests.
constexpr int kBX = 32, kBY = 8, kAChunk = 256;

template <typename T>
__global__ void __launch_bounds__(kBX *kBY)
pixel_back_kernel(const T *__restrict__ b, ColRef bc, int N, int n_angles, int n_det,
                  const BackAngle *__restrict__ tab, const float *__restrict__ add,
                  float *__restrict__ x, const SolveIo *__restrict__ io) {
    __shared__ float4 sp[kAChunk];
    if (io) add = io->x0, x = io->x;
    b += col_offset(bc);
    const int j0 = blockIdx.x * kBX, i0 = blockIdx.y * kBY;
    const int dj = threadIdx.x, di = threadIdx.y;
    const int tid = di * kBX + dj;
    const float fdj = (float)dj, fdi = (float)di;
    float acc = 0.0f;
    for (int a0 = 0; a0 < n_angles; a0 += kAChunk) {
        const int na = min(kAChunk, n_angles - a0);
        __syncthreads();
        if (tid < na) {
            const BackAngle t = tab[a0 + tid];
            const long long U0 = t.C + (long long)j0 * t.COS + (long long)i0 * t.SIN;
            sp[tid] = make_float4(t.cf, t.sf, fx_frac(U0),
                                  __int_as_float((int)(U0 >> CTG_FX_BITS)));
        }
        __syncthreads();
        const T *brow = b + (size_t)a0 * n_det;
#pragma unroll 4
        for (int k = 0; k < na; ++k, brow += n_det) {
            const float4 p = sp[k];
            const float u = fmaf(fdi, p.y, fmaf(fdj, p.x, p.z));
            const float fl = floorf(u);
            const int dd = __float_as_int(p.w) + (int)fl;
            const float f = u - fl;
            const float v0 = ((unsigned)dd < (unsigned)n_det) ? to_f(__ldg(brow + dd)) : 0.0f;
            const float v1 = ((unsigned)(dd + 1) < (unsigned)n_det) ? to_f(__ldg(brow + dd + 1)) : 0.0f;
            acc += fmaf(f, v1 - v0, v0);
        }
    }
    const int i = i0 + di, j = j0 + dj;
    if (i < N && j < N) {
        const size_t p = (size_t)i * N + j;
        x[p] = add ? acc + add[p] : acc;
    }
}

}  // namespace

namespace {
// Dynamic shared memory of the tiled back projectors: the staged windows (kept
// to 40 KB, so that no launch needs an opt-in), or the partial sums that take
// their place.
constexpr size_t kBackSmem = 40 * 1024;
constexpr int kPairChunkMin = 8;
constexpr int kBackWindowMaxTiled = (int)(kBackSmem / (sizeof(float4) * kPairChunkMin));
bool back_chunk_fits(int chunk, int window) { return (size_t)chunk * window * sizeof(float4) <= kBackSmem; }
// the chunk asked for, or the largest one whose windows fit
int back_chunk_for(int chunk, int window) {
    if (chunk != 16) chunk = kPairChunk;
    while (chunk > kPairChunkMin && !back_chunk_fits(chunk, window)) chunk /= 2;
    return chunk;
}
size_t pair_smem(int chunk, int window) {
    return std::max((size_t)chunk * window * sizeof(float4), sizeof(float) * 2 * kPT * kPT);
}

// CTAs per cluster for an image of `tiles` tiles: eight, halved while a CTA's
// share would be below 30 angles (a tile's start, end and cluster sum then cost
// as much as its angles) and the launch keeps about three CTAs per SM.  B at
// 1024^2: 60 angles 29 us with 8, 23 with 2; 120 angles 37 and 35 (4); 2048^2, 60
// angles 102 and 69 us.
constexpr int kFullGrid = 450;
int split_for(int n_angles, int tiles) {
    int s = kMaxSplit;
    while (s > 2 && n_angles < 30 * s && tiles * (s / 2) >= kFullGrid) s /= 2;
    return s;
}
// Blocks per thread of the block kernel: four (64-row tiles: half the staging
// and parameter loads per pixel, about 6 % per row) unless the image's last tile
// row would waste more than that or the launch would be small (four against two
// blocks: 512^2, 720 angles 48.8 against 50.1 us, 2048^2, 1800 angles 1,434 against
// 1,533; 700^2, 720 angles 90 against 83; 361^2, 187 angles 11.7 against 11.0).
int blocks_for(int N, int split) {
    const int rows4 = 64 * blk_tiles_y(N, 4), rows2 = 32 * blk_tiles_y(N, 2);
    return 100 * rows2 >= 93 * rows4 && back_tiles_x(N) * blk_tiles_y(N, 4) * split >= kFullGrid ? 4 : 2;
}
}  // namespace

bool ctg_back_blocks_ok(const BackAngle *host_tab, int n_angles) {
    // a block spans at most 3 bins where a pixel step is at most one bin in
    // either direction; its lowest corner is phase + oB j + oC i bins from the
    // tile centre's bin, 0 <= phase < 1, j in [-15.5, 14.5] and i in [-(th - 1) / 2,
    // (th - 3) / 2], and the window holds that bin and the next three.  Each bound
    // has a 64th of a bin for the rounding of the positions.
    constexpr double slack = 1.0 / 64;
    for (int a = 0; a < n_angles; ++a) {
        const double oB = std::fabs((double)host_tab[a].cf), oC = std::fabs((double)host_tab[a].sf);
        if (!(oB <= 1.0 && oC <= 1.0)) return false;
        for (const int th : {32, 64}) {
            const double low = 0.5 * (kPT - 1) * oB + 0.5 * (th - 1) * oC;       // bins below the centre's phase
            const double high = 1.0 + 0.5 * (kPT - 3) * oB + 0.5 * (th - 3) * oC; // and above its bin
            if (low > blk_centre(th) - slack || high > blk_window(th) - 3 - blk_centre(th) - slack) return false;
        }
    }
    return true;
}

int ctg_back_chunk_used(BackBlocks blocks, int window, int chunk) {
    const bool pairs = blocks == kBlocksNo && window > 0 && window <= kBackWindowMaxTiled;
    return pairs ? back_chunk_for(chunk, window) : 0;
}

bool ctg_back_blocks_unit(const BackAngle *host_tab, int n_angles) {
    // the far corner's distance from b2, f + (oB - 1) + (oC - 1), must not round
    // to below -1: a margin, or an angle along an axis, whose steps are exact
    for (int a = 0; a < n_angles; ++a) {
        const double oB = std::fabs((double)host_tab[a].cf), oC = std::fabs((double)host_tab[a].sf);
        const bool axis = (oB == 1.0 && oC == 0.0) || (oB == 0.0 && oC == 1.0);
        if (!axis && !(oB + oC >= 1.0 + 1e-6)) return false;
    }
    return true;
}

namespace {

// The arguments of one back projection.
template <typename T> struct BackArgs {
    const T *b;
    ColRef bc;
    int N, n_angles, n_det;
    const BackAngle *tab;
    int window;
    const MatchedAngle *mt;
    float thr;
    const float *add;
    float *x;
    cudaStream_t st;
    const SolveIo *io;
};

template <int kModel, int kChunk, int kRows, int kSplit, typename T>
void launch_pair(const BackArgs<T> &a) {
    const dim3 grid(back_tiles_x(a.N), back_tiles_y(a.N), kSplit);
    pixel_pair_kernel<T, kModel, kChunk, kRows, kSplit>
        <<<grid, pair_threads<kRows>(), pair_smem(kChunk, a.window), a.st>>>(
            a.b, a.bc, a.N, a.n_angles, a.n_det, a.tab, a.window, a.mt, a.thr, a.add, a.x, a.io);
}

template <int kNB, int kSplit, typename T>
void launch_blocks(const BackArgs<T> &a, bool unit) {
    const dim3 grid(back_tiles_x(a.N), blk_tiles_y(a.N, kNB), kSplit);
    auto run = [&](auto kernel) {
        kernel<<<grid, kBlkThreads, blk_smem(kNB), a.st>>>(a.b, a.bc, a.N, a.n_angles, a.n_det, a.tab, a.add, a.x, a.io);
    };
    if (unit) run(pixel_back_blocks_kernel<T, kNB, kSplit, true>);
    else run(pixel_back_blocks_kernel<T, kNB, kSplit, false>);
}

// blocks: the 2 x 2 block kernel and its form.  back_chunk: angles
// staged per pass of the one-pixel tiled kernel, 16 or (any other value, where
// it fits) 32.  Each pixel sums its angles in the same order whatever the
// chunk, so the result does not depend on it.
template <typename T>
cudaError_t launch_back_t(const BackArgs<T> &a, BackBlocks blocks, int back_chunk) {
    if (blocks != kBlocksNo) {
        const bool unit = blocks == kBlocksUnit;
        const int split = split_for(a.n_angles, back_tiles_x(a.N) * blk_tiles_y(a.N, 2));
        const bool four = blocks_for(a.N, split) == 4;
        if (split == 8) four ? launch_blocks<4, 8>(a, unit) : launch_blocks<2, 8>(a, unit);
        else if (split == 4) four ? launch_blocks<4, 4>(a, unit) : launch_blocks<2, 4>(a, unit);
        else four ? launch_blocks<4, 2>(a, unit) : launch_blocks<2, 2>(a, unit);
    } else if (a.window > 0 && a.window <= kBackWindowMaxTiled) {
        // four rows per thread (a finer pitch's windows leave room for few
        // CTAs); two CTAs per cluster once that fills the device (pitch 0.75:
        // 512^2, 1000 angles 138 us with 8, 1024^2 408 with 2 against 467 with 8)
        const int chunk = back_chunk_for(back_chunk, a.window);
        const bool two = back_tiles_x(a.N) * back_tiles_y(a.N) * 2 >= 2 * kFullGrid;
        if (chunk == 8) two ? launch_pair<0, 8, 4, 2>(a) : launch_pair<0, 8, 4, 8>(a);
        else if (chunk == 16) two ? launch_pair<0, 16, 4, 2>(a) : launch_pair<0, 16, 4, 8>(a);
        else two ? launch_pair<0, kPairChunk, 4, 2>(a) : launch_pair<0, kPairChunk, 4, 8>(a);
    } else {
        dim3 grid((a.N + kBX - 1) / kBX, (a.N + kBY - 1) / kBY);
        pixel_back_kernel<T><<<grid, dim3(kBX, kBY), 0, a.st>>>(a.b, a.bc, a.N, a.n_angles, a.n_det, a.tab, a.add,
                                                                a.x, a.io);
    }
    return cudaGetLastError();
}

// A^T or B_tau: four rows per thread (256 threads, more warps) for small
// launches, eight (half the parameter loads and weights) from about six CTAs
// per SM on (A^T, 200^2, 1000 angles: 35 against 41 us; 1001^2, 900 angles: 302
// against 280); four CTAs per cluster for few angles.
template <int kModel, int kChunk, typename T>
void launch_matched(const BackArgs<T> &a) {
    const int tiles = back_tiles_x(a.N) * back_tiles_y(a.N);
    if (tiles * kMaxSplit < 2 * kFullGrid) launch_pair<kModel, kChunk, 4, 8>(a);
    else if (split_for(a.n_angles, tiles) == kMaxSplit) launch_pair<kModel, kChunk, 8, 8>(a);
    else launch_pair<kModel, kChunk, 8, 4>(a);
}

template <typename T>
cudaError_t launch_matched_tiled_t(const BackArgs<T> &a) {
    const bool full = back_chunk_for(kPairChunk, a.window) == kPairChunk;
    if (a.thr > 0.0f) full ? launch_matched<2, kPairChunk>(a) : launch_matched<2, 16>(a);
    else full ? launch_matched<1, kPairChunk>(a) : launch_matched<1, 16>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t ctg_launch_back_matched_tiled(const void *b, int dtype, int N, int n_angles, int n_det,
                                          const BackAngle *tab, int window, const MatchedAngle *mt,
                                          float thr, const float *add, float *x, cudaStream_t st,
                                          ColRef bc, const SolveIo *io) {
    if (window <= 0 || window > ctg_back_window_max()) return cudaErrorInvalidValue;
    auto run = [&](auto *p) {
        using T = typename std::remove_const<typename std::remove_pointer<decltype(p)>::type>::type;
        return launch_matched_tiled_t(BackArgs<T>{p, bc, N, n_angles, n_det, tab, window, mt, thr, add, x, st, io});
    };
    switch (dtype) {
        case CTG_BASIS_FP32: return run(static_cast<const float *>(b));
        case CTG_BASIS_BF16: return run(static_cast<const __nv_bfloat16 *>(b));
        case CTG_BASIS_FP16: return run(static_cast<const __half *>(b));
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t ctg_launch_back(const void *b, int dtype, int N, int n_angles, int n_det,
                            const BackAngle *tab, int window, BackBlocks blocks, const float *add, float *x,
                            cudaStream_t st, int back_chunk, ColRef bc, const SolveIo *io) {
    auto run = [&](auto *p) {
        using T = typename std::remove_const<typename std::remove_pointer<decltype(p)>::type>::type;
        return launch_back_t(BackArgs<T>{p, bc, N, n_angles, n_det, tab, window, nullptr, 0.0f, add, x, st, io}, blocks,
                             back_chunk);
    };
    switch (dtype) {
        case CTG_BASIS_FP32: return run(static_cast<const float *>(b));
        case CTG_BASIS_BF16: return run(static_cast<const __nv_bfloat16 *>(b));
        case CTG_BASIS_FP16: return run(static_cast<const __half *>(b));
        default: return cudaErrorInvalidValue;
    }
}

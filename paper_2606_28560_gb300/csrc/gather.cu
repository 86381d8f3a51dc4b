// gather.cu -- forward and backward passes that read their rows through L1/L2
// and compute in fp32 on the CUDA cores (arXiv 2606.28560, Section 2): the
// path of fp32 I/O (whose 1e-4 bar rules out 16-bit score operands) and of
// windows and rung counts beyond the tensor-core kernels'.
//
// Blocking.  A group of 8 lanes owns R = 4 consecutive rows (queries, or keys
// in the key pass), each lane 8 of the 64 dims; a warp works on 16 consecutive
// rows.  The rows that neighbours read overlap: window rows by all but one, and
// a rung's far row of one query is the floor row of the one before it.  So R
// queries load W + R window rows instead of R (W + 1), and R + 1 rows a rung
// instead of 2 R.
//
// Phases.  Every dot product of a warp comes first (loads that depend on
// nothing, sums reduce-scattered over the group), its slot values then sit in
// shared memory as [slot][row], the softmax or its gradient runs over that
// table, and a second sweep adds weighted rows.  A window beyond kChunk slots
// goes through the table chunk by chunk.
//
// Split.  While a warp per 16 rows leaves an SM few warps, the four warps of a
// block take the same 16 rows and share out the window rows and the rungs; the
// table is then the block's, and the four partial sums meet in shared memory.
//
// Bound by load latency and issue, not bytes: 113-128 registers leave 16 warps
// an SM at the narrow windows of the paper; the query pass's tables (a quarter KB
// a block for each 2 W + 13 + 2 rungs) leave 12 from W of about 100 on, 8 from 140,
// and 4 at W 207 with 15 rungs beyond it.  Issue is active 44-47 % of cycles, L1
// 56-60 % (fp32 B16 T1024 W 8).  Against one 4-lane group a row that
// walked its slots one after another (us):
//   fp32 W 8 B4 H8 T1000   forward 34.5 -> 24.5, query pass with the rotation of
//                          q 58 -> 36.6, key pass 61 -> 24.4
//   fp32 W 8 B16 H8 T1024  forward 105.8 -> 61.4
//   bf16 W 32 B4 H8 T1024  35.8 -> 30.3, 65 -> 46.8, 67 -> 28.5
// and graph-replayed, forward and backward: bf16 W 200 B2 H8 T1000 400 -> 245,
// W 1024 B2 H8 T2048 2717 -> 2259, W 300 B4 H8 T4096 2681 -> 2147.
// (Two rows a group: layer 118 us for the 73.8 of fp32 B4 T1000; two or eight
// warps a block: 93 us and worse.)
//
// kChunk, the most window slots a table holds: wider windows pay for passes over
// the table, and narrower ones that would fit must not.  104: fp32 B4 T1000 W150
// forward 61.7 -> 83.4 us, W200 76.5 -> 103; but with more warps an SM the backward
// of W300 B4 T4096 takes 1444 instead of 1789.  312: W 208 to 311 gain up to a
// fifth in the backward (253 -> 204 at B2 T1000 W208), wider ones lose up to half
// (W300 B4 T4096, a table 1.4 times as large: 1789 -> 2439).
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "fibattn_internal.cuh"
#include "mma_common.cuh"

namespace fibattn {
namespace {

constexpr int kWarps = 4;                     // warps of a block
constexpr int kGroups = 4;                    // 8-lane groups of a warp
constexpr int R = 4;                          // consecutive rows of a group
constexpr int QW = kGroups * R;               // rows of a warp
constexpr int kChunk = 208;                   // window slots of the shared table at a time
constexpr float kLog2e = 1.4426950408889634f;
constexpr unsigned kAll = 0xffffffffu;

// The active rungs, compact, in the caller's order.
struct RungList {
    int n;
    int k[kMaxRungs], s0[kMaxRungs];
    float w[kMaxRungs], d[kMaxRungs];
};

RungList rung_list(const RungParams& r) {
    RungList l;
    std::memset(&l, 0, sizeof(l));
    for (int k = 0; k < r.K; ++k) {
        if (!((r.active >> k) & 1u)) continue;
        l.k[l.n] = k; l.s0[l.n] = r.s0[k]; l.w[l.n] = r.w[k]; l.d[l.n] = r.d[k];
        ++l.n;
    }
    return l;
}

// A lane's 8 dims of a row, as 4 pairs.  fp32: dims 4c..4c+3 and 32 + 4c..,
// two 16-byte loads that cover 128 contiguous bytes over the group; 16-bit:
// dims 8c..8c+7, one 16-byte load.
// Raw: the loaded words, expanded to fp32 where they are used.  kBatch,
// kPair: window rows and rungs whose loads a warp issues before the first use
// (few warps share an SM, so a warp needs many loads in flight; the registers
// of 128-thread blocks, four an SM, hold these).
template <typename T> struct Lane;
template <> struct Lane<float> {
    struct Raw { float4 a, b; };
    static constexpr int kBatch = 6, kPair = 1;
    static __device__ __forceinline__ Raw raw(const float* row, int c) {
        return {*reinterpret_cast<const float4*>(row + 4 * c), *reinterpret_cast<const float4*>(row + kHalf + 4 * c)};
    }
    static __device__ __forceinline__ Raw zero() { return {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)}; }
    static __device__ __forceinline__ void expand(const Raw& v, float2 (&x)[4]) {
        x[0] = make_float2(v.a.x, v.a.y); x[1] = make_float2(v.a.z, v.a.w);
        x[2] = make_float2(v.b.x, v.b.y); x[3] = make_float2(v.b.z, v.b.w);
    }
    static __device__ __forceinline__ void store(float* row, int c, const float2 (&x)[4]) {
        *reinterpret_cast<float4*>(row + 4 * c) = make_float4(x[0].x, x[0].y, x[1].x, x[1].y);
        *reinterpret_cast<float4*>(row + kHalf + 4 * c) = make_float4(x[2].x, x[2].y, x[3].x, x[3].y);
    }
    // Rotation of N consecutive rows by the angles at pos, pos + 1, ...
    // (inverse: by their negatives); RoPE pairs (m, m + 32) are the lane's own.
    // The angles of one row, and of one step, are evaluated; the others follow
    // by the step.
    template <int N>
    static __device__ __forceinline__ void rope(const RopeParams& rp, int pos, int c, float2 (&x)[N][4], bool inverse) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = u & 1, h = u >> 1;      // dims 4c + 2h + e
            float cs, sn, c1 = 0.f, s1 = 0.f;
            rope_cs_exact(rp, 4 * c + u, pos, cs, sn);
            if (N > 1) rope_cs_exact(rp, 4 * c + u, 1, c1, s1);
#pragma unroll
            for (int r = 0; r < N; ++r) {
                float& a = e ? x[r][h].y : x[r][h].x;
                float& b = e ? x[r][2 + h].y : x[r][2 + h].x;
                const float sg = inverse ? -sn : sn, a0 = a, b0 = b;
                a = a0 * cs - b0 * sg;
                b = b0 * cs + a0 * sg;
                const float cn = cs * c1 - sn * s1;
                sn = sn * c1 + cs * s1;
                cs = cn;
            }
        }
    }
};
struct Lane16 {
    using Raw = uint4;
    static constexpr int kBatch = 8, kPair = 2;
    static __device__ __forceinline__ Raw raw(const void* row, int c) { return reinterpret_cast<const uint4*>(row)[c]; }
    static __device__ __forceinline__ Raw zero() { return make_uint4(0u, 0u, 0u, 0u); }
    // partner dims m +- 32 are lane c ^ 4's
    template <int N>
    static __device__ __forceinline__ void rope(const RopeParams& rp, int pos, int c, float2 (&x)[N][4], bool inverse) {
#pragma unroll
        for (int r = 0; r < N; ++r) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float c0, s0, c1, s1;
                rope_cs(rp, 8 * (c & 3) + 2 * u, pos + r, c0, s0);
                rope_cs(rp, 8 * (c & 3) + 2 * u + 1, pos + r, c1, s1);
                const float px = __shfl_xor_sync(kAll, x[r][u].x, 4), py = __shfl_xor_sync(kAll, x[r][u].y, 4);
                // (the products fused as in rope_rows_bf16_kernel, so that a row
                // rounds to the same fp16 row there and here)
                if (inverse != (c < 4)) { s0 = -s0; s1 = -s1; }
                x[r][u] = make_float2(__fmaf_rn(x[r][u].x, c0, __fmul_rn(px, s0)),
                                      __fmaf_rn(x[r][u].y, c1, __fmul_rn(py, s1)));
            }
        }
    }
};
template <> struct Lane<__nv_bfloat16> : Lane16 {
    static __device__ __forceinline__ void expand(const Raw& v, float2 (&x)[4]) {
        const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = make_float2(__uint_as_float(w[u] << 16), __uint_as_float(w[u] & 0xffff0000u));
    }
    static __device__ __forceinline__ void store(__nv_bfloat16* row, int c, const float2 (&x)[4]) {
        unsigned w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(x[u].x, x[u].y);
            w[u] = *reinterpret_cast<const unsigned*>(&h);
        }
        *reinterpret_cast<uint4*>(row + 8 * c) = make_uint4(w[0], w[1], w[2], w[3]);
    }
};
template <> struct Lane<__half> : Lane16 {
    static __device__ __forceinline__ void expand(const Raw& v, float2 (&x)[4]) {
        const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = __half22float2(*reinterpret_cast<const __half2*>(&w[u]));
    }
    static __device__ __forceinline__ void store(__half* row, int c, const float2 (&x)[4]) {
        unsigned w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const __half2 h = __floats2half2_rn(x[u].x, x[u].y);
            w[u] = *reinterpret_cast<const unsigned*>(&h);
        }
        *reinterpret_cast<uint4*>(row + 8 * c) = make_uint4(w[0], w[1], w[2], w[3]);
    }
};

// N consecutive rows from row j; rows outside [0, T) read as zero.  lo, hi: the
// first and last row that the warp's lanes ask for together; while they are
// inside, a lane's loads share one address and carry no predicates.
template <int N, typename T>
__device__ __forceinline__ void load_rows(const T* base, int j, int lo, int hi, int T_, int c,
                                          typename Lane<T>::Raw (&x)[N]) {
    if (lo >= 0 && hi < T_) {
        const T* p = base + (unsigned)j * kHeadDim;
#pragma unroll
        for (int u = 0; u < N; ++u) x[u] = Lane<T>::raw(p + u * kHeadDim, c);
    } else {
#pragma unroll
        for (int u = 0; u < N; ++u) {
            x[u] = Lane<T>::zero();
            if ((unsigned)(j + u) < (unsigned)T_) x[u] = Lane<T>::raw(base + (unsigned)(j + u) * kHeadDim, c);
        }
    }
}
template <typename T>
__device__ __forceinline__ void load_row(const T* row, int c, float2 (&x)[4]) {
    Lane<T>::expand(Lane<T>::raw(row, c), x);
}

__device__ __forceinline__ float dot(const float2 (&a)[4], const float2 (&b)[4]) {
    float2 s = __fmul2_rn(a[0], b[0]);
#pragma unroll
    for (int e = 1; e < 4; ++e) s = __ffma2_rn(a[e], b[e], s);
    return s.x + s.y;
}
__device__ __forceinline__ void axpy(float a, const float2 (&x)[4], float2 (&y)[4]) {
    const float2 a2 = make_float2(a, a);
#pragma unroll
    for (int e = 0; e < 4; ++e) y[e] = __ffma2_rn(a2, x[e], y[e]);
}
__device__ __forceinline__ void scale(float a, float2 (&y)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) y[e] = __fmul2_rn(y[e], make_float2(a, a));
}
__device__ __forceinline__ void clear(float2 (&acc)[R][4]) {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[r][e] = make_float2(0.f, 0.f);
}

// Sum of each of the R values over the group's 8 lanes; a lane ends with that
// of its own row c >> 1 (lanes 2r and 2r + 1 hold row r's).
__device__ __forceinline__ float group_sums(const float (&v)[R], int c) {
    const bool u4 = c & 4, u2 = c & 2;
    const float a = (u4 ? v[2] : v[0]) + __shfl_xor_sync(kAll, u4 ? v[0] : v[2], 4);
    const float b = (u4 ? v[3] : v[1]) + __shfl_xor_sync(kAll, u4 ? v[1] : v[3], 4);
    const float x = (u2 ? b : a) + __shfl_xor_sync(kAll, u2 ? a : b, 2);
    return x + __shfl_xor_sync(kAll, x, 1);
}

// The rows of one block and the share of one warp of it.  SPLIT: the warps
// share rows iw .. iw + 15 and warp w takes the w-th of every kWarps load
// batches and rung groups; else each has 16 rows of its own.
template <bool SPLIT>
struct Place {
    int lane, c, g, warp;
    int iw;                                       // the warp's first row
    int row;                                      // the row whose sums this lane gets (lanes 2r, 2r + 1 of a group)
    bool writer;                                  // one lane of the two
    int step, first;                              // batches: first, first + step, ...
    __device__ __forceinline__ Place(int tile) {
        lane = threadIdx.x & 31; c = lane & 7; g = lane >> 3;
        // (through a shuffle, which makes it and all that follows from it uniform:
        // with the bounds below the fp32 key pass spilled 128 bytes without it;
        // layer B4 H8 T1000 W8 75.5 us without, 71.0 with)
        warp = __shfl_sync(kAll, threadIdx.x >> 5, 0);
        iw = SPLIT ? tile * QW : (tile * kWarps + warp) * QW;
        row = iw + g * R + (c >> 1);
        writer = (c & 1) == 0;
        step = SPLIT ? kWarps : 1;
        first = SPLIT ? warp : 0;
    }
    __device__ __forceinline__ void sync() const {
        if (SPLIT) __syncthreads();
        else __syncwarp();
    }
    // Window slots that any row of the warp has: as queries (slot t of query i is
    // row i - t), as keys (slot t of query j + t reads key j).  A window longer
    // than that is not walked: B4 H8 T128 W1024, fp32, forward 186 -> 30 us,
    // backward 751 -> 88 (13 and 39 with tables for the sequence, see window_slots);
    // B2 T2048 W1024 forward 495 -> 443, backward 2312 -> 1953.
    // Slots beyond are in no table, nor in the workspace: no key has them either.
    __device__ __forceinline__ int query_slots(const Shape& s) const { return min(min(s.W + 1, s.T), iw + QW); }
    __device__ __forceinline__ int key_slots(const Shape& s) const { return min(s.W + 1, s.T - iw); }
};
template <bool SPLIT> constexpr int kTileRows16 = SPLIT ? QW : kWarps * QW;

// put(t, x) for every window slot t in [t0, t1) of the lane's own row, x the
// product of vec of that row with row i - t, summed over the group.
template <bool SPLIT, typename T, typename Put>
__device__ __forceinline__ void dot_window(const Place<SPLIT>& p, const float2 (&vec)[R][4], const T* base, int T_,
                                           int t0, int t1, Put put) {
    constexpr int kBatch = Lane<T>::kBatch;
    const int n = R - 1 + t1 - t0, jw = p.iw - (t1 - 1);
#pragma unroll 1
    for (int y0 = p.first * kBatch; y0 < n; y0 += p.step * kBatch) {
        typename Lane<T>::Raw row[kBatch];
        load_rows<kBatch>(base, jw + p.g * R + y0, jw + y0, jw + 3 * R + y0 + kBatch - 1, T_, p.c, row);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            float2 x[4];
            Lane<T>::expand(row[u], x);
            float v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = dot(vec[r], x);
            const float sum = group_sums(v, p.c);
            const int t = (p.c >> 1) + t1 - 1 - (y0 + u);
            if (t >= t0 && t < t1) put(t, sum);
        }
    }
}

// put(n, x0, x1) for every active rung n that some query of the warp attends
// (d <= its last query; skip(n) for the others): x0, x1 the products of vec of
// the lane's own row with its floor and far rows, row -1 being a zero row.
// kPair rungs at a time.
template <bool SPLIT, typename T, typename Put, typename Skip>
__device__ __forceinline__ void dot_rungs(const Place<SPLIT>& p, const float2 (&vec)[R][4], const T* base, int T_,
                                          const RungList& L, Put put, Skip skip) {
    constexpr int NP = Lane<T>::kPair;
    const float dmax = (float)(p.iw + QW - 1);
#pragma unroll 1
    for (int n0 = p.first * NP; n0 < L.n; n0 += p.step * NP) {
        typename Lane<T>::Raw row[NP][R + 1];
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int jw = p.iw - L.s0[n0 + u] - 1;
            if (n0 + u < L.n && L.d[n0 + u] <= dmax)          // warp-uniform
                load_rows<R + 1>(base, jw + p.g * R, jw, jw + QW, T_, p.c, row[u]);
        }
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            if (n0 + u >= L.n) break;
            if (L.d[n0 + u] <= dmax) {
                float v[R], w[R];
                float2 x[2][4];
                Lane<T>::expand(row[u][0], x[0]);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    Lane<T>::expand(row[u][r + 1], x[(r + 1) & 1]);
                    v[r] = dot(vec[r], x[(r + 1) & 1]);
                    w[r] = dot(vec[r], x[r & 1]);
                }
                const float x0 = group_sums(v, p.c), x1 = group_sums(w, p.c);
                put(n0 + u, x0, x1);
            } else {
                skip(n0 + u);
            }
        }
    }
}

// acc[r] += sum over window slots t in [t0, t1) of tab[t - t0][r] row(i - t),
// i the group's row r: each row is loaded once for the R queries that read it.
// tab: the warp's table (row stride QW).
template <bool SPLIT, typename T>
__device__ __forceinline__ void add_window(const Place<SPLIT>& p, float2 (&acc)[R][4], const T* base, int T_, int t0,
                                           int t1, const float* tab) {
    constexpr int kBatch = Lane<T>::kBatch;
    const int n = R - 1 + t1 - t0, jw = p.iw - (t1 - 1);
    const float* tabg = tab + p.g * R;
#pragma unroll 1
    for (int y0 = p.first * kBatch; y0 < n; y0 += p.step * kBatch) {
        typename Lane<T>::Raw row[kBatch];
        load_rows<kBatch>(base, jw + p.g * R + y0, jw + y0, jw + 3 * R + y0 + kBatch - 1, T_, p.c, row);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            float2 x[4];
            Lane<T>::expand(row[u], x);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int t = r + t1 - 1 - (y0 + u);          // warp-uniform
                if (t >= t0 && t < t1) axpy(tabg[(t - t0) * QW + r], x, acc[r]);
            }
        }
    }
}

// acc[r] += tab[n][r] ((1 - w) row(i - s0) + w row(i - s0 - 1)) over the
// active rungs, for the queries i they are attended from (d <= i).  kPair
// rungs at a time.
template <bool SPLIT, typename T>
__device__ __forceinline__ void add_rungs(const Place<SPLIT>& p, float2 (&acc)[R][4], const T* base, int T_,
                                          const RungList& L, const float* tab) {
    constexpr int NP = Lane<T>::kPair;
    const int i0 = p.iw + p.g * R;
    const float dmax = (float)(p.iw + QW - 1);
#pragma unroll 1
    for (int n0 = p.first * NP; n0 < L.n; n0 += p.step * NP) {
        typename Lane<T>::Raw row[NP][R + 1];
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int jw = p.iw - L.s0[n0 + u] - 1;
            if (n0 + u < L.n && L.d[n0 + u] <= dmax)          // warp-uniform
                load_rows<R + 1>(base, jw + p.g * R, jw, jw + QW, T_, p.c, row[u]);
        }
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            if (n0 + u >= L.n || L.d[n0 + u] > dmax) continue;
            const float d = L.d[n0 + u], w = L.w[n0 + u];
            const float* q = tab + (n0 + u) * QW + p.g * R;
            const bool all = d <= (float)p.iw;                // warp-uniform
#pragma unroll
            for (int r = 0; r <= R; ++r) {                    // row r: far of query r, floor of query r - 1
                float2 x[4];
                Lane<T>::expand(row[u][r], x);
                if (r < R && w != 0.f && (all || d <= (float)(i0 + r))) axpy(q[r] * w, x, acc[r]);
                if (r > 0 && (all || d <= (float)(i0 + r - 1))) axpy(q[r - 1] * (1.f - w), x, acc[r - 1]);
            }
        }
    }
}

// SPLIT: adds up the warps' partial sums; the group then holds row
// 4 warp + g of the block's 16 in acc[0].  red: kWarps QW kHeadDim floats.
__device__ __forceinline__ void join(const Place<true>& p, float2 (&acc)[R][4], float* red) {
    float4* r4 = reinterpret_cast<float4*>(red);
    __syncthreads();                                          // the last reads of red are done
#pragma unroll
    for (int r = 0; r < R; ++r) {
        float4* to = r4 + ((p.warp * QW + p.g * R + r) * 8 + p.c) * 2;
        to[0] = make_float4(acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y);
        to[1] = make_float4(acc[r][2].x, acc[r][2].y, acc[r][3].x, acc[r][3].y);
    }
    __syncthreads();
    float4 x[kWarps][2];
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const float4* from = r4 + ((w * QW + p.warp * kGroups + p.g) * 8 + p.c) * 2;
        x[w][0] = from[0]; x[w][1] = from[1];
    }
    auto sum = [&](int h, float float4::*e) { return (x[0][h].*e + x[1][h].*e) + (x[2][h].*e + x[3][h].*e); };
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        acc[0][2 * h] = make_float2(sum(h, &float4::x), sum(h, &float4::y));
        acc[0][2 * h + 1] = make_float2(sum(h, &float4::z), sum(h, &float4::w));
    }
}
static_assert(kWarps == 4 && QW == kWarps * kGroups, "a group joins one row of the block's");

// f(r, i) for the rows i of the sequence that a group writes, which acc[r]
// holds: its R, or (SPLIT) the one it joined.
template <bool SPLIT, typename F>
__device__ __forceinline__ void each_row(const Place<SPLIT>& p, int T_, F f) {
#pragma unroll
    for (int r = 0; r < (SPLIT ? 1 : R); ++r) {
        const int i = SPLIT ? p.iw + p.warp * kGroups + p.g : p.iw + p.g * R + r;
        if (i < T_) f(r, i);
    }
}
// Scales those rows and rotates them back.
template <typename T, bool SPLIT>
__device__ __forceinline__ void rotate_back(const Place<SPLIT>& p, const RopeParams& rp, float sc, float2 (&acc)[R][4]) {
#pragma unroll
    for (int r = 0; r < (SPLIT ? 1 : R); ++r) scale(sc, acc[r]);
    if constexpr (SPLIT) {
        float2 one[1][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) one[0][e] = acc[0][e];
        Lane<T>::rope(rp, p.iw + p.warp * kGroups + p.g, p.c, one, true);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[0][e] = one[0][e];
    } else {
        Lane<T>::rope(rp, p.iw + p.g * R, p.c, acc, true);
    }
}

// ------------------------------------------------------------- forward ----

// Shared table: [slots of a chunk, then active rungs][QW rows], a warp's or
// (SPLIT) the block's; SPLIT: then the row sums of the warps, and the join.
// MULTI: the window takes more than one chunk (not with SPLIT).
template <typename T, bool SPLIT, bool MULTI>
__global__ void __launch_bounds__(kWarps * 32, MULTI ? 2 : 4) fwd_gather_kernel(FwdArgs a, RungList L, int chunk) {
    grid_dependency_sync();
    extern __shared__ __align__(16) float tab_all[];
    const Shape& s = a.s;
    const int tiles = (s.T + kTileRows16<SPLIT> - 1) / kTileRows16<SPLIT>;
    const int bh = blockIdx.x / tiles;
    const Place<SPLIT> p(blockIdx.x - bh * tiles);
    if (p.iw >= s.T) return;                                  // (SPLIT: the whole block, which has no such tile)
    const int b = bh / s.H, hk = (bh - b * s.H) / s.G;
    const size_t rows = (size_t)(chunk + L.n) * QW;
    float* tab = SPLIT ? tab_all + kWarps * QW * kHeadDim : tab_all + p.warp * rows;
    float* own = tab + (p.row - p.iw);                        // the lane's own column

    const T* Q = reinterpret_cast<const T*>(a.q) + (size_t)bh * s.T * kHeadDim;
    using KT = typename RotOf<T>::type;
    const KT* Kt = reinterpret_cast<const KT*>(a.kt) + (size_t)(b * s.Hkv + hk) * s.T * kHeadDim;
    const T* V = reinterpret_cast<const T*>(a.v) + (size_t)(b * s.Hkv + hk) * s.T * kHeadDim;

    float2 q[R][4], acc[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = min(p.iw + p.g * R + r, s.T - 1);
        load_row(Q + (size_t)i * kHeadDim, p.c, q[r]);
    }
    Lane<T>::rope(a.rope, p.iw + p.g * R, p.c, q, false);
    if constexpr (MULTI) clear(acc);
    const float sc2 = s.scale * kLog2e;                       // scores stay raw until p = 2^(sc2 (s - max))
    const bool vo = p.row < s.T;
    float m = -INFINITY, l = 0.f;                             // of the lane's own row

    const int slots = p.query_slots(s);
    for (int t0 = 0; t0 < slots; t0 += chunk) {
        const int t1 = MULTI ? min(slots, t0 + chunk) : slots;
        const bool last = !MULTI || t1 == slots;
        const float m_old = m;
        // ---- scores of the chunk's window slots, and of the rungs at the end
        auto put = [&](int n, float sco) {
            m = fmaxf(m, sco);
            if (p.writer) own[n * QW] = sco;
        };
        const int nw = t1 - t0;
        dot_window(p, q, Kt, s.T, t0, t1,
                   [&](int t, float x) { put(t - t0, (vo && p.row >= t) ? x : -INFINITY); });
        if (last) {
            dot_rungs(p, q, Kt, s.T, L,
                      [&](int n, float x0, float x1) {
                          const float w = L.w[n];
                          float x = (1.f - w) * x0;
                          if (w != 0.f) x = fmaf(w, x1, x);
                          put(nw + n, (vo && L.d[n] <= (float)p.row) ? x : -INFINITY);
                      },
                      [&](int n) { put(nw + n, -INFINITY); });
        }
        p.sync();
        const int ns = nw + (last ? L.n : 0);
        if constexpr (SPLIT) {                                // the other warps' scores
            for (int n = p.c & 1; n < ns; n += 2) m = fmaxf(m, own[n * QW]);
            m = fmaxf(m, __shfl_xor_sync(kAll, m, 1));
            __syncthreads();
        }
        // ---- p = 2^(sc2 (s - max)): the lanes of a row take its slots in turn
        const float mm = m == -INFINITY ? 0.f : m;
        float part = 0.f;
        for (int n = 2 * p.first + (p.c & 1); n < ns; n += 2 * p.step) {
            const float e = exp2f((own[n * QW] - mm) * sc2);
            own[n * QW] = e;
            part += e;
        }
        part += __shfl_xor_sync(kAll, part, 1);
        if constexpr (SPLIT) {
            float* ls = tab + rows;
            if (p.writer) ls[p.warp * QW + p.row - p.iw] = part;
            __syncthreads();
            const float* lr = ls + (p.row - p.iw);
            part = (lr[0] + lr[QW]) + (lr[2 * QW] + lr[3 * QW]);
        }
        if (MULTI && t0 > 0) {                                // rescale what earlier chunks added
            const float corr = m_old == -INFINITY ? 0.f : exp2f((m_old - mm) * sc2);
            l = l * corr + part;
#pragma unroll
            for (int r = 0; r < R; ++r) scale(__shfl_sync(kAll, corr, (p.lane & ~7) | (2 * r)), acc[r]);
        } else {
            l = part;
        }
        p.sync();
        // ---- values
        if constexpr (!MULTI) clear(acc);
        add_window(p, acc, V, s.T, t0, t1, tab);
        if (last) add_rungs(p, acc, V, s.T, L, tab + nw * QW);
        if (!MULTI) break;
        __syncwarp();                                         // the table is read before it is rewritten
    }
    const float inv = 1.f / l;
    T* O = reinterpret_cast<T*>(a.out) + (size_t)bh * s.T * kHeadDim;
    if constexpr (SPLIT) join(p, acc, tab_all);
    // 1 / l of row r sits in lanes 2r of its group; SPLIT: of row 4 warp + g in
    // lane 2g of group `warp` (every warp has them all)
#pragma unroll
    for (int r = 0; r < (SPLIT ? 1 : R); ++r)
        scale(__shfl_sync(kAll, inv, SPLIT ? p.warp * 8 + 2 * p.g : (p.lane & ~7) | (2 * r)), acc[r]);
    each_row(p, s.T, [&](int r, int i) { Lane<T>::store(O + (size_t)i * kHeadDim, p.c, acc[r]); });
    if (p.writer && vo && (!SPLIT || p.warp == 0)) a.lse[(size_t)bh * s.T + p.row] = fmaf(m, s.scale, logf(l));
}

// ------------------------------------------------------------ backward ----

// Query pass.  With p = exp(score - lse), dp = dO . val, Delta = sum p dp and
// dS = p (dp - Delta) per slot,
//   dq~ = scale sum_slots dS key,
//   dL/dd_k += p (scale (s1 - s0) (dp - Delta) + dp1 - dp0)
// (s1, s0, dp1, dp0: the far and floor rows' raw products; row -1 is a zero
// row).  One sweep over key rows forms p, one over value rows dp and Delta,
// and one more over key rows adds them by dS.  p and dS go to the workspace,
// slot-major, and so do the rotated queries.
// Shared tables (a warp's, SPLIT: the block's): p, then dp (then dS), [slots of
// a chunk, active rungs][QW rows] each; with DD s1 - s0 and dp1 - dp0 of the
// rungs; Delta (SPLIT: of each warp's slots).
template <typename T, bool SPLIT, bool DD>
__global__ void __launch_bounds__(kWarps * 32, 4) bwd_query_gather_kernel(BwdArgs a, RungList L, int chunk) {
    grid_dependency_sync();
    extern __shared__ __align__(16) float tab_all[];
    __shared__ float gsm[kWarps][kMaxRungs];                  // per-warp rung-gradient sums
    const Shape& s = a.s;
    const int tiles = (s.T + kTileRows16<SPLIT> - 1) / kTileRows16<SPLIT>;
    const int bh = blockIdx.x / tiles;
    const Place<SPLIT> p(blockIdx.x - bh * tiles);
    const int ns_max = chunk + L.n;
    const size_t words = (size_t)(2 * ns_max + (DD ? 2 * L.n : 0) + (SPLIT ? kWarps : 1)) * QW;
    float* ptab = SPLIT ? tab_all + kWarps * QW * kHeadDim : tab_all + p.warp * words;
    float* dtab = ptab + ns_max * QW;
    float* stab = dtab + ns_max * QW;                         // DD: s1 - s0, then dp1 - dp0
    float* delta_s = stab + (DD ? 2 * L.n * QW : 0);
    if (DD && p.lane < L.n) gsm[p.warp][p.lane] = 0.f;
    if (p.iw < s.T) {                                         // (SPLIT: always)
        const int b = bh / s.H, hk = (bh - b * s.H) / s.G;
        using KT = typename RotOf<T>::type;
        const T* Q = reinterpret_cast<const T*>(a.q) + (size_t)bh * s.T * kHeadDim;
        const T* dO = reinterpret_cast<const T*>(a.dout) + (size_t)bh * s.T * kHeadDim;
        const KT* Kt = reinterpret_cast<const KT*>(a.kt) + (size_t)(b * s.Hkv + hk) * s.T * kHeadDim;
        const T* V = reinterpret_cast<const T*>(a.v) + (size_t)(b * s.Hkv + hk) * s.T * kHeadDim;
        KT* Qt = reinterpret_cast<KT*>(a.qt) + (size_t)bh * s.T * kHeadDim;
        float* Pg = a.Ps + (size_t)bh * a.S * s.T;            // [slot][T] of this head
        float* DSg = a.DSs + (size_t)bh * a.S * s.T;

        const bool vo = p.row < s.T;
        const float lse = vo ? a.lse[(size_t)bh * s.T + p.row] : 0.f;
        auto prob = [&](float x) { return exp2f(fmaf(x, s.scale, -lse) * kLog2e); };
        // a lane's place in a sweep over the table: row ql, slots sl, sl + sstep, ...
        const int ql = p.lane & (QW - 1), sl = 2 * p.first + p.lane / QW, sstep = 2 * p.step;
        const int iq = p.iw + ql;
        float* po = ptab + (p.row - p.iw);                    // the lane's own column of the tables
        float* dpo = dtab + (p.row - p.iw);
        float* so = stab + (p.row - p.iw);

        // ---- p of every slot (key rows)
        float2 vec[R][4];
        float qmax = 0.f;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = min(p.iw + p.g * R + r, s.T - 1);
            load_row(Q + (size_t)i * kHeadDim, p.c, vec[r]);
        }
        Lane<T>::rope(a.rope, p.iw + p.g * R, p.c, vec, false);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = p.iw + p.g * R + r;
            if (i >= s.T) continue;
            if (!SPLIT || p.warp == 0) Lane<KT>::store(Qt + (size_t)i * kHeadDim, p.c, vec[r]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                qmax = fmaxf(qmax, fmaxf(fabsf(vec[r][e].x), fabsf(vec[r][e].y)));
                if constexpr (sizeof(KT) == 2) vec[r][e] = __half22float2(__float22half2_rn(vec[r][e]));   // as stored
            }
        }
        if (sizeof(KT) == 2 && qmax >= 65520.f) raise_status(a.status, kStatusRange);   // fp16 rows hold < 65520
        const int slots = p.query_slots(s);
        const int n_chunks = (slots + chunk - 1) / chunk;     // 1 with SPLIT
        const int tl = (n_chunks - 1) * chunk, nw = slots - tl;     // the last chunk's window slots
        // a chunk's table to the workspace, where it waits for Delta
        auto spill = [&](const float* tab, float* to, int t0) {
            __syncwarp();
            for (int u = sl; u < chunk; u += sstep)
                if (iq < s.T) to[(size_t)(t0 + u) * s.T + iq] = tab[u * QW + ql];
            __syncwarp();
        };
        for (int t0 = 0; t0 < slots; t0 += chunk) {
            dot_window(p, vec, Kt, s.T, t0, min(slots, t0 + chunk), [&](int t, float x) {
                const float e = (vo && p.row >= t) ? prob(x) : 0.f;
                if (p.writer) po[(t - t0) * QW] = e;
            });
            if (t0 < tl) spill(ptab, Pg, t0);
        }
        auto skip = [&](float* tab, float* d) {
            return [=](int n) {
                if (p.writer) {
                    tab[(nw + n) * QW] = 0.f;
                    if (DD) d[n * QW] = 0.f;
                }
            };
        };
        dot_rungs(p, vec, Kt, s.T, L,
                  [&](int n, float x0, float x1) {
                      const float w = L.w[n];
                      const bool ok = vo && L.d[n] <= (float)p.row;
                      const float e = ok ? prob((1.f - w) * x0 + w * x1) : 0.f;
                      if (p.writer) {
                          po[(nw + n) * QW] = e;
                          if (DD) so[n * QW] = ok ? x1 - x0 : 0.f;
                      }
                  }, skip(po, so));
        p.sync();
        // ---- dp of every slot (value rows) and Delta
#pragma unroll
        for (int r = 0; r < R; ++r) load_row(dO + (size_t)min(p.iw + p.g * R + r, s.T - 1) * kHeadDim, p.c, vec[r]);
        float delta = 0.f;
        for (int t0 = 0; t0 < slots; t0 += chunk) {
            const bool here = t0 == tl;
            dot_window(p, vec, V, s.T, t0, min(slots, t0 + chunk), [&](int t, float x) {
                const float dp = (vo && p.row >= t) ? x : 0.f;
                const float e = here ? po[(t - t0) * QW] : vo ? Pg[(size_t)t * s.T + p.row] : 0.f;
                delta = fmaf(e, dp, delta);
                if (p.writer) dpo[(t - t0) * QW] = dp;
            });
            if (!here) spill(dtab, DSg, t0);
        }
        float* so1 = so + L.n * QW;
        dot_rungs(p, vec, V, s.T, L,
                  [&](int n, float x0, float x1) {
                      const float w = L.w[n];
                      const bool ok = vo && L.d[n] <= (float)p.row;
                      const float dp = ok ? (1.f - w) * x0 + w * x1 : 0.f;
                      delta = fmaf(po[(nw + n) * QW], dp, delta);
                      if (p.writer) {
                          dpo[(nw + n) * QW] = dp;
                          if (DD) so1[n * QW] = ok ? x1 - x0 : 0.f;
                      }
                  }, skip(dpo, so1));
        if (p.writer) delta_s[(SPLIT ? p.warp * QW : 0) + p.row - p.iw] = delta;
        p.sync();
        // ---- dS of the last chunk and the rungs; p and dS to the workspace
        float dlt = delta_s[ql];
        if constexpr (SPLIT) dlt = (dlt + delta_s[QW + ql]) + (delta_s[2 * QW + ql] + delta_s[3 * QW + ql]);
        const int tot = nw + L.n;
        for (int u0 = sl - p.lane / QW; u0 < tot; u0 += sstep) {      // uniform over the warp
            const int u = u0 + p.lane / QW;
            const bool in = u < tot, rung = in && u >= nw;
            const float e = in ? ptab[u * QW + ql] : 0.f, f = in ? dtab[u * QW + ql] - dlt : 0.f;
            const float ds = e * f;
            if (in) dtab[u * QW + ql] = ds;
            if (in && iq < s.T) {
                const int slot = rung ? s.W + 1 + L.k[u - nw] : tl + u;
                Pg[(size_t)slot * s.T + iq] = e;
                DSg[(size_t)slot * s.T + iq] = ds;
            }
            if constexpr (DD) {                               // the rung's sum over the warp's queries
                float x = 0.f;
                if (rung) x = e * fmaf(s.scale * stab[(u - nw) * QW + ql], f, stab[(L.n + u - nw) * QW + ql]);
#pragma unroll
                for (int o = QW / 2; o > 0; o >>= 1) x += __shfl_xor_sync(kAll, x, o);
                if (rung && ql == 0) gsm[p.warp][u - nw] = x;
            }
        }
        p.sync();
        // ---- dq~ += dS key rows
        float2 acc[R][4];
        clear(acc);
        add_window(p, acc, Kt, s.T, tl, slots, dtab);
        add_rungs(p, acc, Kt, s.T, L, dtab + nw * QW);
        for (int ch = 0; ch + 1 < n_chunks; ++ch) {           // the earlier chunks, from the workspace
            const int t0 = ch * chunk, t1 = t0 + chunk;
            __syncwarp();
            for (int u = sl; u < chunk; u += sstep) {
                const size_t at = (size_t)(t0 + u) * s.T + iq;
                const float ds = iq < s.T ? Pg[at] * (DSg[at] - dlt) : 0.f;
                dtab[u * QW + ql] = ds;
                if (iq < s.T) DSg[at] = ds;
            }
            __syncwarp();
            add_window(p, acc, Kt, s.T, t0, t1, dtab);
        }
        if constexpr (SPLIT) join(p, acc, tab_all);
        T* dQ = reinterpret_cast<T*>(a.dq) + (size_t)bh * s.T * kHeadDim;
        rotate_back<T>(p, a.rope, s.scale, acc);
        each_row(p, s.T, [&](int r, int i) { Lane<T>::store(dQ + (size_t)i * kHeadDim, p.c, acc[r]); });
    }
    if constexpr (DD) {                                       // per-block rung partials, warps in a fixed order
        __syncthreads();
        const int k = threadIdx.x;
        if (k < a.r.K) {
            float x = 0.f;
            for (int n = 0; n < L.n; ++n)
                if (L.k[n] == k)
                    for (int w = 0; w < kWarps; ++w) x += gsm[w][n];
            a.rpart[(size_t)k * a.nblk_q + blockIdx.x] = __float2ll_rn(x * 4294967296.0f);
        }
    }
}

// Key pass.  Key row j receives, from every query head of its group, the slots
// that read it: window slot t of query j + t (weight 1), rung k of query
// j + s0_k (floor row, weight 1 - w_k) and of query j + s0_k + 1 (far row,
// weight w_k):  dk~_j = scale sum c dS q~_i,  dv_j = sum c p dO_i.  R
// consecutive keys share the query rows as R queries share key rows above.
// Shared table (a warp's, SPLIT: the block's): dS or p [window slots of a
// chunk, then each rung's as its floor and as its far row][QW keys].
template <typename T, bool SPLIT>
__global__ void __launch_bounds__(kWarps * 32, 4) bwd_key_gather_kernel(BwdArgs a, RungList L, int chunk) {
    grid_dependency_sync();
    extern __shared__ __align__(16) float tab_all[];
    const Shape& s = a.s;
    if (a.want_dd && blockIdx.x == 0) {                       // the first block only adds up the rung partials
        __shared__ double red[kMaxRungs];
        convert_rung_sums(a, red);
        return;
    }
    const int blk = (int)blockIdx.x - (a.want_dd ? 1 : 0);
    const int tiles = (s.T + kTileRows16<SPLIT> - 1) / kTileRows16<SPLIT>;
    const int bhk = blk / tiles;                              // b Hkv + hk
    const Place<SPLIT> p(blk - bhk * tiles);
    if (p.iw >= s.T) return;                                  // (SPLIT: no such tile)
    const int jw = p.iw, j0 = jw + p.g * R;
    const int b = bhk / s.Hkv, hk = bhk - b * s.Hkv;
    float* tab = SPLIT ? tab_all + kWarps * QW * kHeadDim : tab_all + (size_t)p.warp * ((chunk + 2 * L.n) * QW);
    float* tabg = tab + p.g * R;
    const int kl = p.lane & (QW - 1), sl = 2 * p.first + p.lane / QW;   // a lane's key and first slot in a sweep
    const int slots = p.key_slots(s);

    // One output (dk~ from q~ rows and dS, then dv from dO rows and p) of the
    // warp's keys; weights: slot-major, S T values a head.
    auto sum = [&](const auto* rows, const float* weights, float2 (&acc)[R][4]) {
        using X = std::remove_cv_t<std::remove_reference_t<decltype(*rows)>>;
        constexpr int kBatch = Lane<X>::kBatch, NP = Lane<X>::kPair;
        clear(acc);
        for (int gq = 0; gq < s.G; ++gq) {
            const size_t bh = (size_t)b * s.H + hk * s.G + gq;
            const auto* base = rows + bh * s.T * kHeadDim;
            const float* Xh = weights + bh * a.S * s.T;
            for (int t0 = 0; t0 < slots; t0 += chunk) {
                const int t1 = min(slots, t0 + chunk), nw = t1 - t0;
                const int nr = t1 == slots ? L.n : 0;
                // ---- the weights of the keys, all copies in flight together
                for (int u = sl; u < nw + 2 * nr; u += 2 * p.step) {
                    const int rr = u - nw, n = rr >> 1;
                    const int slot = rr < 0 ? t0 + u : s.W + 1 + L.k[n];
                    const int i = jw + kl + (rr < 0 ? t0 + u : L.s0[n] + (rr & 1));
                    const bool in = i < s.T;
                    mma::cp_async4(tab + u * QW + kl, Xh + (in ? (unsigned)slot * s.T + i : 0u), in);
                }
                asm volatile("cp.async.commit_group;\n" ::: "memory");
                asm volatile("cp.async.wait_group 0;\n" ::: "memory");
                p.sync();
                // ---- window: query j0 + t0 + y is slot t0 + y - r of key r
                const int n = nw + R - 1;
#pragma unroll 1
                for (int y0 = p.first * kBatch; y0 < n; y0 += p.step * kBatch) {
                    typename Lane<X>::Raw row[kBatch];
                    load_rows<kBatch>(base, j0 + t0 + y0, jw + t0 + y0, jw + 3 * R + t0 + y0 + kBatch - 1, s.T, p.c, row);
#pragma unroll
                    for (int u = 0; u < kBatch; ++u) {
                        float2 x[4];
                        Lane<X>::expand(row[u], x);
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const int t = y0 + u - r;         // relative to t0; warp-uniform
                            if (t >= 0 && t < nw) axpy(tabg[t * QW + r], x, acc[r]);
                        }
                    }
                }
                // ---- rungs: query j0 + s0 + u reads key u as its floor row and key u - 1 as its far row
#pragma unroll 1
                for (int m0 = p.first * NP; m0 < nr; m0 += p.step * NP) {
                    typename Lane<X>::Raw row[NP][R + 1];
#pragma unroll
                    for (int v = 0; v < NP; ++v) {
                        const int iw = jw + L.s0[m0 + v];
                        if (m0 + v < nr && iw < s.T)          // warp-uniform
                            load_rows<R + 1>(base, iw + p.g * R, iw, iw + QW, s.T, p.c, row[v]);
                    }
#pragma unroll
                    for (int v = 0; v < NP; ++v) {
                        if (m0 + v >= nr || jw + L.s0[m0 + v] >= s.T) continue;
                        const float* t = tabg + (nw + 2 * (m0 + v)) * QW;
                        const float w = L.w[m0 + v];
#pragma unroll
                        for (int r = 0; r <= R; ++r) {
                            float2 x[4];
                            Lane<X>::expand(row[v][r], x);
                            if (r < R) axpy((1.f - w) * t[r], x, acc[r]);
                            if (r > 0 && w != 0.f) axpy(w * t[QW + r - 1], x, acc[r - 1]);
                        }
                    }
                }
                p.sync();                                     // the table is read before it is rewritten
            }
        }
        if constexpr (SPLIT) join(p, acc, tab_all);
    };
    using KT = typename RotOf<T>::type;
    const size_t off = (size_t)bhk * s.T * kHeadDim;
    float2 acc[R][4];
    sum(reinterpret_cast<const KT*>(a.qt), a.DSs, acc);
    rotate_back<T>(p, a.rope, s.scale, acc);
    each_row(p, s.T, [&](int r, int j) { Lane<T>::store(reinterpret_cast<T*>(a.dk) + off + (size_t)j * kHeadDim, p.c, acc[r]); });
    sum(reinterpret_cast<const T*>(a.dout), a.Ps, acc);
    each_row(p, s.T, [&](int r, int j) { Lane<T>::store(reinterpret_cast<T*>(a.dv) + off + (size_t)j * kHeadDim, p.c, acc[r]); });
}

// ------------------------------------------------------------ host side ----

// Window slots that any row has.  Tables are made for these, not for the window,
// and so is the choice of the kernel: at T 20 and W 1024 (fp32 B64 H16 Hkv2) tables
// of kChunk slots left one block an SM, forward 34.5 us, backward 114.7; now 15.7
// and 62.1.  B4 H8 T128 W1024, whose rows are now shared: 30 -> 13 us, 88 -> 39.
int window_slots(const Shape& s) { return std::min(s.W + 1, s.T); }

// Whether the warps of a block share their rows: while the blocks that takes
// all fit the GPU at once (four on each of 152 SMs; a constant, because the
// size of the workspace depends on it).  A training layer (fp32, W 8, H 8,
// T 1000) split / not: B1, 504 blocks, 36 / 56 us; B2, 1008 blocks, 62.9 /
// 66.8 us, but its key pass 22.5 / 18.6 us; B3, 1512 blocks, 86.9 / 73.7 us.
bool split_rows(const Shape& s, int heads) {
    return window_slots(s) <= kChunk && (long long)((s.T + QW - 1) / QW) * heads <= 4 * 152;
}

int blocks_of(const Shape& s, int heads) {
    const int rows = split_rows(s, heads) ? QW : kWarps * QW;
    return (int)((long long)((s.T + rows - 1) / rows) * heads);
}

// Shared memory of a block: tables of `words` rows of QW floats a warp (SPLIT:
// a block, with the join's and the warps' row sums).
size_t smem_of(bool split, size_t words) {
    return sizeof(float) * QW * (split ? kWarps * kHeadDim + words + kWarps : kWarps * words);
}

// words(window slots of the table, rungs): the rows a kernel's table has.
template <typename A, typename Words>
cudaError_t launch(void (*kern)(A, RungList, int), int grid, bool split, Words words, cudaStream_t st, const A& a,
                   const RungList& L, int chunk) {
    return launch_kernel_dynamic(kern, dim3((unsigned)grid), dim3(kWarps * 32), smem_of(split, words(chunk, L.n)),
                                 smem_of(split, words(kChunk, kMaxRungs)), st, a, L, chunk);
}

template <typename T>
cudaError_t launch_fwd(const FwdArgs& a, cudaStream_t st) {
    const RungList L = rung_list(a.r);
    const int heads = a.s.B * a.s.H, chunk = std::min(window_slots(a.s), kChunk);
    const bool split = split_rows(a.s, heads);
    auto kern = split ? fwd_gather_kernel<T, true, false>
                      : window_slots(a.s) > chunk ? fwd_gather_kernel<T, false, true> : fwd_gather_kernel<T, false, false>;
    return launch(kern, blocks_of(a.s, heads), split, [](size_t w, size_t n) { return w + n; }, st, a, L, chunk);
}

template <typename T>
cudaError_t launch_query(const BwdArgs& a, cudaStream_t st) {
    const RungList L = rung_list(a.r);
    const int heads = a.s.B * a.s.H, chunk = std::min(window_slots(a.s), kChunk);
    const bool split = split_rows(a.s, heads), dd = a.want_dd;
    auto kern = split ? (dd ? bwd_query_gather_kernel<T, true, true> : bwd_query_gather_kernel<T, true, false>)
                      : (dd ? bwd_query_gather_kernel<T, false, true> : bwd_query_gather_kernel<T, false, false>);
    return launch(kern, blocks_of(a.s, heads), split,
                  [dd](size_t w, size_t n) { return 2 * (w + n) + (dd ? 2 * n : 0) + 1; }, st, a, L, chunk);
}

template <typename T>
cudaError_t launch_key(const BwdArgs& a, cudaStream_t st) {
    const RungList L = rung_list(a.r);
    const int heads = a.s.B * a.s.Hkv, chunk = std::min(window_slots(a.s), kChunk);
    const bool split = split_rows(a.s, heads);
    auto kern = split ? bwd_key_gather_kernel<T, true> : bwd_key_gather_kernel<T, false>;
    return launch(kern, blocks_of(a.s, heads) + (a.want_dd ? 1 : 0), split,
                  [](size_t w, size_t n) { return w + 2 * n; }, st, a, L, chunk);
}

}  // namespace

int bwd_gather_blocks(const Shape& s) { return blocks_of(s, s.B * s.H); }

cudaError_t launch_fwd_gather(const FwdArgs& a, bool bf16, cudaStream_t st) {
    if ((long long)a.s.B * a.s.H * a.s.T <= 0) return cudaSuccess;
    return bf16 ? launch_fwd<__nv_bfloat16>(a, st) : launch_fwd<float>(a, st);
}
cudaError_t launch_bwd_query_gather(const BwdArgs& a, bool bf16, cudaStream_t st) {
    if ((long long)a.s.B * a.s.H * a.s.T <= 0) return cudaSuccess;
    return bf16 ? launch_query<__nv_bfloat16>(a, st) : launch_query<float>(a, st);
}
cudaError_t launch_bwd_key_gather(const BwdArgs& a, bool bf16, cudaStream_t st) {
    if ((long long)a.s.B * a.s.H * a.s.T <= 0) return cudaSuccess;
    return bf16 ? launch_key<__nv_bfloat16>(a, st) : launch_key<float>(a, st);
}

}  // namespace fibattn

// kernels_simple.cu -- the RoPE prologue (arXiv 2606.28560, Section 2): rotates
// the rows of k into the library's score operands before a pass gathers them.
#include <algorithm>

#include "fibattn_internal.cuh"

namespace fibattn {

namespace {

// ---------------------------------------------------------------- RoPE ----

// bf16 rows in, fp16 rotated rows out.  A block tile is kRopePos consecutive
// positions of TH heads: the tile's cos/sin (one pair and position per
// thread, evaluated before the wait for the previous kernel) go to shared
// memory, and every row of the tile reads them from there, so an angle is
// evaluated once per tile instead of once per head.  Thread item = (head,
// position, chunk c): dims 8c..8c+7 and their RoPE partners 32+8c..32+8c+7;
// a warp covers the tile's 8 positions x 4 chunks of one head (1 KB
// contiguous), and a thread issues the loads of all its items (TH / 8)
// before any arithmetic.  Four blocks an SM (64 registers; 70 allowed three):
// the 512 tiles of B16 H8 T1024 are then all resident at once, where the last
// 56 had to wait for a slot (forward with the rotation 38.7 -> 38.3 us, at B4
// T4096 41.2 -> 40.6 us).
constexpr int kRopePos = 8;
constexpr int kRopeTabStride = 34;            // floats per position (32 + pad: conflict-free float2 reads)
template <int TH>
__global__ void __launch_bounds__(256, 4) rope_rows_bf16_kernel(const __nv_bfloat16* __restrict__ src,
                                                             __half* __restrict__ dst, int heads, int T_,
                                                             RopeParams rp, unsigned* status) {
    constexpr int kItems = TH / 8;                // per thread (256 threads)
    __shared__ __align__(16) float ctab[kRopePos * kRopeTabStride], stab[kRopePos * kRopeTabStride];
    const int tid = threadIdx.x;
    const int c = tid & 3, pr = (tid >> 2) & 7, hr0 = tid >> 5;
    const int tiles_p = (T_ + kRopePos - 1) / kRopePos;
    const long long tiles = (long long)tiles_p * ((heads + TH - 1) / TH);
    float rmax = 0.f;                             // largest |rotated entry|: fp16 holds < 65520
    bool waited = false;
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int tp = (int)(tile % tiles_p), th = (int)(tile / tiles_p);
        const int p0 = tp * kRopePos, h0 = th * TH;
        {                                         // pair m = tid & 31 at position p0 + (tid >> 5)
            float cs, sn;
            rope_cs(rp, tid & 31, p0 + (tid >> 5), cs, sn);
            ctab[(tid >> 5) * kRopeTabStride + (tid & 31)] = cs;
            stab[(tid >> 5) * kRopeTabStride + (tid & 31)] = sn;
        }
        if (!waited) {
            grid_dependency_sync();
            waited = true;
        }
        const int p = p0 + pr;
        uint4 raw[kItems][2];
#pragma unroll
        for (int u = 0; u < kItems; ++u) {
            const int h = h0 + hr0 + 8 * u;
            if (h < heads && p < T_) {
                const __nv_bfloat16* row = src + ((size_t)h * T_ + p) * kHeadDim;
                raw[u][0] = *reinterpret_cast<const uint4*>(row + 8 * c);
                raw[u][1] = *reinterpret_cast<const uint4*>(row + kHalf + 8 * c);
            }
        }
        __syncthreads();                          // the tile's cos/sin are in shared memory
        const float2* cp = reinterpret_cast<const float2*>(ctab + pr * kRopeTabStride + 8 * c);
        const float2* sp = reinterpret_cast<const float2*>(stab + pr * kRopeTabStride + 8 * c);
        // The thread's items share their position.  With two items their angles,
        // read once, fit the 64 registers (B2 H8 T16384: this kernel 16.7 -> 16.1 us,
        // a layer's forward and backward 305.9 -> 304.6 at W 0, 274.0 -> 273.4 at W 8);
        // with four they spill (forward B16 H8 T1024 38.0 -> 41.0 us).
        constexpr bool kKeep = kItems <= 2;
        float2 cv[4], sv[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if constexpr (kKeep) { cv[e] = cp[e]; sv[e] = sp[e]; }
        }
#pragma unroll
        for (int u = 0; u < kItems; ++u) {
            const int h = h0 + hr0 + 8 * u;
            if (h >= heads || p >= T_) continue;
            const unsigned* wa = reinterpret_cast<const unsigned*>(&raw[u][0]);
            const unsigned* wb = reinterpret_cast<const unsigned*>(&raw[u][1]);
            unsigned oa[4], ob[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float a0 = __uint_as_float(wa[e] << 16), a1 = __uint_as_float(wa[e] & 0xffff0000u);
                const float b0 = __uint_as_float(wb[e] << 16), b1 = __uint_as_float(wb[e] & 0xffff0000u);
                // pairs (8c + 2e, 32 + 8c + 2e) and the next
                const float2 ce = kKeep ? cv[e] : cp[e], se = kKeep ? sv[e] : sp[e];
                const float xa0 = a0 * ce.x - b0 * se.x, xa1 = a1 * ce.y - b1 * se.y;
                const float xb0 = b0 * ce.x + a0 * se.x, xb1 = b1 * ce.y + a1 * se.y;
                rmax = fmaxf(rmax, fmaxf(fmaxf(fabsf(xa0), fabsf(xa1)), fmaxf(fabsf(xb0), fabsf(xb1))));
                __half2 ra = __floats2half2_rn(xa0, xa1);
                __half2 rb = __floats2half2_rn(xb0, xb1);
                oa[e] = *reinterpret_cast<unsigned*>(&ra);
                ob[e] = *reinterpret_cast<unsigned*>(&rb);
            }
            __half* row = dst + ((size_t)h * T_ + p) * kHeadDim;
            *reinterpret_cast<uint4*>(row + 8 * c) = make_uint4(oa[0], oa[1], oa[2], oa[3]);
            *reinterpret_cast<uint4*>(row + kHalf + 8 * c) = make_uint4(ob[0], ob[1], ob[2], ob[3]);
        }
        __syncthreads();                          // read before the next tile rewrites them
    }
    if (!waited) grid_dependency_sync();
    if (rmax >= 65520.f) raise_status(status, kStatusRange);
}

// fp32 rows in and out, with the same tiles; thread item = (head, position,
// chunk c of 8): dims 4c..4c+3 and 32+4c..32+4c+3.
template <int TH>
__global__ void __launch_bounds__(256) rope_rows_f32_kernel(const float* __restrict__ src, float* __restrict__ dst,
                                                            int heads, int T_, RopeParams rp) {
    constexpr int kItems = TH / 4;                // per thread (256 threads)
    __shared__ __align__(16) float ctab[kRopePos][kHalf], stab[kRopePos][kHalf];
    const int tid = threadIdx.x;
    const int c = tid & 7, pr = (tid >> 3) & 7, hr0 = tid >> 6;
    const int tiles_p = (T_ + kRopePos - 1) / kRopePos;
    const int th = (int)(blockIdx.x / (unsigned)tiles_p), tp = (int)blockIdx.x - th * tiles_p;
    const int p0 = tp * kRopePos, h0 = th * TH, p = p0 + pr;
    rope_cs_exact(rp, tid & 31, p0 + (tid >> 5), ctab[tid >> 5][tid & 31], stab[tid >> 5][tid & 31]);
    grid_dependency_sync();
    float4 a[kItems], b[kItems];
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
        const int h = h0 + hr0 + 4 * u;
        if (h < heads && p < T_) {
            const float* row = src + ((size_t)h * T_ + p) * kHeadDim + 4 * c;
            a[u] = *reinterpret_cast<const float4*>(row);
            b[u] = *reinterpret_cast<const float4*>(row + kHalf);
        }
    }
    __syncthreads();                              // the tile's cos/sin are in shared memory
    const float4 cs = *reinterpret_cast<const float4*>(&ctab[pr][4 * c]);
    const float4 sn = *reinterpret_cast<const float4*>(&stab[pr][4 * c]);
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
        const int h = h0 + hr0 + 4 * u;
        if (h >= heads || p >= T_) continue;
        float* row = dst + ((size_t)h * T_ + p) * kHeadDim + 4 * c;
        const float4 x = a[u], y = b[u];
        *reinterpret_cast<float4*>(row) = make_float4(x.x * cs.x - y.x * sn.x, x.y * cs.y - y.y * sn.y,
                                                      x.z * cs.z - y.z * sn.z, x.w * cs.w - y.w * sn.w);
        *reinterpret_cast<float4*>(row + kHalf) = make_float4(y.x * cs.x + x.x * sn.x, y.y * cs.y + x.y * sn.y,
                                                              y.z * cs.z + x.z * sn.z, y.w * cs.w + x.w * sn.w);
    }
}

}  // namespace

cudaError_t launch_rope_rows(const void* src, void* dst, long long rows, int T, const RopeParams& rp,
                             bool bf16, cudaStream_t st, unsigned* status) {
    if (rows <= 0) return cudaSuccess;
    const int heads = (int)(rows / T);
    const long long tp = (T + kRopePos - 1) / kRopePos;
    if (bf16) {
        // one tile per block (the hardware hands the blocks to the SMs as
        // they free up, which balances the load better than a grid-stride
        // loop); tiles of 32 heads while they still give two blocks per SM,
        // else of 16 (B16 H8 T1024: 2.296 -> 2.281 ms per 16-layer step;
        // with two kv heads, 512 tiles of 16 heads beat 128 of 32), and never
        // of 32 where 16 rows are all there are (B2 H8 T16384: rotation 17.9
        // -> 16.2 us)
        static int sms = 0;
        if (sms == 0) {
            int dev = 0;
            if (cudaGetDevice(&dev) != cudaSuccess ||
                cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
                sms = 152;
        }
        const long long t32 = tp * ((heads + 31) / 32), t16 = tp * ((heads + 15) / 16);
        const __nv_bfloat16* s16 = reinterpret_cast<const __nv_bfloat16*>(src);
        __half* d16 = reinterpret_cast<__half*>(dst);
        if (t32 >= 2LL * sms && heads > 16)
            return launch_kernel(rope_rows_bf16_kernel<32>, dim3((unsigned)std::min(t32, 0x7fffffffLL)), dim3(256),
                                 0, st, s16, d16, heads, T, rp, status);
        return launch_kernel(rope_rows_bf16_kernel<16>, dim3((unsigned)std::min(t16, 0x7fffffffLL)), dim3(256), 0,
                             st, s16, d16, heads, T, rp, status);
    }
    // 16 heads a tile while that still gives two blocks per SM, else 4
    const float* s32 = reinterpret_cast<const float*>(src);
    float* d32 = reinterpret_cast<float*>(dst);
    const long long t16 = tp * ((heads + 15) / 16), t4 = tp * ((heads + 3) / 4);
    if (t16 >= 2 * 152)
        return launch_kernel(rope_rows_f32_kernel<16>, dim3((unsigned)t16), dim3(256), 0, st, s32, d32, heads, T, rp);
    return launch_kernel(rope_rows_f32_kernel<4>, dim3((unsigned)t4), dim3(256), 0, st, s32, d32, heads, T, rp);
}

}  // namespace fibattn

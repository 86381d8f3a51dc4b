// fibattn_internal.cuh -- shared definitions of the CUDA library (not part of
// the C ABI).  Depth-staggered scaled-Fibonacci sparse attention,
// arXiv 2606.28560, Section 2.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace fibattn {

constexpr int kHeadDim = 64;      // D; every kernel is specialised for it
constexpr int kHalf = kHeadDim / 2;
constexpr int kMaxRungs = 32;     // K limit of the ABI
constexpr int kMaxWindow = 1024;  // W limit of the ABI

// Per-rung data prepared on the host (Section 2: d_k = alpha * f_k, read by
// linear interpolation between the floor and floor-plus-one rows).
struct RungParams {
    int K;                    // number of rungs passed by the caller
    unsigned active;          // bit k: rung k can ever be attended (dedup, reach)
    int s0[kMaxRungs];        // floor(d_k)
    float w[kMaxRungs];       // d_k - floor(d_k): weight of the far row i-s0-1
    float d[kMaxRungs];       // d_k in fp32; the rung is masked for queries i < d_k
    float f[kMaxRungs];       // base value f_k (for dL/dalpha = sum_k f_k dL/dd_k)
};

// RoPE phase increments: the rotation angle of pair m at position p is
// 2*pi * frac(p * F[m] / 2^64), F[m] = round(2^64 * theta_m / (2*pi)),
// theta_m = base^(-2m/D).  The integer product wraps modulo one turn exactly,
// so the angle is reduced without any floating-point range reduction.
struct RopeParams {
    unsigned long long F[kHalf];
};

// Division by a divisor fixed at launch, for numerators below 2^31: the
// quotient is (umulhi(n, mul) + n) >> shift with shift = ceil(log2 d) and
// mul = floor(2^32 (2^shift - d) / d) + 1 (the round-up multiplier method).
struct FastDiv {
    unsigned d, mul, shift;
#ifdef __CUDACC__
    __host__ __device__
#endif
    static FastDiv make(unsigned d) {
        FastDiv f;
        f.d = d;
        f.shift = 0;
        while ((1ull << f.shift) < d) ++f.shift;
        f.mul = (unsigned)(((1ull << 32) * ((1ull << f.shift) - d)) / d + 1);
        return f;
    }
};
#ifdef __CUDACC__
__device__ __forceinline__ unsigned fdiv(unsigned n, const FastDiv& f) {
    return (__umulhi(n, f.mul) + n) >> f.shift;
}
#endif

struct Shape {
    int B, H, Hkv, T, W, G;   // G = H / Hkv
    float scale;              // score scale (1/sqrt(D) by default)
    FastDiv dH, dHkv, dG, dTiles;   // by H, Hkv, G and the tensor-core tiles per head
};

// Device status word (one per device, read and cleared by
// fibattn_check_status): kernels OR these bits into it.
constexpr unsigned kStatusWaitTimeout = 1u;   // a bounded wait on a staging copy ran out
constexpr unsigned kStatusRange = 2u;         // a rotated row overflowed its fp16 storage
__device__ __forceinline__ void raise_status(unsigned* st, unsigned bits) {
    if (st) atomicOr(st, bits);
}

struct FwdArgs {
    const void* q;            // [B,H,T,D]
    const void* kt;           // rotated keys [B,Hkv,T,D] (workspace)
    const void* k;            // raw keys (prologue input)
    const void* v;            // [B,Hkv,T,D]
    void* out;                // [B,H,T,D]
    float* lse;               // [B,H,T]
    // Optional residuals for the backward (tensor-core forward only; all
    // nullptr when not asked for): the rotated queries, the unnormalised
    // probability exp(s - max) of every slot (0 where not attended), the
    // far-minus-floor raw score of every rung row and 1 / (row sum) per query.
    void* res_qt;             // bf16 [B,H,T,D]
    float* res_P;             // slot-major [B,H,S,T], S = W + 1 + K
    float* res_sd;            // rung-major [B,H,K,T]
    float* res_il;            // [B,H,T]
    unsigned* status;         // device status word
    int S;
    Shape s;
    RungParams r;
    RopeParams rope;
};

struct BwdArgs {
    const void* q;            // [B,H,T,D]
    const void* k;            // [B,Hkv,T,D]
    const void* v;
    const float* lse;         // [B,H,T]
    const void* dout;         // [B,H,T,D]
    const void* out;          // forward output [B,H,T,D] or nullptr
    void* dq;                 // [B,H,T,D]
    void* dk;                 // [B,Hkv,T,D]
    void* dv;
    float* dtheta;            // device scalar or nullptr
    int want_dd;              // compute dL/dd_k (dtheta or dd requested)
    float* dd;                // device [K] or nullptr
    // workspace views
    void* qt;                 // rotated q [B,H,T,D] from the query pass (tensor-core: bf16; row-gather: fp16, or fp32 for fp32 I/O)
    void* kt;                 // rotated k [B,Hkv,T,D]
    float* Ps;                // slot-major [B,H,S,T]: p
    float* DSs;               //                       dS = p (dp - Delta)
    long long* rpart;         // per query-pass block dL/dd_k partials, 2^-32 fixed point [K][nblk_q]
    const float* res_il;      // forward residual 1 / (row sum) [B,H,T] (p = Ps[slot] * res_il)
    const float* res_sd;      // forward residual far-minus-floor rung scores [B,H,K,T], or nullptr;
                              // when the forward residuals are used, Ps and qt point into them
    int saved;                // tensor-core passes read p (Ps, unnormalised), sd and q~ (qt) from the forward residuals
    unsigned* status;         // device status word
    int nblk_q;               // query-pass blocks
    int S;                    // slots per query = W + 1 + K
    float alpha;
    Shape s;
    RungParams r;
    RopeParams rope;
};

// ---------------------------------------------------------------- RoPE ----

// cos/sin of the angle of pair m at position pos (see RopeParams).
__device__ __forceinline__ void rope_cs(const RopeParams& rp, int m, int pos, float& c, float& s) {
    unsigned long long ph = (unsigned long long)(unsigned)pos * rp.F[m];
    int hi = (int)(unsigned)(ph >> 32);              // signed turn fraction in [-1/2, 1/2)
    float ang = (float)hi * 1.4629180792671596e-09f; // 2*pi / 2^32
    __sincosf(ang, &s, &c);
}

// cos/sin of the same angle to fp32 rounding, for fp32 I/O (rope_cs is off by
// up to 4e-7, the largest error of that path: dL/dd_k 3.3e-7 off 64 bits with
// it, 2e-7 without).  The phase is reduced to an eighth of a turn either side
// of a multiple of a quarter turn as an integer, exactly; the Taylor
// polynomials of sine and cosine to the 9th and 10th power do the rest (the
// first terms left out are below 2e-9).
__device__ __forceinline__ void rope_cs_exact(const RopeParams& rp, int m, int pos, float& c, float& s) {
    const unsigned ph = (unsigned)(((unsigned long long)(unsigned)pos * rp.F[m]) >> 32);
    const unsigned quarter = (ph + 0x20000000u) >> 30;            // nearest multiple of a quarter turn
    const float x = (float)(int)(ph - (quarter << 30)) * 1.4629180792671596e-09f;   // 2 pi / 2^32
    const float y = x * x;
    const float sn = fmaf(x * y, fmaf(y, fmaf(y, fmaf(y, 1.f / 362880.f, -1.f / 5040.f), 1.f / 120.f), -1.f / 6.f), x);
    const float cn = fmaf(y, fmaf(y, fmaf(y, fmaf(y, fmaf(y, -1.f / 3628800.f, 1.f / 40320.f), -1.f / 720.f), 1.f / 24.f),
                                  -0.5f), 1.f);
    const bool swap = quarter & 1u;
    c = swap ? sn : cn;
    s = swap ? cn : sn;
    if (quarter == 1u || quarter == 2u) c = -c;
    if (quarter >= 2u) s = -s;
}

// Storage type of rotated rows: fp32 for fp32 I/O, fp16 for bf16 I/O (10
// mantissa bits against bf16's 7 keep the score error well inside the bf16
// tolerance).
template <typename T> struct RotOf { using type = float; };
template <> struct RotOf<__nv_bfloat16> { using type = __half; };

// ------------------------------------------------- rung-gradient reduction --

// dL/dd_k is the sum of the query blocks' partials.  Each block writes its
// partials as 64-bit fixed point (2^-32 units; threads k < K hold rung k's);
// one block of the key pass, which waits for the query pass to complete,
// adds them up -- integer addition is exact and order-free, so the result
// does not depend on scheduling -- and applies the chain rule
// dL/dalpha = sum_k f_k dL/dd_k, dL/dtheta = dL/dalpha (alpha - 0.5)(1.5 - alpha),
// alpha = 0.5 + sigmoid(theta).
__device__ __forceinline__ void write_rung_partials(const BwdArgs& a, float partial) {
    if ((int)threadIdx.x < a.r.K)
        a.rpart[(size_t)threadIdx.x * a.nblk_q + blockIdx.x] = __float2ll_rn(partial * 4294967296.0f);
}

// Called by every thread of one block of the key pass (blockDim a multiple of
// 32).  red: shared scratch of at least K doubles.  A warp sums whole rungs,
// kCols columns a lane in flight at a time.  Bound by load latency: one thread
// block adds K x (query-pass blocks) words while others may already be done.
// Rung after rung over all threads (a latency and a warp sum
// each) it was the end of the whole backward on small grids: key pass at B1
// H8 T1000 17.7 -> 12.5 us, at B4 22.6 -> 18.4 us, at B16 H8 Hkv2 T1024 (its
// blocks fit one wave) 47.3 -> 41.7 us; unchanged where several waves hide it.
__device__ __forceinline__ void convert_rung_sums(const BwdArgs& a, double* red) {
    constexpr int kCols = 8;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nw = blockDim.x >> 5;
    for (int k = warp; k < a.r.K; k += nw) {
        const long long* col = a.rpart + (size_t)k * a.nblk_q;
        long long v = 0;
        for (int b0 = lane; b0 < a.nblk_q; b0 += 32 * kCols) {
            long long x[kCols];
#pragma unroll
            for (int u = 0; u < kCols; ++u) x[u] = b0 + 32 * u < a.nblk_q ? __ldcg(col + b0 + 32 * u) : 0;
#pragma unroll
            for (int u = 0; u < kCols; ++u) v += x[u];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) {
            red[k] = (double)v * 2.3283064365386962890625e-10;
            if (a.dd) a.dd[k] = (float)red[k];
        }
    }
    __syncthreads();
    if (t == 0 && a.dtheta) {
        double da = 0.0;                          // (the terms cancel: an fp32 sum would add error of its own)
        for (int k = 0; k < a.r.K; ++k) da += (double)a.r.f[k] * red[k];
        *a.dtheta = (float)(da * ((double)a.alpha - 0.5) * (1.5 - (double)a.alpha));
    }
}

// ------------------------------------------- programmatic dependent launch --

// Every kernel starts with this, before its first global-memory access: it
// waits until the previous kernel in the stream has completed and its writes
// are visible (a no-op when the launch carries no programmatic dependency),
// then lets the next kernel be scheduled, so that its blocks can become
// resident and run up to their own wait while this grid's last blocks run.
__device__ __forceinline__ void grid_dependency_sync() {
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
// The two halves, for a kernel that knows which of its inputs the kernel
// before it (launched by the same library call) does not write: it lets the
// next launch be scheduled at once, reads those inputs, and waits only before
// touching anything the previous kernel may produce.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// Host: whether launches carry the programmatic-serialisation attribute
// (environment FIBATTN_PDL=0 turns it off).
bool pdl_enabled();

template <typename... KArgs, typename... Args>
cudaError_t launch_kernel(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                          Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// The same with dynamic shared memory, `most` being the largest that any call
// asks of this kernel.  The limit belongs to the function, and other host threads
// launch it with other sizes at the same time: it is always set to `most`, so no
// thread lowers it between another's set and launch.
template <typename... KArgs, typename... Args>
cudaError_t launch_kernel_dynamic(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, size_t most,
                                  cudaStream_t st, Args... args) {
    if (smem > most) return cudaErrorInvalidValue;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    return e != cudaSuccess ? e : launch_kernel(kern, grid, block, smem, st, args...);
}
constexpr size_t kBlockSmem = 227 * 1024;         // shared memory of a block, static and dynamic

// ----------------------------------------------------------- launchers ----

cudaError_t launch_rope_rows(const void* src, void* dst, long long rows, int T, const RopeParams& rp,
                             bool bf16, cudaStream_t st, unsigned* status);
// The row-gather passes (gather.cu).
cudaError_t launch_fwd_gather(const FwdArgs& a, bool bf16, cudaStream_t st);
cudaError_t launch_bwd_query_gather(const BwdArgs& a, bool bf16, cudaStream_t st);
cudaError_t launch_bwd_key_gather(const BwdArgs& a, bool bf16, cudaStream_t st);
int bwd_gather_blocks(const Shape& s);            // query-pass blocks: columns of BwdArgs::rpart

// Records a message for fibattn_last_error() and returns `code`.
int set_error(int code, const char* msg);

// Opt-in per-kernel timing: when enabled, each launch is bracketed by CUDA
// events recorded on the caller's stream (see fibattn_profile_* in the ABI).
struct ProfScope {
    ProfScope(const char* name, cudaStream_t st);
    ~ProfScope();
    const char* name_;
    cudaStream_t st_;
    cudaEvent_t start_;
    bool on_;
};

}  // namespace fibattn

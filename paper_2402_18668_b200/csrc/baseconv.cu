// baseconv_gate_forward / baseconv_gate_step: the gated short convolution at the core of the
// BaseConv layer (App. "Extended Architecture Details", paragraph "Convolution"):
//
//   out[b,i,c] = a[b,i,c] * SiLU( sum_{j<w, j<=i} h[j,c] * g[b,i-j,c] + b2[c] )
//
// a = u W1 + b1 and g = u W2 are the layer's two up-projections (plain matrix products, not
// part of this file); h is the depthwise causal filter of width w (the paper suggests 3), h[0]
// the tap on the current token.
//
// The op is one pass over a, g and out: 3 elements of traffic per output element and a dozen
// flops, so it is bound by HBM bandwidth.  A thread owns 8 consecutive channels (one 16-byte
// piece of a bf16 row, two of an fp32 row) and walks a run of up to 64 tokens with the last w-1 rows
// of g in registers, so g is read once (plus w-1 halo rows per run, which the neighbouring run
// has just brought into L2); a warp covers 256 consecutive channels of a row.  The loop is
// software-pipelined: the rows of the next four tokens are in flight (kept packed, as loaded)
// while the current four are converted, combined and stored.
#include "common.cuh"

namespace based {

namespace {
constexpr int kMaxRun = 64;     // tokens per thread run, at most
constexpr int kUnroll = 4;      // tokens whose loads are in flight together
constexpr int kThreadsBC = 128;

template <typename T> struct Row8;
template <> struct Row8<__nv_bfloat16> {
    struct Raw { uint4 u; };
    static __device__ __forceinline__ void load_raw(const __nv_bfloat16* p, Raw& r) {
        r.u = __ldcs(reinterpret_cast<const uint4*>(p));
    }
    static __device__ __forceinline__ void unpack(const Raw& r, float (&x)[8]) {
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&r.u);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 f = __bfloat1622float2(h[i]);
            x[2 * i] = f.x;
            x[2 * i + 1] = f.y;
        }
    }
    static __device__ __forceinline__ void store_raw(__nv_bfloat16* p, const Raw& r) { __stcs(reinterpret_cast<uint4*>(p), r.u); }
    static __device__ __forceinline__ void load(const __nv_bfloat16* p, float (&x)[8]) {
        const uint4 u = __ldcs(reinterpret_cast<const uint4*>(p));
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 f = __bfloat1622float2(h[i]);
            x[2 * i] = f.x;
            x[2 * i + 1] = f.y;
        }
    }
    static __device__ __forceinline__ void store(__nv_bfloat16* p, const float (&x)[8]) {
        uint4 u;
        __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&u);
#pragma unroll
        for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(x[2 * i], x[2 * i + 1]);
        __stcs(reinterpret_cast<uint4*>(p), u);
    }
};
template <> struct Row8<float> {
    struct Raw { float4 a, b; };
    static __device__ __forceinline__ void load_raw(const float* p, Raw& r) {
        r.a = __ldcs(reinterpret_cast<const float4*>(p));
        r.b = __ldcs(reinterpret_cast<const float4*>(p) + 1);
    }
    static __device__ __forceinline__ void unpack(const Raw& r, float (&x)[8]) {
        x[0] = r.a.x; x[1] = r.a.y; x[2] = r.a.z; x[3] = r.a.w; x[4] = r.b.x; x[5] = r.b.y; x[6] = r.b.z; x[7] = r.b.w;
    }
    static __device__ __forceinline__ void store_raw(float* p, const Raw& r) {
        __stcs(reinterpret_cast<float4*>(p), r.a);
        __stcs(reinterpret_cast<float4*>(p) + 1, r.b);
    }
    static __device__ __forceinline__ void load(const float* p, float (&x)[8]) {
        const float4 a = __ldcs(reinterpret_cast<const float4*>(p)), b = __ldcs(reinterpret_cast<const float4*>(p) + 1);
        x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
    }
    static __device__ __forceinline__ void store(float* p, const float (&x)[8]) {
        __stcs(reinterpret_cast<float4*>(p), make_float4(x[0], x[1], x[2], x[3]));
        __stcs(reinterpret_cast<float4*>(p) + 1, make_float4(x[4], x[5], x[6], x[7]));
    }
};

// 8 fp32 values of a filter row or the bias
__device__ __forceinline__ void load8(const float* p, float (&x)[8]) {
    const float4 lo = __ldg(reinterpret_cast<const float4*>(p)), hi = __ldg(reinterpret_cast<const float4*>(p) + 1);
    x[0] = lo.x; x[1] = lo.y; x[2] = lo.z; x[3] = lo.w; x[4] = hi.x; x[5] = hi.y; x[6] = hi.z; x[7] = hi.w;
}

// SiLU(x) = x * sigmoid(x); the fast exponential and division are exact enough for bf16 outputs,
// fp32 io takes the accurate ones
template <bool FAST>
__device__ __forceinline__ float silu(float x) {
    return FAST ? __fdividef(x, 1.0f + __expf(-x)) : x / (1.0f + expf(-x));
}
}  // namespace

template <typename T, int W>
__global__ void __launch_bounds__(kThreadsBC) baseconv_gate_kernel(const T* __restrict__ a, const T* __restrict__ g,
                                                                   const float* __restrict__ h,
                                                                   const float* __restrict__ b2, T* __restrict__ out,
                                                                   int N, int C, int run) {
    constexpr bool FAST = sizeof(T) == 2;
    const int c0 = (blockIdx.x * kThreadsBC + threadIdx.x) * 8;
    if (c0 >= C) return;
    const int i0 = blockIdx.y * run;
    const int i1 = min(N, i0 + run);
    const size_t base = (size_t)blockIdx.z * N * C + c0;

    // prev[j] = g of the token j+1 steps back (zero before the sequence start)
    float prev[W > 1 ? W - 1 : 1][8];
#pragma unroll
    for (int j = 0; j < W - 1; ++j) {
        const int i = i0 - 1 - j;
        if (i >= 0) Row8<T>::load(g + base + (size_t)i * C, prev[j]);
        else {
#pragma unroll
            for (int e = 0; e < 8; ++e) prev[j][e] = 0.f;
        }
    }

    // software pipeline: the loads of the next kUnroll tokens are in flight while these are used
    typename Row8<T>::Raw gr[kUnroll], ar[kUnroll], gn[kUnroll], an[kUnroll];
    auto fetch = [&](int i, typename Row8<T>::Raw (&gq)[kUnroll], typename Row8<T>::Raw (&aq)[kUnroll]) {
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            if (i + u < i1) {
                Row8<T>::load_raw(g + base + (size_t)(i + u) * C, gq[u]);
                Row8<T>::load_raw(a + base + (size_t)(i + u) * C, aq[u]);
            }
        }
    };
    fetch(i0, gr, ar);
    float taps[W][8], bias[8];
#pragma unroll
    for (int j = 0; j < W; ++j) load8(h + (size_t)j * C + c0, taps[j]);
    load8(b2 + c0, bias);
    for (int i = i0; i < i1; i += kUnroll) {
        fetch(i + kUnroll, gn, an);
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            if (i + u < i1) {
                float gx[8], ax[8], y[8];
                Row8<T>::unpack(gr[u], gx);
                Row8<T>::unpack(ar[u], ax);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    float acc = fmaf(taps[0][e], gx[e], bias[e]);
#pragma unroll
                    for (int j = 1; j < W; ++j) acc = fmaf(taps[j][e], prev[j - 1][e], acc);
                    y[e] = ax[e] * silu<FAST>(acc);
                }
                Row8<T>::store(out + base + (size_t)(i + u) * C, y);
#pragma unroll
                for (int j = W - 2; j >= 1; --j)
#pragma unroll
                    for (int e = 0; e < 8; ++e) prev[j][e] = prev[j - 1][e];
                if (W > 1) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) prev[0][e] = gx[e];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            gr[u] = gn[u];
            ar[u] = an[u];
        }
    }
}

// One token: state [B, W-1, C], row j = g of the token j+1 steps back; shifted in place.  A thread owns 8 channels of ROWS
// sequences: their taps and bias are read once (as 128-bit words) and the rows' loads are all in flight together.
// HBM bound, latency-limited at this size: B128 C8192 width 3 moves 14.7 MB (2.2 us of copy) in 3.4 us; one sequence per
// thread with scalar tap loads took 7.7 (ncu).
template <typename T, int W, int ROWS>
__global__ void __launch_bounds__(kThreadsBC) baseconv_step_kernel(const T* __restrict__ a, const T* __restrict__ g,
                                                                   const float* __restrict__ h,
                                                                   const float* __restrict__ b2, T* __restrict__ state,
                                                                   T* __restrict__ out, int B, int C) {
    enter_dependent();
    constexpr bool FAST = sizeof(T) == 2;
    const int c0 = (blockIdx.x * kThreadsBC + threadIdx.x) * 8;
    if (c0 >= C) return;
    const int b0 = blockIdx.y * ROWS;
    typename Row8<T>::Raw gr[ROWS], ar[ROWS], pr[ROWS][W > 1 ? W - 1 : 1];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const size_t b = b0 + r;
        if (b0 + r < B) {
            Row8<T>::load_raw(g + b * C + c0, gr[r]);
            Row8<T>::load_raw(a + b * C + c0, ar[r]);
#pragma unroll
            for (int j = 0; j < W - 1; ++j) Row8<T>::load_raw(state + (b * (W - 1) + j) * C + c0, pr[r][j]);
        }
    }
    float taps[W][8], bias[8];
#pragma unroll
    for (int j = 0; j < W; ++j) load8(h + (size_t)j * C + c0, taps[j]);
    load8(b2 + c0, bias);
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const size_t b = b0 + r;
        if (b0 + r >= B) break;
        float gx[8], x[8], acc[8];
        Row8<T>::unpack(gr[r], gx);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = fmaf(taps[0][e], gx[e], bias[e]);
#pragma unroll
        for (int j = 1; j < W; ++j) {
            Row8<T>::unpack(pr[r][j - 1], x);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] = fmaf(taps[j][e], x[e], acc[e]);
        }
        Row8<T>::unpack(ar[r], x);
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] *= silu<FAST>(acc[e]);
        Row8<T>::store(out + b * C + c0, x);
        T* st = state + b * (size_t)(W - 1) * C + c0;
#pragma unroll
        for (int j = W - 2; j >= 1; --j) Row8<T>::store_raw(st + (size_t)j * C, pr[r][j - 1]);
        if (W > 1) Row8<T>::store_raw(st, gr[r]);
    }
}

template <typename T, int W>
static void launch_w(const void* a, const void* g, const float* h, const float* b2, void* state, void* out, int B,
                     int N, int C, bool step, cudaStream_t stream) {
    const int gx = (C / 8 + kThreadsBC - 1) / kThreadsBC;
    static std::atomic<bool> split[3][64];
    prefer_l1(baseconv_step_kernel<T, W, 4>, 0, split[0]);       // (a preference only: the launch reports what fails)
    prefer_l1(baseconv_step_kernel<T, W, 1>, 0, split[1]);
    prefer_l1(baseconv_gate_kernel<T, W>, 0, split[2]);
    // a step is a dependent launch: its blocks come in while the kernel ahead drains (behind the other mixers' steps at batch
    // 128 1.0 us less a token; back to back with itself 0.5 more); four sequences per thread once that still gives every SM a block
    if (step && gx * ((B + 3) / 4) >= kSMs)
        launch_ex(baseconv_step_kernel<T, W, 4>, dim3(gx, (B + 3) / 4), dim3(kThreadsBC), 0, 1, true, stream,
            static_cast<const T*>(a), static_cast<const T*>(g), h, b2, static_cast<T*>(state), static_cast<T*>(out), B, C);
    else if (step)
        launch_ex(baseconv_step_kernel<T, W, 1>, dim3(gx, B), dim3(kThreadsBC), 0, 1, true, stream,
            static_cast<const T*>(a), static_cast<const T*>(g), h, b2, static_cast<T*>(state), static_cast<T*>(out), B, C);
    else {
        // runs of 64 tokens (a halo of width - 1 rows each) while the last wave of blocks is a small part of the grid, 32
        // below, shorter ones until the grid has a block or two for every SM (us with runs of 64 / 32 / 16 / 8 / 4 tokens:
        // B3 N128 C5208 12.8 / 7.4 / 5.0 / 4.4 / 5.7, B2 N1024 C2048 12.9 / 7.7 / 6.4 / 6.9 / 7.1, B4 N1024 C8192 width 4
        // 41 / 37 / 38 / 42 / 51; B8 N4096 C8192 267 / 264 / 270 / 295 / 350, but 276.5 / 277.8 on alternating inputs)
        auto blocks = [&](int run) { return (long long)gx * ((N + run - 1) / run) * B; };
        int run = kMaxRun;
        if (blocks(run) < 2048) run /= 2;
        while (run > 4 && blocks(run) < 240) run /= 2;
        baseconv_gate_kernel<T, W><<<dim3(gx, (N + run - 1) / run, B), kThreadsBC, 0, stream>>>(
            static_cast<const T*>(a), static_cast<const T*>(g), h, b2, static_cast<T*>(out), N, C, run);
    }
}

template <typename T>
static void launch_t(const void* a, const void* g, const float* h, const float* b2, void* state, void* out, int B,
                     int N, int C, int width, bool step, cudaStream_t stream) {
    switch (width) {
        case 1: launch_w<T, 1>(a, g, h, b2, state, out, B, N, C, step, stream); break;
        case 2: launch_w<T, 2>(a, g, h, b2, state, out, B, N, C, step, stream); break;
        case 3: launch_w<T, 3>(a, g, h, b2, state, out, B, N, C, step, stream); break;
        default: launch_w<T, 4>(a, g, h, b2, state, out, B, N, C, step, stream); break;
    }
}

based_status launch_baseconv(const void* a, const void* g, const float* h, const float* b2, void* state, void* out,
                             int B, int N, int C, int width, bool step, based_dtype io, cudaStream_t stream) {
    if (io == BASED_F32) launch_t<float>(a, g, h, b2, state, out, B, N, C, width, step, stream);
    else launch_t<__nv_bfloat16>(a, g, h, b2, state, out, B, N, C, width, step, stream);
    note_launch();
    return check_launch(step ? "baseconv_step_kernel" : "baseconv_gate_kernel");
}

}  // namespace based

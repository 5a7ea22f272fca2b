// baseconv_gate_forward / baseconv_gate_step: the gated short convolution at the core of the
// BaseConv layer (App. "Extended Architecture Details", paragraph "Convolution"):
//
//   out[b,i,c] = a[b,i,c] * SiLU( sum_{j<w, j<=i} h[j,c] * g[b,i-j,c] + b2[c] )
//
// a = u W1 + b1 and g = u W2 are the layer's two up-projections (plain matrix products, not
// part of this file); h is the depthwise causal filter of width w (the paper suggests 3), h[0]
// the tap on the current token.
//
// The op is one pass over a, g and out: 3 elements of traffic per output element and a dozen flops, so it is bound by HBM
// bandwidth.  A thread owns 8 consecutive channels (one 16-byte piece of a bf16 row, two of an fp32 row) of 2, 4 or 8
// consecutive tokens (baseconv_block_kernel): their rows of a and g, and the w - 1 rows of g before them, which a neighbouring
// block brings into L2 at the same time, are all requested at once, and the blocks sweep the arrays in the order they lie in
// memory.  That is what HBM rewards: with runs of 64 tokens a thread, the rows of g carried along and the next four tokens' in
// flight, 2368 blocks were at as many places 1 MB apart.  B8 N4096 C8192 w 3 bf16 261 -> 228 us = 7.06 TB/s (a product a * g by torch
// over the same arrays: 230), B8 N1024 C8192 72 -> 60, fp32 B8 N2048 C4096 152 -> 123.
#include <type_traits>

#include "common.cuh"

namespace based {

namespace {
constexpr int kThreadsBC = 128, kThreadsBlock = 64;

template <typename T> struct Row8;
template <> struct Row8<__nv_bfloat16> {
    struct Raw { uint4 u; };
    static __device__ __forceinline__ void load_raw(const __nv_bfloat16* p, Raw& r) {
        r.u = __ldcs(reinterpret_cast<const uint4*>(p));
    }
    // (rows that another block reads too)
    static __device__ __forceinline__ void load_shared(const __nv_bfloat16* p, Raw& r) { r.u = __ldg(reinterpret_cast<const uint4*>(p)); }
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
    static __device__ __forceinline__ void load_shared(const float* p, Raw& r) {
        r.a = __ldg(reinterpret_cast<const float4*>(p));
        r.b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    }
    static __device__ __forceinline__ void unpack(const Raw& r, float (&x)[8]) {
        x[0] = r.a.x; x[1] = r.a.y; x[2] = r.a.z; x[3] = r.a.w; x[4] = r.b.x; x[5] = r.b.y; x[6] = r.b.z; x[7] = r.b.w;
    }
    static __device__ __forceinline__ void store_raw(float* p, const Raw& r) {
        __stcs(reinterpret_cast<float4*>(p), r.a);
        __stcs(reinterpret_cast<float4*>(p) + 1, r.b);
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

// two channels at a time: fp32 pairs, two multiply-adds per instruction
__device__ __forceinline__ uint32_t& word(uint4& v, int i) { return reinterpret_cast<uint32_t*>(&v)[i]; }
__device__ __forceinline__ uint32_t word(const uint4& v, int i) { return reinterpret_cast<const uint32_t*>(&v)[i]; }
__device__ __forceinline__ uint64_t pair_of(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ uint64_t pair_of_bf16(uint32_t w) { return pair_of(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }
__device__ __forceinline__ uint64_t fma_pairs(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t mul_pairs(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ void load_pairs(const float* p, uint64_t (&x)[4]) {
    const ulonglong2 lo = __ldg(reinterpret_cast<const ulonglong2*>(p)), hi = __ldg(reinterpret_cast<const ulonglong2*>(p) + 1);
    x[0] = lo.x; x[1] = lo.y; x[2] = hi.x; x[3] = hi.y;
}
// a SiLU(x) of two channels, rounded to bf16: x / (1 + 2^(-x log2 e)) with the fast exponential and reciprocal
__device__ __forceinline__ uint32_t gated_pair(uint64_t x, uint64_t a) {
    float s0, s1;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(s0), "=f"(s1) : "l"(mul_pairs(x, pair_of(-1.4426950408889634f, -1.4426950408889634f))));
    asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(s0));
    asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(s1));
    s0 += 1.0f;
    s1 += 1.0f;
    asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(s0));
    asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(s1));
    float y0, y1;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(y0), "=f"(y1) : "l"(mul_pairs(a, mul_pairs(x, pair_of(s0, s1)))));
    const __nv_bfloat162 r = __floats2bfloat162_rn(y0, y1);
    return *reinterpret_cast<const uint32_t*>(&r);
}

// SiLU(x) = x * sigmoid(x); the fast exponential and division are exact enough for bf16 outputs,
// fp32 io takes the accurate ones
template <bool FAST>
__device__ __forceinline__ float silu(float x) {
    return FAST ? __fdividef(x, 1.0f + __expf(-x)) : x / (1.0f + expf(-x));
}
}  // namespace

// Blocks per SM: what is in flight on an SM is TOK rows times its threads, so each instance is held to the registers that let one
// more block in where it is a few above (bf16 w 3: 8 tokens 130 -> 128, seven blocks -> eight, B8 N4096 C8192 241 -> 228 us; 4
// tokens 102 -> 96, B1 37.6 -> 32.2).
__host__ __device__ constexpr int blocks_per_sm(int elem, int W, int tok) {
    if (elem == 4) return tok == 4 ? (W == 1 ? 10 : W < 4 ? 8 : 6) : W == 1 ? 16 : W == 2 ? 11 : W == 3 ? 10 : 8;
    if (tok == 8) return W == 1 ? 10 : W < 4 ? 8 : 6;
    if (tok == 4) return W == 1 ? 14 : W == 2 ? 12 : W == 3 ? 10 : 8;
    return W == 1 ? 18 : W == 2 ? 16 : W == 3 ? 12 : 10;
}
// TOK tokens of 8 channels per thread; grid: blocks of 512 channels, of TOK tokens, sequences.  FLAT: the first two in one dimension, for
// more blocks of tokens than a grid has rows (for all calls, its division cost B8 N4096 C8192 228 -> 239 us).
template <typename T, int W, int TOK, bool FLAT>
__global__ void __launch_bounds__(kThreadsBlock, blocks_per_sm(sizeof(T), W, TOK)) baseconv_block_kernel(const T* __restrict__ a, const T* __restrict__ g,
                                                                       const float* __restrict__ h, const float* __restrict__ b2,
                                                                       T* __restrict__ out, int N, int C, int gb) {
    enter_dependent();
    constexpr bool FAST = sizeof(T) == 2;
    const int row = FLAT ? blockIdx.x / gb : blockIdx.y, col = FLAT ? blockIdx.x - row * gb : blockIdx.x;
    const int c0 = (col * kThreadsBlock + threadIdx.x) * 8;
    if (c0 >= C) return;
    const size_t base = (size_t)(FLAT ? blockIdx.y : blockIdx.z) * N * C + c0;
    const int i0 = row * TOK;
    typename Row8<T>::Raw gr[TOK + W - 1], ar[TOK];
#pragma unroll
    for (int u = 0; u < W - 1; ++u) {
        const int i = i0 + u - (W - 1);
        if (i >= 0) Row8<T>::load_shared(g + base + (size_t)i * C, gr[u]);
        else gr[u] = typename Row8<T>::Raw{};                        // before the sequence
    }
#pragma unroll
    for (int u = 0; u < TOK; ++u)
        if (i0 + u < N) Row8<T>::load_shared(g + base + (size_t)(i0 + u) * C, gr[u + W - 1]);
#pragma unroll
    for (int u = 0; u < TOK; ++u)
        if (i0 + u < N) Row8<T>::load_raw(a + base + (size_t)(i0 + u) * C, ar[u]);
    if constexpr (FAST) {
        uint64_t taps[W][4], bias[4];
#pragma unroll
        for (int j = 0; j < W; ++j) load_pairs(h + (size_t)j * C + c0, taps[j]);
        load_pairs(b2 + c0, bias);
#pragma unroll
        for (int u = 0; u < TOK; ++u) {
            if (i0 + u >= N) break;
            uint4 y;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uint64_t acc = bias[e];
#pragma unroll
                for (int j = 0; j < W; ++j) acc = fma_pairs(taps[j][e], pair_of_bf16(word(gr[u + W - 1 - j].u, e)), acc);
                word(y, e) = gated_pair(acc, pair_of_bf16(word(ar[u].u, e)));
            }
            __stcs(reinterpret_cast<uint4*>(out + base + (size_t)(i0 + u) * C), y);
        }
    } else {
        float taps[W][8], bias[8];
#pragma unroll
        for (int j = 0; j < W; ++j) load8(h + (size_t)j * C + c0, taps[j]);
        load8(b2 + c0, bias);
#pragma unroll
        for (int u = 0; u < TOK; ++u) {
            if (i0 + u >= N) break;
            float acc[8], x[8];
            Row8<T>::unpack(gr[u + W - 1], x);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] = fmaf(taps[0][e], x[e], bias[e]);
#pragma unroll
            for (int j = 1; j < W; ++j) {
                Row8<T>::unpack(gr[u + W - 1 - j], x);
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[e] = fmaf(taps[j][e], x[e], acc[e]);
            }
            Row8<T>::unpack(ar[u], x);
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] *= silu<FAST>(acc[e]);
            Row8<T>::store(out + base + (size_t)(i0 + u) * C, x);
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
    static std::atomic<bool> split[2][64];
    prefer_l1(baseconv_step_kernel<T, W, 4>, 0, split[0]);       // (a preference only: the launch reports what fails)
    prefer_l1(baseconv_step_kernel<T, W, 1>, 0, split[1]);
    // a step is a dependent launch: its blocks come in while the kernel ahead drains (behind the other mixers' steps at batch
    // 128 1.0 us less a token; back to back with itself 0.5 more); four sequences per thread once that still gives every SM a block
    if (step && gx * ((B + 3) / 4) >= kSMs)
        launch_ex(baseconv_step_kernel<T, W, 4>, dim3(gx, (B + 3) / 4), dim3(kThreadsBC), 0, 1, true, stream,
            static_cast<const T*>(a), static_cast<const T*>(g), h, b2, static_cast<T*>(state), static_cast<T*>(out), B, C);
    else if (step)
        launch_ex(baseconv_step_kernel<T, W, 1>, dim3(gx, B), dim3(kThreadsBC), 0, 1, true, stream,
            static_cast<const T*>(a), static_cast<const T*>(g), h, b2, static_cast<T*>(state), static_cast<T*>(out), B, C);
    else {
        // Tokens per thread, us with runs of 64 before / 8 / 4 / 2 (bf16): w 3 B8 N4096 C8192 261 / 228 / 233 / 290, B8 N1024 C8192 72 /
        // 60 / 61 / 75, B4 N3000 C3200 52 / 37 / 38 / 47, B1 N512 C8192 9.4 / 7.7 / 6.8 / 7.7, B3 N200 C1000 5.7 / 4.9 / 5.1 / 5.0; w 4 B8 N4096
        // C8192 265 / 246 / 262; fp32 w 3 B8 N2048 C4096 152 / - / 123 / 133, B8 N64 C4096 10.6 / - / 8.2 / 7.7.
        const int gb = (C / 8 + kThreadsBlock - 1) / kThreadsBlock;
        auto blocks = [&](int tok) { return (long long)gb * ((N + tok - 1) / tok) * B; };
        auto block = [&](auto tok_tag, auto flat_tag) {
            constexpr int TOK = decltype(tok_tag)::value;
            constexpr bool FLAT = decltype(flat_tag)::value;
            const unsigned rows = (N + TOK - 1) / TOK;
            // (behind a kernel that left the SM to shared memory, us without / with the preference, B8 N1024 C8192 59 alone: behind the
            // sliding window 102 / 62, a prefill 89 / 59; B8 N4096 227 alone: 385 / 230, 343 / 226; B1 N512 4.8 alone: 8.3 / 5.4, 6.9 / 5.5)
            static std::atomic<bool> split_block[64];
            prefer_l1(baseconv_block_kernel<T, W, TOK, FLAT>, 0, split_block);
            launch_ex(baseconv_block_kernel<T, W, TOK, FLAT>, FLAT ? dim3(gb * rows, B) : dim3(gb, rows, B), dim3(kThreadsBlock), 0, 1, true, stream,
                      static_cast<const T*>(a), static_cast<const T*>(g), h, b2, static_cast<T*>(out), N, C, gb);
        };
        using Four = std::integral_constant<int, 4>;
        using Most = std::integral_constant<int, sizeof(T) == 2 ? 8 : 4>;
        if (N > 2 * 65535) block(Four{}, std::true_type{});
        else if (sizeof(T) == 2 && blocks(8) >= 12288) block(Most{}, std::false_type{});
        else if (blocks(4) >= 2048) block(Four{}, std::false_type{});
        else block(std::integral_constant<int, 2>{}, std::false_type{});
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
    return check_launch(step ? "baseconv_step_kernel" : "baseconv_block_kernel");
}

}  // namespace based

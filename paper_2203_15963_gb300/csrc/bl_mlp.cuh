// Learned thermal-synchrotron coefficient model: a 3 -> 64 -> 64 -> 7 SiLU perceptron whose
// seven outputs replace the transcendental parts of the fits of Sec. 2.5 (Bessel factors of
// the Maxwell-Juettner normalisation, the emissivity shape polynomials, the Faraday shapes);
// the closed-form prefactors stay exact. Weights are BF16 in shared memory, products run on
// the tensor cores (tcgen05, FP32 accumulation in tensor memory), one 128-sample tile per
// CTA with one sample per thread.
//
// Model (all float):
//   inputs  log10 x in [-3, 6] (x = nu / nu_c, nu_c = 1.5 nu_B sin(theta) Theta^2),
//           log10 Theta_e in [-1, 2], |cos theta_B| in [0, 1], each mapped to [-1, 1], and a
//           constant 1 that carries the first layer's bias;
//   outputs o = offset + scale * y + A f, y = W3 silu(W2 silu(W1 [f, 1]) + b2) + b3, with
//           o1..o3 = ln of the I, Q, V shape prefactors (the exp(-1.8899 x^1/3) factor kept
//           exact), o4, o5 = f_m, g_m (Faraday conversion and rotation shapes),
//           o6 = ln(e^z K_2(z)), o7 = ln(K_0(z) / K_2(z)), z = 1 / Theta_e.
// Parameter vector (float, kParams values): W1 [64][4], W2 [64][64], b2 [64], W3 [7][64],
// b3 [7], offset [7], scale [7], A [7][3]. Offset, A and scale are fixed before training (the
// least-squares affine fit of the targets and its residual's standard deviation), so the
// network learns only the non-linear remainder.
#pragma once
#include "bl_internal.cuh"
#include "bl_math.cuh"
#include "bl_tc.cuh"

namespace bl {
namespace mlp {

constexpr int kHidden = 64, kOut = 7;
constexpr int kOffW1 = 0, kOffW2 = 256, kOffB2 = 4352, kOffW3 = 4416, kOffB3 = 4864,
              kOffMean = 4871, kOffScale = 4878, kOffA = 4885, kParams = 4906;
constexpr float kLxLo = -3.0f, kLxHi = 6.0f, kLtLo = -1.0f, kLtHi = 2.0f;
constexpr long long kWaitCycles = 1ll << 31;   // ~1 s at 2 GHz

__device__ __forceinline__ float silu(float z) { return __fdividef(z, 1.0f + __expf(-z)); }
// z sigma(z) = z/2 (1 + tanh(z/2)) with the hardware tanh (relative error about 2^-11, below
// the bf16 rounding of the stored activation, 2^-9): one special-function operation instead
// of two. Inference in the trace only; training keeps silu above.
__device__ __forceinline__ float silu_tanh(float z) {
    const float hz = 0.5f * z;
    float t;
    asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(hz));
    return fmaf(hz, t, hz);
}
__device__ __forceinline__ float silu_grad(float z) {
    const float s = __fdividef(1.0f, 1.0f + __expf(-z));
    return s * (1.0f + z * (1.0f - s));
}

// ---------------------------------------------------------------------------------------
// Model inputs of one plasma sample and the reconstruction of the eight coefficients
// ---------------------------------------------------------------------------------------
struct ModelIn {
    float f[3];     // network inputs in [-1, 1]
    bool ok;        // inside the trained domain
};

__device__ __forceinline__ ModelIn model_inputs(float th, float bg, float nu, float cth) {
    ModelIn m;
    const float sth = sqrtf(fmaxf(1.0f - cth * cth, 0.0f));
    const float nub = (float)(kE / (2.0 * kPi * kMe * kC)) * bg;
    const float nuc = 1.5f * nub * sth * th * th;
    const float lx = log10f(nu / nuc);
    const float lt = log10f(th);
    m.ok = th > 0.0f && bg > 0.0f && nuc > 0.0f && lx >= kLxLo && lx <= kLxHi && lt >= kLtLo &&
           lt <= kLtHi;
    m.f[0] = m.ok ? 2.0f * (lx - kLxLo) / (kLxHi - kLxLo) - 1.0f : 0.0f;
    m.f[1] = m.ok ? 2.0f * (lt - kLtLo) / (kLtHi - kLtLo) - 1.0f : 0.0f;
    m.f[2] = 2.0f * fabsf(cth) - 1.0f;
    return m;
}

// j_{I,Q,V}, alpha_{I,Q,V}, rho_{Q,V} from the learned quantities o[7] and the exact
// prefactors (same formulae as synchrotron_coefficients with its transcendental parts
// replaced). Requires ne, th, bg > 0 and sin(theta_B) > 0 (guaranteed by model_inputs).
__device__ __forceinline__ void coefficients_from(const float o[7], float ne, float th, float bg,
                                                  float nu, float cth, float out[8]) {
    const float sth2 = fmaxf(1.0f - cth * cth, 0.0f);
    const float sth = sqrtf(sth2);
    const float nub = (float)(kE / (2.0 * kPi * kMe * kC)) * bg;
    const float z = 1.0f / th;
    const float x = nu / (1.5f * nub * sth * th * th);
    const float lex = -1.8899f * cbrtf(x) + z - o[5];
    const float pre = ne * (float)(kE * kE / (1.7320508075688772 * kC)) * nu;
    out[0] = pre * expf(o[0] + lex);
    out[1] = pre * expf(o[1] + lex);
    out[2] = pre * (4.0f / (3.0f * th)) * (cth / sth) * expf(o[2] + lex);
    const float hkt = (float)(kH / (kMe * kC * kC)) * nu / th;
    const float cnu = (float)kC / nu;
    const float ibnu = expm1f(hkt) * (cnu * cnu) * ((float)(0.5 / kH) / nu);
    out[3] = out[0] * ibnu;
    out[4] = out[1] * ibnu;
    out[5] = out[2] * ibnu;
    const float k0k2 = expf(o[6]);
    const float k1k2 = (1.0f - k0k2) * z * 0.5f;
    const float base = ne * (float)(kE * kE / (kMe * kC));
    out[6] = base * nub * nub * sth2 / (nu * nu * nu) * o[3] * (k1k2 + 6.0f * th);
    out[7] = 2.0f * base * nub * cth / (nu * nu) * k0k2 * o[4];
}

// The seven learned quantities from the exact fits, in FP64 (training targets).
__device__ __forceinline__ void exact_targets(double lx, double lt, double o[7]) {
    const double x = pow(10.0, lx);
    const double u = 1.0 / cbrt(x);
    const double X = sqrt(1.4142135623730951e3 / (1.5 * x));
    o[0] = log(2.5651 * (1.0 + 1.92 * u + 0.9977 * u * u));
    o[1] = log(2.5651 * (1.0 + 0.932 * u + 0.4998 * u * u));
    o[2] = log(1.8138 / x + 3.423 * u * u + 0.02955 / sqrt(x) + 2.0377 * u);
    o[3] = 2.011 * exp(-pow(X, 1.035) / 4.7) - cos(0.5 * X) * exp(-pow(X, 1.2) / 2.73) -
           0.011 * exp(-X / 47.2);
    o[4] = 1.0 - 0.11 * log1p(0.035 * X);
    double k0, k1, k2;
    bessel_k012_scaled<double>(pow(10.0, -lt), k0, k1, k2);
    o[5] = log(k2);
    o[6] = log(k0 / k2);
}

// SplitMix64 (Steele, Lea & Flood 2014): the i-th output of the generator seeded with seed.
__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t i) {
    uint64_t z = seed + (i + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__host__ __device__ __forceinline__ double uniform01(uint64_t seed, uint64_t i) {
    return (double)(splitmix64(seed, i) >> 11) * 0x1.0p-53;
}

// ---------------------------------------------------------------------------------------
// Inference: one 128-sample tile per call, all 128 threads of the CTA take part
// ---------------------------------------------------------------------------------------
struct __align__(128) FwdSmem {
    unsigned char w1[64 * 16 * 2];   // [64][16]: W1 columns 0-2, bias in column 3
    unsigned char w2[64 * 64 * 2];   // [64][64]
    unsigned char w3[16 * 64 * 2];   // [16][64], rows 7-15 zero
    unsigned char x[128 * 16 * 2];   // [128][16]: inputs, 1, zeros
    unsigned char h[128 * 64 * 2];   // [128][64]: hidden activations
    float b2[64], b3[8], mean[8], scale[8], A[24];
    uint64_t bar;
    uint32_t tmem;
};
constexpr uint32_t kFwdCols = 64;

// Stage the weights and set up tensor memory and the barrier (every thread calls this).
__device__ __forceinline__ void fwd_init(FwdSmem& S, const float* __restrict__ P) {
    const int t = threadIdx.x, nt = blockDim.x;
    for (int i = t; i < 64 * 16; i += nt) {
        const int j = i >> 4, k = i & 15;
        tc::st_bf16(S.w1, j, k, 16, k < 4 ? P[kOffW1 + 4 * j + k] : 0.0f);
    }
    for (int i = t; i < 64 * 64; i += nt) tc::st_bf16(S.w2, i >> 6, i & 63, 64, P[kOffW2 + i]);
    for (int i = t; i < 16 * 64; i += nt) {
        const int o = i >> 6, j = i & 63;
        tc::st_bf16(S.w3, o, j, 64, o < kOut ? P[kOffW3 + 64 * o + j] : 0.0f);
    }
    for (int i = t; i < 128 * 16; i += nt) {
        const int r = i >> 4, k = i & 15;
        tc::st_bf16(S.x, r, k, 16, k == 3 ? 1.0f : 0.0f);
    }
    for (int i = t; i < 64; i += nt) S.b2[i] = P[kOffB2 + i];
    for (int i = t; i < 8; i += nt) {
        S.b3[i] = i < kOut ? P[kOffB3 + i] : 0.0f;
        S.mean[i] = i < kOut ? P[kOffMean + i] : 0.0f;
        S.scale[i] = i < kOut ? P[kOffScale + i] : 0.0f;
    }
    for (int i = t; i < 24; i += nt) S.A[i] = i < 3 * kOut ? P[kOffA + i] : 0.0f;
    if (t < 32) tc::tmem_alloc(&S.tmem, kFwdCols);
    if (t == 0) tc::mbar_init(&S.bar, 1);
    tc::fence_smem_to_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
}

// Wait for the MMA group committed in phase `phase`, the same outcome on every thread.
__device__ __forceinline__ bool cta_wait(FwdSmem& S, uint32_t& phase) {
    const bool ok = tc::mbar_wait(&S.bar, phase, kWaitCycles);
    phase ^= 1u;
    const bool all = __syncthreads_and(ok) != 0;
    tc::fence_after_sync();
    return all;
}

// hidden layer epilogue: 64 accumulator columns of this thread's row (+ bias), SiLU, BF16
// row of the next A operand
template <bool kTanh>
__device__ __forceinline__ void hidden_epilogue(FwdSmem& S, const float* bias) {
    auto act = [](float z) { return kTanh ? silu_tanh(z) : silu(z); };
    const int t = threadIdx.x;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float v[16];
        tc::tmem_ld16(tc::tmem_lane_addr(S.tmem, 16 * c), v);
        // 8 consecutive columns of a row are one 16-byte row of a core matrix: one vector store
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            uint32_t w[4];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int j = 8 * g + 2 * p;
                w[p] = tc::pack_bf16x2(act(v[j] + (bias ? bias[16 * c + j] : 0.0f)),
                                       act(v[j + 1] + (bias ? bias[16 * c + j + 1] : 0.0f)));
            }
            *reinterpret_cast<uint4*>(S.h + tc::kmajor(t, 16 * c + 8 * g, 64)) =
                make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

__device__ __forceinline__ void issue_barrier_then(FwdSmem& S) {
    tc::fence_smem_to_async();
    tc::fence_before_sync();
    __syncthreads();
}

// Forward pass of this thread's sample (f[3]; rows whose thread passes valid = false are
// computed on zero inputs and ignored; a tile without a valid row issues no MMA and leaves o
// at zero). kTanh selects the hardware-tanh activation. Returns false if a tensor-core wait
// timed out.
// Columns 0-3 of a sample's A-operand row as two packed bf16 pairs: the three inputs and the
// constant 1 of the first-layer bias.
__device__ __forceinline__ uint2 input_row(const float f[3]) {
    return make_uint2(tc::pack_bf16x2(f[0], f[1]), tc::pack_bf16x2(f[2], 1.0f));
}

// The network of a tile whose rows arrive packed (input_row); o is y = W3 h2 + b3 before the
// affine output map. Same waits and masking as fwd_tile.
template <bool kTanh>
__device__ __forceinline__ bool fwd_tile_y(FwdSmem& S, uint32_t& phase, uint2 row, bool valid,
                                           float y[7]) {
    const int t = threadIdx.x;
    *reinterpret_cast<uint2*>(S.x + tc::kmajor(t, 0, 16)) = valid ? row : make_uint2(0u, 0u);
    tc::fence_smem_to_async();
    tc::fence_before_sync();
    if (!__syncthreads_or(valid)) {
        tc::fence_after_sync();
#pragma unroll
        for (int k = 0; k < kOut; ++k) y[k] = 0.0f;
        return true;
    }
    if (t == 0) {
        tc::fence_after_sync();
        tc::gemm_bf16(S.tmem, S.x, S.w1, 64, 16);
        tc::mma_commit(&S.bar);
    }
    if (!cta_wait(S, phase)) return false;
    hidden_epilogue<kTanh>(S, nullptr);          // first-layer bias is in W1
    issue_barrier_then(S);
    if (t == 0) {
        tc::fence_after_sync();
        tc::gemm_bf16(S.tmem, S.h, S.w2, 64, 64);
        tc::mma_commit(&S.bar);
    }
    if (!cta_wait(S, phase)) return false;
    hidden_epilogue<kTanh>(S, S.b2);
    issue_barrier_then(S);
    if (t == 0) {
        tc::fence_after_sync();
        tc::gemm_bf16(S.tmem, S.h, S.w3, 16, 64);
        tc::mma_commit(&S.bar);
    }
    if (!cta_wait(S, phase)) return false;
    float v[16];
    tc::tmem_ld16(tc::tmem_lane_addr(S.tmem, 0), v);
#pragma unroll
    for (int k = 0; k < kOut; ++k) y[k] = v[k] + S.b3[k];
    tc::fence_before_sync();
    return true;
}

template <bool kTanh = false>
__device__ __forceinline__ bool fwd_tile(FwdSmem& S, uint32_t& phase, const float f[3], bool valid,
                                         float o[7]) {
    const int t = threadIdx.x;
    // columns 0-3 of the row: the three inputs and the constant 1 of the first-layer bias
    *reinterpret_cast<uint2*>(S.x + tc::kmajor(t, 0, 16)) =
        make_uint2(tc::pack_bf16x2(valid ? f[0] : 0.0f, valid ? f[1] : 0.0f),
                   tc::pack_bf16x2(valid ? f[2] : 0.0f, 1.0f));
    tc::fence_smem_to_async();
    tc::fence_before_sync();
    if (!__syncthreads_or(valid)) {
        tc::fence_after_sync();
#pragma unroll
        for (int k = 0; k < kOut; ++k) o[k] = 0.0f;
        return true;
    }
    if (t == 0) {
        tc::fence_after_sync();
        tc::gemm_bf16(S.tmem, S.x, S.w1, 64, 16);
        tc::mma_commit(&S.bar);
    }
    if (!cta_wait(S, phase)) return false;
    hidden_epilogue<kTanh>(S, nullptr);          // first-layer bias is in W1
    issue_barrier_then(S);
    if (t == 0) {
        tc::fence_after_sync();
        tc::gemm_bf16(S.tmem, S.h, S.w2, 64, 64);
        tc::mma_commit(&S.bar);
    }
    if (!cta_wait(S, phase)) return false;
    hidden_epilogue<kTanh>(S, S.b2);
    issue_barrier_then(S);
    if (t == 0) {
        tc::fence_after_sync();
        tc::gemm_bf16(S.tmem, S.h, S.w3, 16, 64);
        tc::mma_commit(&S.bar);
    }
    if (!cta_wait(S, phase)) return false;
    float v[16];
    tc::tmem_ld16(tc::tmem_lane_addr(S.tmem, 0), v);
#pragma unroll
    for (int k = 0; k < kOut; ++k)
        o[k] = S.mean[k] + S.scale[k] * (v[k] + S.b3[k]) + S.A[3 * k] * f[0] +
               S.A[3 * k + 1] * f[1] + S.A[3 * k + 2] * f[2];
    tc::fence_before_sync();
    return true;
}

// Release tensor memory. After a timed-out wait the outstanding MMA group is waited for
// once more (bounded) before the columns are freed.
__device__ __forceinline__ void fwd_finish(FwdSmem& S, uint32_t phase, bool ok) {
    if (!ok) tc::mbar_wait(&S.bar, phase ^ 1u, kWaitCycles);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (threadIdx.x < 32) tc::tmem_dealloc(S.tmem, kFwdCols);
}

// outputs o [n][7] for raw inputs [n][3] (log10 x, log10 Theta_e, |cos|); persistent tiles
__global__ void __launch_bounds__(128) forward_kernel(const float* __restrict__ P, int64_t n,
                                                      const float* __restrict__ in,
                                                      float* __restrict__ out, int* err) {
    __shared__ FwdSmem S;
    fwd_init(S, P);
    uint32_t phase = 0;
    bool ok = true;
    const int64_t tiles = (n + 127) / 128;
    for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        const int64_t i = tile * 128 + threadIdx.x;
        const bool valid = i < n;
        float f[3] = {0.0f, 0.0f, 0.0f};
        if (valid) {
            f[0] = 2.0f * (in[3 * i] - kLxLo) / (kLxHi - kLxLo) - 1.0f;
            f[1] = 2.0f * (in[3 * i + 1] - kLtLo) / (kLtHi - kLtLo) - 1.0f;
            f[2] = 2.0f * fabsf(in[3 * i + 2]) - 1.0f;
        }
        float o[7];
        ok = fwd_tile(S, phase, f, valid, o);
        if (ok && valid)
            for (int k = 0; k < kOut; ++k) out[7 * i + k] = o[k];
    }
    if (!ok && threadIdx.x == 0) atomicExch(err, 1);
    fwd_finish(S, phase, ok);
}

// The learned model over a trace's work list (the middle pass of the learned-coefficient
// transfer): row i of the list (fp32_samples_kernel) holds a sample's packed inputs in the first 8
// of its 32 bytes, which the model's outputs y[7] (padded to 8) replace. Full 128-row tiles, the
// row count read on the device, so the launch needs no host round trip. 1024^2: 2.6 ms; scanning the
// pool for the rows, 15.8 ms.
__global__ void __launch_bounds__(128) forward_list_kernel(const float* __restrict__ P,
                                                           const unsigned long long* __restrict__ n_rows,
                                                           float* __restrict__ list,
                                                           unsigned long long* timeouts) {
    __shared__ FwdSmem S;
    const int64_t n = (int64_t)*n_rows;
    const int64_t tiles = (n + 127) / 128;
    if ((int64_t)blockIdx.x >= tiles) return;
    fwd_init(S, P);
    uint32_t phase = 0;
    bool ok = true;
    const int t = threadIdx.x;
    uint2 next = make_uint2(0u, 0u);
    if ((int64_t)blockIdx.x * 128 + t < n)
        next = *reinterpret_cast<const uint2*>(list + 8 * ((int64_t)blockIdx.x * 128 + t));
    for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        const int64_t k = tile * 128 + t, kn = k + (int64_t)gridDim.x * 128;
        const uint2 row = next;
        if (kn < n) next = *reinterpret_cast<const uint2*>(list + 8 * kn);
        float y[7];
        ok = fwd_tile_y<true>(S, phase, row, k < n, y);
        if (ok && k < n) {
            float4* q = reinterpret_cast<float4*>(list + 8 * k);
            q[0] = make_float4(y[0], y[1], y[2], y[3]);
            q[1] = make_float4(y[4], y[5], y[6], 0.0f);
        }
    }
    if (!ok && t == 0) atomicAdd(timeouts, 1ull);
    fwd_finish(S, phase, ok);
}

// The affine output map o = offset + scale y + A f of the model, for a sample whose inputs f
// were those of its packed row (the transfer reads y from the pool pass and applies it).
__device__ __forceinline__ void model_outputs_from_y(const float* __restrict__ P, const float y[7],
                                                     const float f[3], float o[7]) {
#pragma unroll
    for (int k = 0; k < kOut; ++k)
        o[k] = __ldg(P + kOffMean + k) + __ldg(P + kOffScale + k) * y[k] +
               __ldg(P + kOffA + 3 * k) * f[0] + __ldg(P + kOffA + 3 * k + 1) * f[1] +
               __ldg(P + kOffA + 3 * k + 2) * f[2];
}

// coefficients [n][8] of plasma samples in [n][5] (n_e, Theta_e, B, nu, cos theta_B): the
// model inside its domain, the exact fits (FP32) outside it
__global__ void __launch_bounds__(128) coefficients_kernel(const float* __restrict__ P, int64_t n,
                                                           const double* __restrict__ in,
                                                           double* __restrict__ out, int* err) {
    __shared__ FwdSmem S;
    fwd_init(S, P);
    uint32_t phase = 0;
    bool ok = true;
    const int64_t tiles = (n + 127) / 128;
    for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        const int64_t i = tile * 128 + threadIdx.x;
        const bool valid = i < n;
        float s[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (valid)
            for (int q = 0; q < 5; ++q) s[q] = (float)in[5 * i + q];
        const ModelIn m = model_inputs(s[1], s[2], s[3], s[4]);
        const bool use = valid && m.ok && s[0] > 0.0f;
        float o[7];
        ok = fwd_tile(S, phase, m.f, use, o);
        if (ok && valid) {
            float c[8];
            if (use) coefficients_from(o, s[0], s[1], s[2], s[3], s[4], c);
            else synchrotron_coefficients<float>(s[0], s[1], s[2], s[3], s[4], c);
            for (int q = 0; q < 8; ++q) out[8 * i + q] = (double)c[q];
        }
    }
    if (!ok && threadIdx.x == 0) atomicExch(err, 1);
    fwd_finish(S, phase, ok);
}

// ---------------------------------------------------------------------------------------
// Training: forward and backward of one 128-sample tile per CTA, all nine products on the
// tensor cores. Weight gradients contract over the samples (K = 128): the same shared-memory
// tiles as the forward and backward operands are then read MN-major (samples along K), with a
// column of ones appended to the activations, whose accumulator column yields the bias gradient;
// accumulator rows beyond the layer's units come from whatever follows the tile in shared memory
// and are never read.
// A step is a chain of five dependent products, so it is bound by latency, and what is not the
// chain is taken off it: the weights arrive as one bulk copy of an image in operand layout (bf16
// tiles, then the FP32 biases and output map) that adam_kernel keeps up to date, everything a
// thread stores to shared memory is 16 bytes wide, tile gradients go out in the order the
// accumulators come (slots), coalesced, and the next kernel's launch and the loads that do not
// depend on the weights overlap the step before (programmatic dependent launch). Batch 16384, a
// step (this kernel and adam_kernel): 41 us with the transposed copies, scalar stores and one
// weight staging a tile, 14.2 us so.
// ---------------------------------------------------------------------------------------
constexpr int kHPitch = 80;           // activation tiles: 64 units, the ones column, zeros
constexpr uint32_t kTX = 0;           // [128][16] X: inputs, ones column 3
constexpr uint32_t kTH1 = 4096;       // [128][80] H1
constexpr uint32_t kTH2 = 24576;      // [128][80] H2
constexpr uint32_t kTdZ3 = 45056;     // [128][16] dY
constexpr uint32_t kTdZ2 = 49152;     // [128][64] dZ2
constexpr uint32_t kTdZ1 = 65536;     // [128][64] dZ1
constexpr uint32_t kTImg = 81920;     // the weight image
constexpr uint32_t kTRed = 105472;    // float [32]
constexpr uint32_t kTBar = 105600;    // two mbarriers, tensor-memory base
constexpr uint32_t kTrainSmem = 105632;
// the weight image: byte offsets of its parts
constexpr uint32_t kIW1 = 0;          // [64][16] W1 (bias in column 3)
constexpr uint32_t kIW2 = 2048;       // [64][64] W2
constexpr uint32_t kIW3 = 10240;      // [16][64] W3 (rows 7-15 zero)
constexpr uint32_t kIW3T = 12288;     // [64][16] W3^T
constexpr uint32_t kIW2T = 14336;     // [64][64] W2^T
constexpr uint32_t kIF32 = 22528;     // float b2[64] b3[8] mean[8] scale[8] A[24]
constexpr uint32_t kImgBytes = kIF32 + 4 * 112;
static_assert(kTImg + kImgBytes <= kTRed && kImgBytes % 16 == 0, "weight image");
// tensor-memory columns (512 allocated)
constexpr int kCZ1 = 0, kCZ2 = 64, kCZ3 = 128, kCdH2 = 160, kCdW3 = 224, kCdH1 = 304,
              kCdW2 = 368, kCdW1 = 448;
constexpr uint32_t kTrainCols = 512;

// Slot order of the trained parameters (tile gradients, Adam state): the accumulators' order, W2
// and W3 by input unit first; the other parameters keep their places.
__device__ __forceinline__ int slot_param(int s) {
    if (s >= kOffW2 && s < kOffB2) {
        const int q = s - kOffW2;
        return kOffW2 + 64 * (q & 63) + (q >> 6);
    }
    if (s >= kOffW3 && s < kOffB3) {
        const int q = s - kOffW3, c = q / kOut;
        return kOffW3 + 64 * (q - kOut * c) + c;
    }
    return s;
}

// Parameter i (value w) in the weight image.
__device__ __forceinline__ void image_store(unsigned char* __restrict__ img, int i, float w) {
    float* fl = reinterpret_cast<float*>(img + kIF32);
    if (i < kOffW2) {
        tc::st_bf16(img + kIW1, i >> 2, i & 3, 16, w);
    } else if (i < kOffB2) {
        const int j = (i - kOffW2) >> 6, k = (i - kOffW2) & 63;
        tc::st_bf16(img + kIW2, j, k, 64, w);
        tc::st_bf16(img + kIW2T, k, j, 64, w);
    } else if (i < kOffW3) {
        fl[i - kOffB2] = w;
    } else if (i < kOffB3) {
        const int o = (i - kOffW3) >> 6, j = (i - kOffW3) & 63;
        tc::st_bf16(img + kIW3, o, j, 64, w);
        tc::st_bf16(img + kIW3T, j, o, 16, w);
    } else if (i < kOffMean) {
        fl[64 + i - kOffB3] = w;
    } else if (i < kOffScale) {
        fl[72 + i - kOffMean] = w;
    } else if (i < kOffA) {
        fl[80 + i - kOffScale] = w;
    } else {
        fl[88 + i - kOffA] = w;
    }
}

// The image of P (img zeroed beforehand: padding rows and columns) and, where w is given, the
// trained parameters in slot order.
__global__ void image_kernel(const float* __restrict__ P, unsigned char* __restrict__ img,
                             float* __restrict__ w) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kParams) return;
    image_store(img, i, P[i]);
    if (w && i < kOffMean) w[i] = P[slot_param(i)];
}
// The trained parameters back into P (not after a step whose wait ran out).
__global__ void unslot_kernel(const float* __restrict__ w, float* __restrict__ P,
                              const int* __restrict__ err) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < kOffMean && *err == 0) P[slot_param(s)] = w[s];
}

// Eight consecutive values of a row of a bf16 operand tile: one 16-byte store.
__device__ __forceinline__ void st_row8(unsigned char* tile, int row, int col, int pitch,
                                        const float v[8]) {
    *reinterpret_cast<uint4*>(tile + tc::kmajor(row, col, pitch)) =
        make_uint4(tc::pack_bf16x2(v[0], v[1]), tc::pack_bf16x2(v[2], v[3]),
                   tc::pack_bf16x2(v[4], v[5]), tc::pack_bf16x2(v[6], v[7]));
}

// Gradients of the mean squared error over n_total samples x 7 outputs and the summed squared
// error; block b takes the 128-sample tile b of the `count` samples starting at sample `first`
// of the n-sample set (wrapping around). With part == nullptr the tiles add into grad[kParams]
// and *loss atomically (summation order, and so the last bits, vary between runs). Otherwise
// tile b stores its own sums, part[b][kOffMean] (every trained parameter, in slot order) and
// part_loss[b], for a reduction in a fixed order (adam_kernel), which makes training
// reproducible bit for bit. *err: set where a wait runs out; a launch that finds it set computes
// nothing, so a run of steps waits out one limit, not one a step.
__global__ void __launch_bounds__(128, 1) train_kernel(const unsigned char* __restrict__ img,
                                                       int64_t n, const float* __restrict__ in,
                                                       const float* __restrict__ tg,
                                                       int64_t first, int64_t count,
                                                       double n_total, float* __restrict__ grad,
                                                       float* __restrict__ loss,
                                                       float* __restrict__ part,
                                                       float* __restrict__ part_loss, int* err) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const float* b2 = (const float*)(sm + kTImg + kIF32);
    const float* b3 = b2 + 64;
    const float* mean = b3 + 8;
    const float* scale = mean + 8;
    const float* Atr = scale + 8;
    float* red = (float*)(sm + kTRed);
    uint64_t* bar = (uint64_t*)(sm + kTBar);
    uint64_t* ibar = bar + 1;
    uint32_t* tbase = (uint32_t*)(sm + kTBar + 16);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;

    // ---- before the step's weights exist: tensor memory, barriers, this thread's sample (block
    // b takes samples first + 128 b + t (mod n), t < count), constant columns
    if (warp == 0) tc::tmem_alloc(tbase, kTrainCols);
    if (t == 0) {
        tc::mbar_init(bar, 1);
        tc::mbar_init(ibar, 1);
    }
    const int64_t base = (int64_t)blockIdx.x * 128;
    const bool valid = base + t < count;
    const int64_t i = (first + base + t) % n;
    float f[3] = {0.0f, 0.0f, 0.0f}, tn[7];
    if (valid) {
        f[0] = 2.0f * (in[3 * i] - kLxLo) / (kLxHi - kLxLo) - 1.0f;
        f[1] = 2.0f * (in[3 * i + 1] - kLtLo) / (kLtHi - kLtLo) - 1.0f;
        f[2] = 2.0f * fabsf(in[3 * i + 2]) - 1.0f;
    }
    for (int k = 0; k < kOut; ++k) tn[k] = valid ? tg[7 * i + k] : 0.0f;
    {
        const float zero[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        const float one[8] = {1.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        const float x[8] = {f[0], f[1], f[2], 1.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        st_row8(sm + kTX, t, 0, 16, x);
        st_row8(sm + kTX, t, 8, 16, zero);
        st_row8(sm + kTH1, t, 64, kHPitch, one);
        st_row8(sm + kTH1, t, 72, kHPitch, zero);
        st_row8(sm + kTH2, t, 64, kHPitch, one);
        st_row8(sm + kTH2, t, 72, kHPitch, zero);
        st_row8(sm + kTdZ3, t, 8, 16, zero);
    }
    tc::fence_smem_to_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tm = *tbase;
    uint32_t phase = 0;
    bool ok = true;
    auto wait = [&]() -> bool {
        const bool w = tc::mbar_wait(bar, phase, kWaitCycles);
        phase ^= 1u;
        const bool all = __syncthreads_and(w) != 0;
        tc::fence_after_sync();
        return all;
    };
    auto barrier = [&]() {
        tc::fence_smem_to_async();
        tc::fence_before_sync();
        __syncthreads();
    };
    // the 64 accumulator columns from `col` of this thread's row
    auto load64 = [&](int col, float v[64]) {
        uint32_t r[4][16];
#pragma unroll
        for (int c = 0; c < 4; ++c) tc::tmem_ld16_issue(tc::tmem_lane_addr(tm, col + 16 * c), r[c]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            tc::tmem_ld16_wait(r[c]);
#pragma unroll
            for (int j = 0; j < 16; ++j) v[16 * c + j] = __uint_as_float(r[c][j]);
        }
    };

    // ---- the weights of this step
    tc::grid_dependency_wait();
    tc::grid_launch_dependents();
    bool stopped = false;
    if (t == 0) {
        tc::bulk_load(sm + kTImg, img, kImgBytes, ibar);
        stopped = *(volatile const int*)err != 0;
    }
    const bool have = __syncthreads_and(tc::mbar_wait(ibar, 0u, kWaitCycles) && !stopped) != 0;

    do {
        if (!(ok = have)) break;
        for (int k = 0; k < kOut; ++k)
            tn[k] = valid ? (tn[k] - mean[k] - Atr[3 * k] * f[0] - Atr[3 * k + 1] * f[1] -
                             Atr[3 * k + 2] * f[2]) / scale[k]
                          : 0.0f;
        // ---- forward
        if (t == 0) {
            tc::fence_after_sync();
            tc::gemm_kmajor(tm + kCZ1, sm + kTX, 16, sm + kTImg + kIW1, 16, 64, 16);
            tc::mma_commit(bar);
        }
        if (!(ok = wait())) break;
        {
            float v[64];
            load64(kCZ1, v);
#pragma unroll
            for (int j = 0; j < 64; ++j) v[j] = silu(v[j]);
#pragma unroll
            for (int c = 0; c < 8; ++c) st_row8(sm + kTH1, t, 8 * c, kHPitch, v + 8 * c);
        }
        barrier();
        if (t == 0) {
            tc::fence_after_sync();
            tc::gemm_kmajor(tm + kCZ2, sm + kTH1, kHPitch, sm + kTImg + kIW2, 64, 64, 64);
            tc::mma_commit(bar);
        }
        if (!(ok = wait())) break;
        {
            float v[64];
            load64(kCZ2, v);
#pragma unroll
            for (int j = 0; j < 64; ++j) v[j] = silu(v[j] + b2[j]);
#pragma unroll
            for (int c = 0; c < 8; ++c) st_row8(sm + kTH2, t, 8 * c, kHPitch, v + 8 * c);
        }
        barrier();
        if (t == 0) {
            tc::fence_after_sync();
            tc::gemm_kmajor(tm + kCZ3, sm + kTH2, kHPitch, sm + kTImg + kIW3, 64, 16, 64);
            tc::mma_commit(bar);
        }
        if (!(ok = wait())) break;
        // ---- loss and output error dY = 2 (y - t) / (n_total 7)
        float se = 0.0f;
        {
            float v[16], dy[8];
            tc::tmem_ld16(tc::tmem_lane_addr(tm, kCZ3), v);
            const float sc = (float)(2.0 / (n_total * kOut));
            dy[7] = 0.0f;
#pragma unroll
            for (int k = 0; k < kOut; ++k) {
                const float e = valid ? v[k] + b3[k] - tn[k] : 0.0f;
                se += e * e;
                dy[k] = sc * e;
            }
            st_row8(sm + kTdZ3, t, 0, 16, dy);
        }
        for (int off = 16; off > 0; off >>= 1) se += __shfl_xor_sync(0xffffffffu, se, off);
        if (lane == 0) red[warp] = se;
        // ---- dH2 = dY W3 (waited for), dW3 (+ db3) = dY^T [H2, 1] (runs on)
        barrier();
        if (t == 0) {
            tc::fence_after_sync();
            tc::gemm_kmajor(tm + kCdH2, sm + kTdZ3, 16, sm + kTImg + kIW3T, 16, 64, 16);
            tc::mma_commit(bar);
            tc::gemm_mnmajor(tm + kCdW3, sm + kTdZ3, 16, sm + kTH2, kHPitch, 80, 128);
            const float tile_loss = red[0] + red[1] + red[2] + red[3];
            if (part_loss) part_loss[blockIdx.x] = tile_loss;
            else atomicAdd(loss, tile_loss);
        }
        if (!(ok = wait())) break;
        // ---- dZ2 = dH2 * silu'(Z2)
        {
            float dh[64], z[64];
            load64(kCdH2, dh);
            load64(kCZ2, z);
#pragma unroll
            for (int j = 0; j < 64; ++j) dh[j] = dh[j] * silu_grad(z[j] + b2[j]);
#pragma unroll
            for (int c = 0; c < 8; ++c) st_row8(sm + kTdZ2, t, 8 * c, 64, dh + 8 * c);
        }
        // ---- dH1 = dZ2 W2 (waited for), dW2 (+ db2) = dZ2^T [H1, 1] (runs on)
        barrier();
        if (t == 0) {
            tc::fence_after_sync();
            tc::gemm_kmajor(tm + kCdH1, sm + kTdZ2, 64, sm + kTImg + kIW2T, 64, 64, 64);
            tc::mma_commit(bar);
            tc::gemm_mnmajor(tm + kCdW2, sm + kTdZ2, 64, sm + kTH1, kHPitch, 80, 128);
        }
        if (!(ok = wait())) break;
        // ---- dZ1 = dH1 * silu'(Z1)
        {
            float dh[64], z[64];
            load64(kCdH1, dh);
            load64(kCZ1, z);
#pragma unroll
            for (int j = 0; j < 64; ++j) dh[j] = dh[j] * silu_grad(z[j]);
#pragma unroll
            for (int c = 0; c < 8; ++c) st_row8(sm + kTdZ1, t, 8 * c, 64, dh + 8 * c);
        }
        // ---- dW1 (+ db1 in column 3) = dZ1^T X; the commit covers every product so far
        barrier();
        if (t == 0) {
            tc::fence_after_sync();
            tc::gemm_mnmajor(tm + kCdW1, sm + kTdZ1, 64, sm + kTX, 16, 16, 128);
            tc::mma_commit(bar);
        }
        if (!(ok = wait())) break;
        // ---- this tile's weight gradients (rows = units: lanes 0-63)
        float* const own = part ? part + (size_t)blockIdx.x * kOffMean : nullptr;
        if (warp < 2) {
            const int j = t;                    // unit of layers 1 and 2
            float v[64], u[16], w1[16];
            load64(kCdW2, v);                   // dW2 columns 0-63, db2 in column 64
            tc::tmem_ld16(tc::tmem_lane_addr(tm, kCdW2 + 64), u);
            tc::tmem_ld16(tc::tmem_lane_addr(tm, kCdW1), w1);
            if (own) {
#pragma unroll
                for (int c = 0; c < 64; ++c) own[kOffW2 + 64 * c + j] = v[c];
                own[kOffB2 + j] = u[0];
#pragma unroll
                for (int q = 0; q < 4; ++q) own[kOffW1 + 4 * j + q] = w1[q];
            } else {
                for (int c = 0; c < 64; ++c) atomicAdd(&grad[kOffW2 + 64 * j + c], v[c]);
                atomicAdd(&grad[kOffB2 + j], u[0]);
                for (int q = 0; q < 4; ++q) atomicAdd(&grad[kOffW1 + 4 * j + q], w1[q]);
            }
        }
        if (warp == 0) {                        // dW3 rows 0-6, db3 in column 64
            float v[64], u[16];
            load64(kCdW3, v);
            tc::tmem_ld16(tc::tmem_lane_addr(tm, kCdW3 + 64), u);
            if (lane < kOut) {
                if (own) {
#pragma unroll
                    for (int c = 0; c < 64; ++c) own[kOffW3 + kOut * c + lane] = v[c];
                    own[kOffB3 + lane] = u[0];
                } else {
                    for (int c = 0; c < 64; ++c) atomicAdd(&grad[kOffW3 + 64 * lane + c], v[c]);
                    atomicAdd(&grad[kOffB3 + lane], u[0]);
                }
            }
        }
    } while (false);
    if (!ok) {
        // no copy and no product of this CTA stays in flight (bounded)
        if (t == 0) atomicExch(err, 1);
        if (!have) tc::mbar_wait(ibar, 0u, kWaitCycles);
        else {
            if (t == 0) tc::mma_commit(bar);
            tc::mbar_wait(bar, phase ^ 1u, kWaitCycles);
            tc::mbar_wait(bar, phase, kWaitCycles);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tm, kTrainCols);
}

// One Adam step (Kingma & Ba 2015) on every trained parameter (slot order) from the tiles'
// gradient sums, added in tile order: a block takes 32 slots, its eight warps bring their columns
// of 128 tiles into shared memory at once (16 loads in flight a thread; one thread a slot walking
// the tiles in device memory took twice the time), one warp adds them. c1, c2 are the bias
// corrections 1 - beta1^t, 1 - beta2^t. Writes the new weight into the next step's image. The
// last block adds the tiles' squared errors into loss_hist (mean over n_total x 7). Where a tile's
// wait ran out (*err) its sums are missing: loss_hist stays, and what becomes of w no longer matters
// (unslot_kernel).
constexpr int kAdamThreads = 256, kAdamTiles = 128;
constexpr int kAdamBlocks = (kOffMean + 31) / 32 + 1;
__global__ void __launch_bounds__(kAdamThreads) adam_kernel(
        float* __restrict__ w, unsigned char* __restrict__ img, const float* __restrict__ part,
        int n_tiles, float* __restrict__ m, float* __restrict__ v, float lr, float beta1,
        float beta2, float eps, float c1, float c2, const float* __restrict__ part_loss,
        float* loss_hist, float inv_count, const int* err) {
    __shared__ float col[kAdamTiles][32];
    __shared__ int stopped;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    tc::grid_dependency_wait();
    tc::grid_launch_dependents();
    const bool is_loss = blockIdx.x == kAdamBlocks - 1;
    const int s = blockIdx.x * 32 + lane;
    const bool on = is_loss ? lane == 0 && loss_hist != nullptr : s < kOffMean;
    const float* src = is_loss ? part_loss : part + s;
    const size_t stride = is_loss ? 1 : kOffMean;
    float mo = 0.0f, vo = 0.0f, wo = 0.0f, g = 0.0f;
    // (an idle lane's load, beside the others': read by the storing lane it costs 0.9 us a step)
    if (is_loss && threadIdx.x == 33) stopped = *(volatile const int*)err;
    if (warp == 0 && on && !is_loss) {
        mo = m[s];
        vo = v[s];
        wo = w[s];
    }
    for (int b0 = 0; b0 < n_tiles; b0 += kAdamTiles) {
        const int nb = n_tiles - b0 < kAdamTiles ? n_tiles - b0 : kAdamTiles;
#pragma unroll
        for (int k = 0; k < kAdamTiles / 8; ++k) {
            const int b = warp + 8 * k;
            if (on && b < nb) col[b][lane] = src[(size_t)(b0 + b) * stride];
        }
        __syncthreads();
        if (warp == 0 && on) {
#pragma unroll 8
            for (int b = 0; b < nb; ++b) g += col[b][lane];
        }
        __syncthreads();
    }
    if (warp != 0 || !on) return;
    if (is_loss) {
        if (!stopped) *loss_hist = g * inv_count;
        return;
    }
    // (roundings written out: a run's bits do not hang on the compiler's choice of products)
    const float mi = __fmaf_rn(1.0f - beta1, g, __fmul_rn(beta1, mo));
    const float vi = __fmaf_rn(__fmul_rn(1.0f - beta2, g), g, __fmul_rn(beta2, vo));
    m[s] = mi;
    v[s] = vi;
    const float wn = wo - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[s] = wn;
    image_store(img, slot_param(s), wn);
}

// n uniform samples of the input box (SplitMix64 stream `seed`: draws 3i, 3i+1, 3i+2) and
// their targets from the exact fits.
__global__ void dataset_kernel(int64_t n, uint64_t seed, float* __restrict__ in,
                               float* __restrict__ tg) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double lx = kLxLo + (kLxHi - kLxLo) * uniform01(seed, 3 * i);
    const double lt = kLtLo + (kLtHi - kLtLo) * uniform01(seed, 3 * i + 1);
    const double c = uniform01(seed, 3 * i + 2);
    in[3 * i] = (float)lx;
    in[3 * i + 1] = (float)lt;
    in[3 * i + 2] = (float)c;
    double o[7];
    exact_targets((double)(float)lx, (double)(float)lt, o);
    for (int k = 0; k < kOut; ++k) tg[7 * i + k] = (float)o[k];
}

__global__ void targets_kernel(int64_t n, const float* __restrict__ in, float* __restrict__ tg) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    double o[7];
    exact_targets((double)in[3 * i], (double)in[3 * i + 1], o);
    for (int k = 0; k < kOut; ++k) tg[7 * i + k] = (float)o[k];
}

// Glorot-uniform weights from SplitMix64 stream `seed` (draw i for parameter i), zero biases,
// output mean 0 and scale 1.
__global__ void init_kernel(float* __restrict__ P, uint64_t seed) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kParams) return;
    const float u = (float)(2.0 * uniform01(seed, (uint64_t)i) - 1.0);
    float v = 0.0f;
    if (i < kOffW2) v = (i & 3) == 3 ? 0.0f : u * sqrtf(6.0f / (3 + 64));
    else if (i < kOffB2) v = u * sqrtf(6.0f / (64 + 64));
    else if (i >= kOffW3 && i < kOffB3) v = u * sqrtf(6.0f / (64 + 7));
    else if (i >= kOffScale && i < kOffA) v = 1.0f;
    P[i] = v;
}

// Offset, trend A and scale of the model from n training samples: least squares of the targets on
// (f, 1), f the mapped inputs, by the normal equations in double precision, and the root mean
// square of the residual. Two passes over the samples, each over the whole device: block sums
// into part[block][38] (10 of f f^T, 28 of f o^T) or part[block][7] (squared residuals), which
// one block then adds in block order. A single
// block, latency and one SM's FP64 lanes deep, took 14.3 ms for 2^19 samples; the whole call now
// takes 0.46 ms (2^22: 1.14 ms).
__device__ __forceinline__ void features_of(const float* in, int64_t i, double f[4]) {
    f[0] = 2.0f * (in[3 * i] - kLxLo) / (kLxHi - kLxLo) - 1.0f;
    f[1] = 2.0f * (in[3 * i + 1] - kLtLo) / (kLtHi - kLtLo) - 1.0f;
    f[2] = 2.0f * fabsf(in[3 * i + 2]) - 1.0f;
    f[3] = 1.0;
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh[w];
    return s;
}

constexpr int kNormSums = 38, kNormThreads = 128;
__global__ void __launch_bounds__(kNormThreads) normalise_sums_kernel(
        int64_t n, const float* __restrict__ in, const float* __restrict__ tg,
        double* __restrict__ part) {
    __shared__ double sh[32];
    double s[kNormSums];
#pragma unroll
    for (int q = 0; q < kNormSums; ++q) s[q] = 0.0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        double f[4];
        features_of(in, i, f);
        int q = 0;
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = a; b < 4; ++b) s[q++] += f[a] * f[b];
#pragma unroll
        for (int k = 0; k < kOut; ++k) {
            const double o = (double)tg[7 * i + k];
#pragma unroll
            for (int a = 0; a < 4; ++a) s[10 + 7 * a + k] += f[a] * o;
        }
    }
#pragma unroll
    for (int q = 0; q < kNormSums; ++q) {
        const double v = block_sum(s[q], sh);
        if (threadIdx.x == 0) part[(size_t)blockIdx.x * kNormSums + q] = v;
    }
}

// beta[a][k]: solution of the normal equations (one block).
__global__ void normalise_solve_kernel(int blocks, const double* __restrict__ part,
                                       double* __restrict__ beta) {
    __shared__ double sum[kNormSums];
    const int t = threadIdx.x;
    if (t < kNormSums) {
        double v = 0.0;
        for (int b = 0; b < blocks; ++b) v += part[(size_t)b * kNormSums + t];
        sum[t] = v;
    }
    __syncthreads();
    if (t != 0) return;
    // Gaussian elimination with partial pivoting on [G | R]
    double M[4][11];
    int q = 0;
    for (int a = 0; a < 4; ++a)
        for (int b = a; b < 4; ++b) M[a][b] = M[b][a] = sum[q++];
    for (int a = 0; a < 4; ++a)
        for (int k = 0; k < kOut; ++k) M[a][4 + k] = sum[10 + 7 * a + k];
    for (int c = 0; c < 4; ++c) {
        int p = c;
        for (int a = c + 1; a < 4; ++a) if (fabs(M[a][c]) > fabs(M[p][c])) p = a;
        for (int b = 0; b < 11; ++b) { const double tmp = M[c][b]; M[c][b] = M[p][b]; M[p][b] = tmp; }
        for (int a = c + 1; a < 4; ++a) {
            const double fct = M[a][c] / M[c][c];
            for (int b = c; b < 11; ++b) M[a][b] -= fct * M[c][b];
        }
    }
    double be[4][7];
    for (int k = 0; k < kOut; ++k)
        for (int a = 3; a >= 0; --a) {
            double v = M[a][4 + k];
            for (int b = a + 1; b < 4; ++b) v -= M[a][b] * be[b][k];
            be[a][k] = v / M[a][a];
        }
    for (int a = 0; a < 4; ++a)
        for (int k = 0; k < kOut; ++k) beta[7 * a + k] = be[a][k];
}

__global__ void __launch_bounds__(kNormThreads) normalise_residual_kernel(
        int64_t n, const float* __restrict__ in, const float* __restrict__ tg,
        const double* __restrict__ beta, double* __restrict__ part) {
    __shared__ double sh[32], be[28];
    if (threadIdx.x < 28) be[threadIdx.x] = beta[threadIdx.x];
    __syncthreads();
    double e[7] = {0, 0, 0, 0, 0, 0, 0};
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        double f[4];
        features_of(in, i, f);
#pragma unroll
        for (int k = 0; k < kOut; ++k) {
            const double d = (double)tg[7 * i + k] - (be[k] * f[0] + be[7 + k] * f[1] +
                                                      be[14 + k] * f[2] + be[21 + k]);
            e[k] += d * d;
        }
    }
#pragma unroll
    for (int k = 0; k < kOut; ++k) {
        const double v = block_sum(e[k], sh);
        if (threadIdx.x == 0) part[(size_t)blockIdx.x * kOut + k] = v;
    }
}

__global__ void normalise_store_kernel(int64_t n, int blocks, const double* __restrict__ part,
                                       const double* __restrict__ beta, float* __restrict__ P) {
    const int k = threadIdx.x;
    if (k >= kOut) return;
    double v = 0.0;
    for (int b = 0; b < blocks; ++b) v += part[(size_t)b * kOut + k];
    const double rms = sqrt(v / (double)n);
    P[kOffMean + k] = (float)beta[21 + k];
    P[kOffScale + k] = (float)(rms > 1e-30 ? rms : 1.0);
    for (int a = 0; a < 3; ++a) P[kOffA + 3 * k + a] = (float)beta[7 * a + k];
}

// Self-test of the bounded mbarrier wait: with arrive = 0 nothing arrives and the wait must
// run out after max_cycles (sets *err); with arrive = 1 the barrier's phase completes first.
__global__ void wait_selftest_kernel(long long max_cycles, int arrive, int* err) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) tc::mbar_init(&bar, 1);
    __syncthreads();
    if (arrive && threadIdx.x == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_addr(&bar)) : "memory");
    __syncthreads();
    const bool ok = tc::mbar_wait(&bar, 0u, max_cycles);
    if (!ok && threadIdx.x == 0) atomicExch(err, 1);
}

}  // namespace mlp
}  // namespace bl

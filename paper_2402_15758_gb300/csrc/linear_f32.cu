// fp32 linear for the fp32 model configuration: Y[M][N] (epilogue)= X[M][K] . W[N][K]^T.
//
// The fp32 model's matrices are small (0.3-2.8 MB, from L2), so a launch is bound by
// latency: how many dependent memory round trips a warp makes and how many warps share
// them.  A warp takes one or two output features for a tile of up to 16 token rows; a
// lane holds its share of a K chunk of the weight rows in registers, all of its loads in
// flight at once (requested before the dependency wait where the caller allows it), and
// the token rows come from shared memory, staged once per CTA.  The 16 (32) sums of a
// warp are reduced together: every butterfly step halves the values a lane still holds,
// 16 (31) shuffles instead of 80 (160).  fp32 FMA in a fixed order, so a launch is
// reproducible.  A second weight (gate and up) shares the launch.
//
// The row operation before a linear can be folded in, which takes a launch and its two
// memory trips off the step's chain: RMSNorm (the gains scale the weights in registers, the
// row's 1 / rms the result) and, for few rows, SwiGLU (in the staging; with 16 rows every CTA
// would work out 11000 of them).
//
// Measured on the GB300 (256-wide model, 2 layers, an event pair around every launch):
// the 9 linears of a 16-node verification 518 -> 78 us, the 28 of the draft (one row)
// 477 -> 191 us, against a kernel whose warps loaded X from global memory row by row and
// reduced each row's sum on its own; a 64-token prompt and eight steps 9.05 -> 2.73 ms.
#include "common.cuh"
#include "launch.cuh"
#include "kernels.h"

namespace chimera {
namespace {

constexpr int WARPS = 4;
constexpr int KC = 512;  // K per chunk: a lane holds KC / 32 weights of a feature

struct F32Args {
  const float* X;
  const float* W;
  const float* W2;  // features N1 .. N-1 (optional)
  float* Y;
  const int* skip;
  const float* g;  // RMSNorm gains of the K inputs (optional)
  float eps;
  int ldx, ldy, M, N, N1, K, epi, early_w;
  int swiglu;      // 1: X holds gate | up, the inputs are SiLU(gate) up
};

// Asynchronous copy of VEC floats into shared memory (zeros when !ok): every staging copy
// of a thread is in flight at once, without registers.
template <int VEC>
__device__ __forceinline__ void stage(float* dst, const float* src, bool ok) {
  if (VEC == 4)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(ok ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(ok ? 4 : 0) : "memory");
}

// Sum v[0..NV) over the warp; lane l returns the total of value (l >> log2(32 / NV)).
template <int NV>
__device__ __forceinline__ float warp_sum_many(float (&v)[NV], int lane) {
  int o = 16;
#pragma unroll
  for (int n = NV / 2; n >= 1; n /= 2, o /= 2) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float send = up ? v[i] : v[i + n];
      const float keep = up ? v[i + n] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  float t = v[0];
  for (; o >= 1; o /= 2) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// NORM: fold RMSNorm in.  Every warp sums the rows' squares along with the products (a lane's
// share of K is the same), so nothing more is exchanged.
// MT token rows x F features per warp; VEC = 4: K, ldx multiples of 4 and X, W (, W2)
// 16-byte aligned, else 1.
template <int MT, int F, int VEC, bool NORM>
__global__ void __launch_bounds__(WARPS * 32) f32_linear_kernel(const F32Args p) {
  constexpr int PER = KC / 32;  // a lane's weights of one feature in a chunk
  __shared__ __align__(16) float xs[MT == 1 ? 1 : MT * KC];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int f0 = (blockIdx.x * WARPS + warp) * F;
  const int m0 = blockIdx.y * MT, mt = min(MT, p.M - m0);
  float w[F][PER];
  auto load_w = [&](int k0) {
#pragma unroll
    for (int f = 0; f < F; ++f) {
      const int n = f0 + f;
      const float* row = n < p.N1 ? p.W + static_cast<size_t>(n) * p.K : p.W2 + static_cast<size_t>(n - p.N1) * p.K;
#pragma unroll
      for (int j = 0; j < PER / VEC; ++j) {
        const int k = k0 + (j * 32 + lane) * VEC;
        if (VEC == 4) {
          const float4 t = (n < p.N && k < p.K) ? *reinterpret_cast<const float4*>(row + k) : make_float4(0.f, 0.f, 0.f, 0.f);
          w[f][4 * j] = t.x;
          w[f][4 * j + 1] = t.y;
          w[f][4 * j + 2] = t.z;
          w[f][4 * j + 3] = t.w;
        } else {
          w[f][j] = (n < p.N && k < p.K) ? row[k] : 0.f;
        }
      }
    }
    if (!NORM) return;
#pragma unroll
    for (int j = 0; j < PER / VEC; ++j) {
      const int k = k0 + (j * 32 + lane) * VEC;
      if (VEC == 4) {
        const float4 g = k < p.K ? *reinterpret_cast<const float4*>(p.g + k) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int f = 0; f < F; ++f) {
          w[f][4 * j] *= g.x;
          w[f][4 * j + 1] *= g.y;
          w[f][4 * j + 2] *= g.z;
          w[f][4 * j + 3] *= g.w;
        }
      } else {
        const float g = k < p.K ? p.g[k] : 0.f;
#pragma unroll
        for (int f = 0; f < F; ++f) w[f][j] *= g;
      }
    }
  };
  pdl_trigger();  // the next kernel may start its prologue
  if (p.early_w) load_w(0);  // weights that no kernel of the stream writes
  pdl_wait();     // inputs of this kernel are complete
  if (p.skip && *reinterpret_cast<const volatile int*>(p.skip)) return;  // output already provided
  if (!p.early_w) load_w(0);
  float acc[F * MT];
#pragma unroll
  for (int i = 0; i < F * MT; ++i) acc[i] = 0.f;
  float ss[MT];
#pragma unroll
  for (int i = 0; i < MT; ++i) ss[i] = 0.f;
  for (int k0 = 0; k0 < p.K; k0 += KC) {
    const int kn = min(KC, p.K - k0);
    if constexpr (MT == 1) {  // one row: every warp reads it itself, next to its weights
      if (k0) load_w(k0);
      const float* src = p.X + static_cast<size_t>(m0) * p.ldx + k0;
      float x[PER];
#pragma unroll
      for (int j = 0; j < PER / VEC; ++j) {
        const int k = (j * 32 + lane) * VEC;
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < kn) {
          if (VEC == 4)
            t = *reinterpret_cast<const float4*>(src + k);
          else
            t.x = src[k];
          if (p.swiglu) {
            float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
            if (VEC == 4)
              u = *reinterpret_cast<const float4*>(src + p.K + k);
            else
              u.x = src[p.K + k];
            t = make_float4(silu_f(t.x) * u.x, silu_f(t.y) * u.y, silu_f(t.z) * u.z, silu_f(t.w) * u.w);
          }
        }
        const float e[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int i = 0; i < VEC; ++i) x[VEC * j + i] = e[i];
      }
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        if (NORM) ss[0] = fmaf(x[i], x[i], ss[0]);
#pragma unroll
        for (int f = 0; f < F; ++f) acc[f] = fmaf(w[f][i], x[i], acc[f]);
      }
      continue;
    }
    if (k0) {
      __syncthreads();  // every warp is done with the previous chunk
      load_w(k0);
    }
    // the token rows' chunk; rows past M are never read, columns past K are zero
    const int kr = (kn + 32 * VEC - 1) / (32 * VEC) * (32 * VEC);
    for (int m = warp; m < mt; m += WARPS) {
      const float* src = p.X + static_cast<size_t>(m0 + m) * p.ldx + k0;
      if (p.swiglu) {
        for (int k = lane * VEC; k < kr; k += 32 * VEC)
#pragma unroll
          for (int e = 0; e < VEC; ++e) xs[m * KC + k + e] = k < kn ? silu_f(src[k + e]) * src[p.K + k + e] : 0.f;
      } else {
        for (int k = lane * VEC; k < kr; k += 32 * VEC) stage<VEC>(xs + m * KC + k, k < kn ? src + k : src, k < kn);
      }
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int j = 0; j < PER / VEC; ++j) {
      if (j * 32 * VEC >= kn) break;
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        if (m >= mt) break;
        const float* x = xs + m * KC + (j * 32 + lane) * VEC;
        if (VEC == 4) {
          const float4 t = *reinterpret_cast<const float4*>(x);
          if (NORM) ss[m] = fmaf(t.w, t.w, fmaf(t.z, t.z, fmaf(t.y, t.y, fmaf(t.x, t.x, ss[m]))));
#pragma unroll
          for (int f = 0; f < F; ++f) {
            float a = acc[f * MT + m];
            a = fmaf(w[f][4 * j], t.x, a);
            a = fmaf(w[f][4 * j + 1], t.y, a);
            a = fmaf(w[f][4 * j + 2], t.z, a);
            acc[f * MT + m] = fmaf(w[f][4 * j + 3], t.w, a);
          }
        } else {
          const float t = *x;
          if (NORM) ss[m] = fmaf(t, t, ss[m]);
#pragma unroll
          for (int f = 0; f < F; ++f) acc[f * MT + m] = fmaf(w[f][j], t, acc[f * MT + m]);
        }
      }
    }
  }
  float s = warp_sum_many(acc, lane);
  constexpr int SUB = 32 / (F * MT);  // lanes that hold the same sum
  const int v = lane / SUB, f = f0 + v / MT, m = m0 + v % MT;
  if (NORM) {
    const float r = rsqrtf(warp_sum_many(ss, lane) / static_cast<float>(p.K) + p.eps);  // of row lane / (32 / MT)
    s *= __shfl_sync(0xffffffffu, r, (v % MT) * (32 / MT));
  }
  if (lane % SUB == 0 && f < p.N && m < p.M) {
    float* y = p.Y + static_cast<size_t>(m) * p.ldy + f;
    if (p.epi == EPI_RESID)
      *y += s;
    else
      *y = (p.epi == EPI_SILU) ? silu_f(s) : s;
  }
}

template <int MT, int F>
void launch(const F32Args& p, bool vec, cudaStream_t s) {
  const dim3 grid((p.N + WARPS * F - 1) / (WARPS * F), (p.M + MT - 1) / MT);
  auto* kernel = vec ? (p.g ? f32_linear_kernel<MT, F, 4, true> : f32_linear_kernel<MT, F, 4, false>)
                     : (p.g ? f32_linear_kernel<MT, F, 1, true> : f32_linear_kernel<MT, F, 1, false>);
  launch_pdl(kernel, grid, dim3(WARPS * 32), 0, s, p);
}

}  // namespace

cudaError_t f32_linear(int M, int N, int K, const float* X, int ldx, const float* W, float* Y,
                       int ldy, int epi, cudaStream_t s, const int* skip, const float* W2, int N2, bool early_w,
                       const F32Prologue& pro) {
  F32Args p{};
  p.X = X;
  p.W = W;
  p.W2 = W2;
  p.Y = Y;
  p.skip = skip;
  p.ldx = ldx;
  p.ldy = ldy;
  p.M = M;
  p.N1 = N;
  p.N = N + (W2 ? N2 : 0);
  p.K = K;
  p.epi = epi;
  p.early_w = early_w ? 1 : 0;
  p.g = pro.g;
  p.eps = pro.eps;
  p.swiglu = pro.swiglu ? 1 : 0;
  const bool vec = K % 4 == 0 && ldx % 4 == 0 && ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(W) |
                                                   reinterpret_cast<uintptr_t>(W2) | reinterpret_cast<uintptr_t>(pro.g)) & 15) == 0;
  // Token tiles of 1, 4 or 16 rows (a one-row tile stages an eighth of what 16 rows take
  // and needs no more registers than its K share).  Two features per warp only when one
  // each would put more than eight warps on every SM: below that the extra warps hide
  // latency, above it the shared-memory reads of the token tile bound the launch and two
  // features halve them.
  if (M == 1)
    launch<1, 1>(p, vec, s);
  else if (M <= 4)
    launch<4, 1>(p, vec, s);
  else if (static_cast<long long>(p.N) * ((M + 15) / 16) <= 4864)
    launch<16, 1>(p, vec, s);
  else
    launch<16, 2>(p, vec, s);
  return cudaGetLastError();
}

}  // namespace chimera

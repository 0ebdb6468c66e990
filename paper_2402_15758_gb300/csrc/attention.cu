// Tree-masked attention over the paged KV cache (tree verification, prefill chunks
// and the draft's full-context layer).
//
// Keys of sequence b: the n_ctx[b] committed rows (visible to every query) followed by
// n_local rows at slots n_ctx..n_ctx+n_local-1; query i sees local row j iff bit j of
// anc[q_local0 + i] is set (a tree node's ancestors-or-self, or a causal chain).
// KV layout: pool[layer][block][head][plane][16 rows][hd], page_table[b][slot / 16];
// planes K, V (fp32 models, plain bf16) or K_hi, K_lo, V_hi, V_lo (bf16 two-term split).
//
// This file holds the SIMT kernel (fp32 models, and bf16 models with head_dim 64), whose
// splits merge in the last CTA of each (b, h) through a global workspace, and the
// dispatch; bf16 models with head_dim 128 take the tensor-core kernel of attention_tc.cu.
// Both can also fuse RoPE and the KV write of the step's fresh rows (fp32 models here).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "attention.cuh"
#include "common.cuh"
#include "launch.cuh"
#include "kernels.h"

namespace chimera {
namespace {

constexpr int WARPS = 8;
constexpr int THREADS = WARPS * 32;
constexpr int KEYS = 64;         // keys of a CTA in flight: a row of each of four pages per half-warp
constexpr int MAX_NQ = 64;       // query rows per block
constexpr int SPLIT_KEYS = 256;  // a split is not worth fewer keys (four passes)
constexpr int MAX_SPLITS = 16;

// Merge the per-split partials (unnormalised output, running max, running sum) of the
// nq queries of one (b, h), in split order.  Run by the last CTA of the pair; every
// thread takes part: first the per-query weights exp(m_s - M) / L into shared memory,
// then the outputs, 4 dims per item, up to 8 items x 4 splits of loads in flight.
template <typename T>
__device__ void combine_splits(const AttnParams& p, const float* wsb, int nq, int hd, int row0, int h, T* out,
                               T* out_lo, float* s_w /* [nq][MAX_SPLITS] */) {
  const size_t rec = hd + 4;
  for (int qi = threadIdx.x; qi < nq; qi += blockDim.x) {
    float mv[MAX_SPLITS], lv[MAX_SPLITS];
#pragma unroll
    for (int sp = 0; sp < MAX_SPLITS; ++sp) {
      mv[sp] = -INFINITY;
      lv[sp] = 0.f;
      if (sp < p.splits) {
        const float* w = wsb + (static_cast<size_t>(sp) * p.nq_max + qi) * rec + hd;
        mv[sp] = __ldcg(w);
        lv[sp] = __ldcg(w + 1);
      }
    }
    float M = -INFINITY;
#pragma unroll
    for (int sp = 0; sp < MAX_SPLITS; ++sp) M = fmaxf(M, mv[sp]);
    float L = 0.f;
#pragma unroll
    for (int sp = 0; sp < MAX_SPLITS; ++sp) {
      mv[sp] = (M == -INFINITY || mv[sp] == -INFINITY) ? 0.f : expf(mv[sp] - M);
      L += mv[sp] * lv[sp];
    }
    const float inv = L > 0.f ? 1.f / L : 0.f;
#pragma unroll
    for (int sp = 0; sp < MAX_SPLITS; ++sp)
      if (sp < p.splits) s_w[qi * MAX_SPLITS + sp] = mv[sp] * inv;
  }
  __syncthreads();
  constexpr int J = 8;
  const int c4n = hd / 4;
  const int items = nq * c4n;
  const int nt = blockDim.x;
  for (int it0 = threadIdx.x; it0 < items; it0 += J * nt) {
    float4 acc[J];
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int sp0 = 0; sp0 < p.splits; sp0 += 4) {
      float4 v[J][4];
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const int it = it0 + j * nt;
        const int qi = it / c4n, c = (it % c4n) * 4;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (it < items && sp0 + u < p.splits)
            v[j][u] = __ldcg(reinterpret_cast<const float4*>(wsb + (static_cast<size_t>(sp0 + u) * p.nq_max + qi) * rec + c));
      }
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const int it = it0 + j * nt;
        if (it >= items) continue;
        const int qi = it / c4n;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (sp0 + u < p.splits) {
            const float e = s_w[qi * MAX_SPLITS + sp0 + u];
            acc[j].x += e * v[j][u].x; acc[j].y += e * v[j][u].y; acc[j].z += e * v[j][u].z; acc[j].w += e * v[j][u].w;
          }
      }
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int it = it0 + j * nt;
      if (it >= items) continue;
      const int qi = it / c4n, c = (it % c4n) * 4;
      const size_t o = static_cast<size_t>(row0 + qi) * p.ldo + h * hd + c;
      store_act4(out, out_lo, o, acc[j]);
    }
  }
}

// Four consecutive elements of a KV row as loaded, one element at a time when the pool is not
// aligned for vectors, and their values.
template <typename TKV>
struct Raw4;
template <>
struct Raw4<float> {
  float4 v;
  __device__ __forceinline__ void load(const float* p, bool vec) {
    v = vec ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
  }
  __device__ __forceinline__ float4 value() const { return v; }
};
template <>
struct Raw4<bf16> {
  uint2 v;
  __device__ __forceinline__ void load(const bf16* p, bool vec) {
    if (vec) {
      v = *reinterpret_cast<const uint2*>(p);
    } else {
      const unsigned short* u = reinterpret_cast<const unsigned short*>(p);
      v = make_uint2(u[0] | static_cast<uint32_t>(u[1]) << 16, u[2] | static_cast<uint32_t>(u[3]) << 16);
    }
  }
  __device__ __forceinline__ float4 value() const {
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
    return make_float4(a.x, a.y, b.x, b.y);
  }
};

// Sum v[0..NV) over each half-warp (NV <= 16): lane l returns the total of value
// (l % 16) / (16 / NV); every step halves the values a lane still holds.
template <int NV>
__device__ __forceinline__ float half_sum_many(float (&v)[NV], int lane) {
  int o = 8;
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

// Latency bounds this kernel (the fp32 model's contexts are a few hundred rows), so it
// keeps dependent memory trips few: a half-warp takes one row of each of four pages, 16
// lanes per row, with the K and V of all four in flight at once, and scores them against
// QG queries from shared memory; the 16 partial sums of a query group are reduced
// together, and a lane keeps the running max and sum of one query.  No tile is staged and
// the warps meet once, at the end.  A CTA takes one query, up to 8, or up to 16 (8 at 128 dims);
// more queries are further CTAs.  (Every query of the group costs its products: 8 queries at 200
// rows, fp32, 15.5 us in a group of 16, 12.6 in one of 8.  bf16 pools took 18.6 and at 4000 rows, 8
// sequences of 16 heads, 378 with a branch on the pool's form around each load, which kept
// the next ones waiting; now 12.6 and 140.  16 queries: 18.9 -> 15.7.)  Measured (GB300,
// fp32, 4 heads of 64, an event pair around every launch): one query at 70 rows 19 -> 9 us,
// 16 tree rows 17 -> 13; a 64-token prompt and eight steps 2.70 -> 2.26 ms.  The kernel
// before staged 32-key tiles for all queries, kept seven of eight warps idle for one
// query, and always split 16 ways.
//
// ROPE: the queries come from the projections, and the CTA rotates and writes to the pool
// the fresh rows of its own key range before it reads that range: no other CTA's rows are
// needed, and CTAs of the same range (query groups) write the same values.  Six RoPE
// launches of a step's 73 are saved (fp32, 256 wide, 16-node tree: 186 -> 179 us a step).
template <typename TKV, typename T, int HD, int QG, bool ROPE>
__global__ void __launch_bounds__(THREADS) attn_kernel(const AttnParams p, int groups) {
  pdl_trigger();  // the next kernel may start its prologue
  pdl_wait();     // inputs of this kernel are complete
  constexpr int DV = HD / 64;        // float4 of a row per lane
  constexpr int LPQ = 16 / QG;       // lanes that hold the same query's state
  constexpr bool LO = !std::is_same_v<TKV, float>;  // the pool may hold lo planes
  __shared__ __align__(16) float qs[QG * HD];
  __shared__ __align__(16) float s_acc[WARPS * 1024];  // [WARPS][QG][HD], later combine_splits' weights
  __shared__ float s_m[WARPS * QG], s_l[WARPS * QG];
  __shared__ int s_last;

  const int s = blockIdx.x, h = blockIdx.y, g = blockIdx.z % groups;
  const QueryBlock qb(p, blockIdx.z / groups);
  const int b = qb.b, nctx = qb.nctx, nq = qb.nq;
  const int q0 = g * QG, nqg = max(0, min(QG, nq - q0));
  if (nqg == 0 && p.splits == 1) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, hl = lane & 15, hw = warp * 2 + (lane >> 4);
  const int total = nctx + qb.nloc;
  const int per = ((total + p.splits - 1) / p.splits + KEYS - 1) / KEYS * KEYS;
  const int k0 = s * per, k1 = nqg > 0 ? min(total, k0 + per) : 0;
  const TKV* pool = static_cast<const TKV*>(p.pool) + static_cast<size_t>(p.layer) * p.pool_layer_stride;
  const bool vec = (reinterpret_cast<uintptr_t>(p.pool) & (4 * sizeof(TKV) - 1)) == 0;
  const int v_ofs = p.planes / 2 * 16 * HD, lo_ofs = p.planes == 4 ? 16 * HD : 0;

  const int qi = hl / LPQ;           // this lane's query within the group
  const unsigned long long mask = qi < nqg ? p.anc[p.q_local0 + q0 + qi] : 0ull;
  if constexpr (ROPE) {
    constexpr int HALF = HD / 2, J4 = HALF / 4;
    // (cos, sin) of position n_ctx + pos_base + .. of row i, dims j .. j + 3 of a half
    auto angles = [&](int pos, int j, float4& c, float4& sn) {
      const float4* t = reinterpret_cast<const float4*>(p.rope + static_cast<size_t>(pos) * HALF + j);
      const float4 a = t[0], e = t[1];
      c = make_float4(a.x, a.z, e.x, e.z);
      sn = make_float4(a.y, a.w, e.y, e.w);
    };
    auto pos_of = [&](int i) { return nctx + p.pos_base + (p.pos_off ? p.pos_off[i] : i); };
    for (int it = threadIdx.x; it < QG * J4; it += THREADS) {
      const int i = it / J4, j = it % J4 * 4;
      float4 y1 = make_float4(0.f, 0.f, 0.f, 0.f), y2 = y1;
      if (i < nqg) {
        float4 c, sn;
        angles(min(max(pos_of(q0 + i), 0), p.max_pos - 1), j, c, sn);
        const float* src = p.qkv + static_cast<size_t>(qb.row0 + q0 + i) * p.ldqkv + h * HD + j;
        const float4 x1 = *reinterpret_cast<const float4*>(src), x2 = *reinterpret_cast<const float4*>(src + HALF);
        y1 = rot_lo(x1, x2, c, sn);
        y2 = rot_hi(x1, x2, c, sn);
      }
      *reinterpret_cast<float4*>(qs + i * HD + j) = y1;
      *reinterpret_cast<float4*>(qs + i * HD + HALF + j) = y2;
    }
    const int fresh0 = nctx + p.q_local0, f0 = max(0, k0 - fresh0), f1 = min(nq, k1 - fresh0);
    for (int it = threadIdx.x; it < (f1 - f0) * J4; it += THREADS) {
      const int i = f0 + it / J4, j = it % J4 * 4, slot = fresh0 + i, pos = pos_of(i);
      if (pos < 0 || pos >= p.max_pos || (slot >> 4) >= p.max_pages) {
        if (p.err) atomicOr(p.err, ERR_CAPACITY);
        continue;
      }
      float4 c, sn;
      angles(pos, j, c, sn);
      const float* src = p.qkv + static_cast<size_t>(qb.row0 + i) * p.ldqkv + (p.H + h) * HD + j;
      const float4 x1 = *reinterpret_cast<const float4*>(src), x2 = *reinterpret_cast<const float4*>(src + HALF);
      const float4 v1 = *reinterpret_cast<const float4*>(src + p.H * HD);
      const float4 v2 = *reinterpret_cast<const float4*>(src + p.H * HD + HALF);
      TKV* row = const_cast<TKV*>(pool) +
                 (static_cast<size_t>(p.page_table[b * p.max_pages + (slot >> 4)]) * p.H + h) * p.planes * 16 * HD +
                 (slot & 15) * HD + j;
      store4<TKV>(row, rot_lo(x1, x2, c, sn));
      store4<TKV>(row + HALF, rot_hi(x1, x2, c, sn));
      store4<TKV>(row + v_ofs, v1);
      store4<TKV>(row + v_ofs + HALF, v2);
    }
  } else {
    for (int it = threadIdx.x; it < QG * (HD / 4); it += THREADS) {
      const int i = it / (HD / 4), c = it % (HD / 4) * 4;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < nqg) {
        const float* src = p.q + static_cast<size_t>(qb.row0 + q0 + i) * p.ldq + h * HD + c;
        x = make_float4(src[0], src[1], src[2], src[3]);
      }
      *reinterpret_cast<float4*>(qs + i * HD + c) = x;
    }
  }
  __syncthreads();

  float m = -INFINITY, l = 0.f;
  float4 acc[QG][DV];
#pragma unroll
  for (int q = 0; q < QG; ++q)
#pragma unroll
    for (int d = 0; d < DV; ++d) acc[q][d] = make_float4(0.f, 0.f, 0.f, 0.f);

  for (int base = k0; base < k1; base += KEYS) {
    // key base + 16 u + hw: row hw of page base / 16 + u
    // (the branches on the pool's form surround all loads of a pass, and nothing is converted
    // before the last one is on its way)
    const TKV* row[4];
    bool in[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      in[u] = base + 16 * u + hw < k1;
      const int page = in[u] ? p.page_table[b * p.max_pages + base / 16 + u] : 0;
      row[u] = pool + (static_cast<size_t>(page) * p.H + h) * p.planes * 16 * HD + hw * HD + hl * 4;
    }
    auto load_rows = [&](Raw4<TKV>(&kr)[4][DV], Raw4<TKV>(&vr)[4][DV], int ofs, bool as_vec) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int d = 0; d < DV; ++d) {
          kr[u][d] = vr[u][d] = Raw4<TKV>{};
          if (in[u]) {
            kr[u][d].load(row[u] + ofs + 64 * d, as_vec);
            vr[u][d].load(row[u] + ofs + v_ofs + 64 * d, as_vec);
          }
        }
    };
    Raw4<TKV> kr[4][DV], vr[4][DV];
    if (vec)
      load_rows(kr, vr, 0, true);
    else
      load_rows(kr, vr, 0, false);
    float4 kk[4][DV], vv[4][DV];
    auto add4 = [](float4 x, float4 y) { return make_float4(x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w); };
    if (LO && lo_ofs) {
      Raw4<TKV> kl[4][DV], vl[4][DV];
      if (vec)
        load_rows(kl, vl, lo_ofs, true);
      else
        load_rows(kl, vl, lo_ofs, false);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int d = 0; d < DV; ++d) {
          kk[u][d] = add4(kr[u][d].value(), kl[u][d].value());
          vv[u][d] = add4(vr[u][d].value(), vl[u][d].value());
        }
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int d = 0; d < DV; ++d) {
          kk[u][d] = kr[u][d].value();
          vv[u][d] = vr[u][d].value();
        }
    }
    float part[4][QG];
#pragma unroll
    for (int q = 0; q < QG; ++q) {
#pragma unroll
      for (int d = 0; d < DV; ++d) {
        const float4 x = *reinterpret_cast<const float4*>(qs + q * HD + 64 * d + hl * 4);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float t = fmaf(x.x, kk[u][d].x, fmaf(x.y, kk[u][d].y, fmaf(x.z, kk[u][d].z, x.w * kk[u][d].w)));
          part[u][q] = d ? part[u][q] + t : t;
        }
      }
    }
    float sc[4], mx = -INFINITY;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int key = base + 16 * u + hw;
      const float t = half_sum_many(part[u], lane);
      const bool vis = key < k1 && (key < nctx || ((mask >> (key - nctx)) & 1ull));
      sc[u] = vis ? t * p.scale : -INFINITY;
      mx = fmaxf(mx, sc[u]);
    }
    const float mn = fmaxf(m, mx);
    const float corr = m == mn ? 1.f : expf(m - mn);  // (m = -inf: 0)
    float pr[4];
    l *= corr;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      pr[u] = sc[u] == -INFINITY ? 0.f : expf(sc[u] - mn);
      l += pr[u];
    }
    m = mn;
    const bool rescale = __any_sync(0xffffffffu, corr != 1.f);
#pragma unroll
    for (int q = 0; q < QG; ++q) {
      const int src = (lane & 16) + q * LPQ;
      if (rescale) {
        const float c = __shfl_sync(0xffffffffu, corr, src);
#pragma unroll
        for (int d = 0; d < DV; ++d) {
          acc[q][d].x *= c; acc[q][d].y *= c; acc[q][d].z *= c; acc[q][d].w *= c;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float w = __shfl_sync(0xffffffffu, pr[u], src);
#pragma unroll
        for (int d = 0; d < DV; ++d) {
          acc[q][d].x = fmaf(w, vv[u][d].x, acc[q][d].x);
          acc[q][d].y = fmaf(w, vv[u][d].y, acc[q][d].y);
          acc[q][d].z = fmaf(w, vv[u][d].z, acc[q][d].z);
          acc[q][d].w = fmaf(w, vv[u][d].w, acc[q][d].w);
        }
      }
    }
  }

  // ---- the two half-warps of a warp, then the eight warps ----
  {
    const float M = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
    const float f = m == -INFINITY ? 0.f : expf(m - M);
    l *= f;
    l += __shfl_xor_sync(0xffffffffu, l, 16);
#pragma unroll
    for (int q = 0; q < QG; ++q) {
      const float c = __shfl_sync(0xffffffffu, f, (lane & 16) + q * LPQ);
#pragma unroll
      for (int d = 0; d < DV; ++d) {
        float4 t = acc[q][d];
        t.x *= c; t.y *= c; t.z *= c; t.w *= c;
        t.x += __shfl_xor_sync(0xffffffffu, t.x, 16);
        t.y += __shfl_xor_sync(0xffffffffu, t.y, 16);
        t.z += __shfl_xor_sync(0xffffffffu, t.z, 16);
        t.w += __shfl_xor_sync(0xffffffffu, t.w, 16);
        if (lane < 16) *reinterpret_cast<float4*>(s_acc + (warp * QG + q) * HD + 64 * d + hl * 4) = t;
      }
    }
    if (lane < 16 && hl % LPQ == 0) {
      s_m[warp * QG + qi] = M;
      s_l[warp * QG + qi] = l;
    }
  }
  __syncthreads();
  T* out = static_cast<T*>(p.out);
  T* out_lo = static_cast<T*>(p.out_lo);
  const size_t rec = HD + 4;
  float* wsb = p.ws + (static_cast<size_t>(b * p.H + h) * p.splits) * p.nq_max * rec;
  for (int it = threadIdx.x; it < nqg * (HD / 4); it += THREADS) {
    const int q = it / (HD / 4), c = it % (HD / 4) * 4;
    float M = -INFINITY, L = 0.f;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) M = fmaxf(M, s_m[w * QG + q]);
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
      const float mw = s_m[w * QG + q];
      const float f = mw == -INFINITY ? 0.f : expf(mw - M);
      L += f * s_l[w * QG + q];
      const float4 t = *reinterpret_cast<const float4*>(s_acc + (w * QG + q) * HD + c);
      o.x = fmaf(f, t.x, o.x); o.y = fmaf(f, t.y, o.y); o.z = fmaf(f, t.z, o.z); o.w = fmaf(f, t.w, o.w);
    }
    if (p.splits == 1) {
      const float inv = L > 0.f ? 1.f / L : 0.f;
      const float4 y = make_float4(o.x * inv, o.y * inv, o.z * inv, o.w * inv);
      const size_t at = static_cast<size_t>(qb.row0 + q0 + q) * p.ldo + h * HD + c;
      store_act(out, out_lo, at, y.x);
      store_act(out, out_lo, at + 1, y.y);
      store_act(out, out_lo, at + 2, y.z);
      store_act(out, out_lo, at + 3, y.w);
    } else {
      float* w = wsb + (static_cast<size_t>(s) * p.nq_max + q0 + q) * rec;
      __stcg(reinterpret_cast<float4*>(w + c), o);
      if (c == 0) {
        __stcg(&w[HD], M);
        __stcg(&w[HD + 1], L);
      }
    }
  }
  if (p.splits == 1) return;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const int old = atomicAdd(&p.counters[b * p.H + h], 1);
    s_last = (old == p.splits * groups - 1) ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  combine_splits(p, wsb, nq, HD, qb.row0, h, out, out_lo, s_acc);
  if (threadIdx.x == 0) p.counters[b * p.H + h] = 0;
}

template <typename TKV, typename T, int HD>
cudaError_t launch(AttnParams p, cudaStream_t s) {
  constexpr int QG = 1024 / HD;  // 16 queries of 64 dims or 8 of 128 per CTA
  static_assert(WARPS * 1024 >= MAX_NQ * MAX_SPLITS, "the merge weights fit over the partials");
  // the page table bounds the context: a split of fewer than SPLIT_KEYS keys only adds a merge
  p.splits = std::max(1, std::min(p.splits, (p.max_pages * 16 + SPLIT_KEYS - 1) / SPLIT_KEYS));
  const int groups = p.nq_max == 1 ? 1 : (p.nq_max + QG - 1) / QG;
  const dim3 grid(p.splits, p.H, p.B * std::max(1, p.q_blocks) * groups);
  auto* kernel = p.nq_max == 1   ? attn_kernel<TKV, T, HD, 1, false>
                 : p.nq_max <= 8 ? attn_kernel<TKV, T, HD, 8, false>
                                 : attn_kernel<TKV, T, HD, QG, false>;
  if constexpr (std::is_same_v<TKV, float>) {
    if (p.qkv)
      kernel = p.nq_max == 1   ? attn_kernel<TKV, T, HD, 1, true>
               : p.nq_max <= 8 ? attn_kernel<TKV, T, HD, 8, true>
                               : attn_kernel<TKV, T, HD, QG, true>;
  }
  launch_pdl(kernel, grid, dim3(THREADS), 0, s, p, groups);
  return cudaGetLastError();
}

}  // namespace

size_t attn_ws_floats(int B, int H, int splits, int nq_max, int hd) {
  return static_cast<size_t>(B) * H * splits * nq_max * (hd + 4);
}

bool attn_on_tensor_cores(int dtype, int hd) { return dtype == 1 && hd == 128; }
// (bf16 models of 64-dim heads, for which no configuration is tuned, rotate in a launch of their own)
bool attn_fuses_rope(int dtype, int hd) { return dtype == 0 || attn_on_tensor_cores(dtype, hd); }

int attn_pick_splits(int dtype, int hd, int planes, int B, int H, int want) {
  if (!attn_on_tensor_cores(dtype, hd)) return want;
  return attention_tc_splits(planes, B * H, want);
}

cudaError_t attention(const AttnParams& p, int dtype, cudaStream_t s) {
  if (p.nq_max > MAX_NQ || p.nq_max < 1 || p.n_local > 64 || p.splits > MAX_SPLITS || p.splits < 1) return cudaErrorInvalidValue;
  if (p.planes != 2 && !(p.planes == 4 && dtype == 1)) return cudaErrorInvalidValue;
  // blocks of prompt rows: device row counts, no fused projections, one split per block
  if (p.q_blocks > 1 && (p.qkv || !p.nq_dev || !p.n_local_dev || p.q_local0 != 0 || p.nq != 64 || p.n_local != 64 || p.splits != 1))
    return cudaErrorInvalidValue;
  if (p.qkv && (!p.rope || !p.err || p.max_pos < 1 || (p.ldqkv & 3))) return cudaErrorInvalidValue;
  if (dtype == 0) {
    if (p.hd == 64) return launch<float, float, 64>(p, s);
    if (p.hd == 128) return launch<float, float, 128>(p, s);
  } else if (p.hd == 128) {
    if (p.splits > 8) return cudaErrorInvalidValue;  // one cluster of at most 8 CTAs per (b, h)
    return attention_tc(p, s);
  } else if (p.hd == 64) {
    if (p.qkv) return cudaErrorInvalidValue;
    return launch<bf16, bf16, 64>(p, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace chimera

// bf16 linear of split activations for many token rows, on CTA pairs (sm_103a,
// tcgen05.mma.cta_group::2 + TMA).
//
//   Y[M][N] (epilogue)= (X + X_lo)[M][K] . W[N][K]^T,  fp32 accumulation.
//
// Past 64 rows a linear on hi + lo activations does so much tensor work per weight byte
// (4 M flops per 2 bytes) that it is bound by the tensor cores and by what feeds them:
// shared-memory reads of the operands, L2 reads of the tiles.  Two SMs share a tile:
//
//   * A (weights): 256 features, 128 per CTA;
//   * B (activations): CTA 0 holds the hi rows and CTA 1 the lo rows of up to 128 tokens,
//     and one MMA with N = 2 x tokens multiplies the weights with both: the weights are
//     read from shared memory once, not once per term, and each half of the columns is
//     its own accumulator, added at the end.
//
// A stage of 128 K is 64 KB per CTA and 1024 tensor cycles (the traffic of a 256 x 256
// tile of a plain GEMM); three of weights and three or more of tokens are in flight.
// Stages of 64 K (six in flight) were 12-19 % slower: a weight request then takes 128 B of
// each row, half of what DRAM pages like.  Two token tiles per weight stage (48 KB per 1024
// cycles, both accumulators taken) won 3-5 % at 1024 rows and lost 2-14 % from 256 to 640
// (more partial tiles to add at the end).
//
// Work split: stream-K over (feature tile, K block) units and groups of pairs.  The W
// pairs of a group take the same units for W token tiles, so a weight tile is read by
// all of them at the same time: from DRAM once.  With the token tiles of a weight tile
// in one pair's range, one after the other, they were read again up to 40 us later
// (256 rows, 22016 x 4096: 85 us; grouped 74; grouped with 128 K stages 66).  Tiles cut
// between groups are added with reductions (EPI_RESID) or through a workspace by the
// last group to arrive, in group order (the other epilogues; deterministic).
//
// The fp32 accumulation in tensor memory rounds toward zero at every 16-wide K step, so
// its error grows with the number of steps.  A chain is cut after SEG_UNITS stages: the
// epilogue warps add each piece to fp32 registers (round to nearest) while the other
// accumulator buffer is being filled.  Error against 64 bits at 256 x 4096 x 11008:
// 1.9e-6, 9.3e-6 for linear_tc.cu.
//
// Measured (GB300, EPI_RESID, against the kernel of linear_tc.cu on the same shape):
// 22016 x 4096: 72 rows 34.8 -> 31.9 us, 128 rows 41.1 -> 35.1, 256 rows 77.5 -> 60.6
// (1.52 PFLOP/s), 512 rows 150.7 -> 108.7 (1.70);  4096 x 11008: 20.0 -> 18.8,
// 23.8 -> 20.7, 41.7 -> 32.5, 76.7 -> 55.2.
// Stored outputs, whose cut tiles go through the workspace (12288 x 4096, plain and SiLU to
// bf16): 100 rows 40.2 and 47 -> 30.0 and 31 us, 256 rows 66.7 and 81 -> 44.1 and 47.
// With the loads left out (wrong results) 256 rows of 22016 x 4096 take 45.7 us, without
// the weights' alone 47.8: what is left is the L2's feed of the SMs.
//
// Roles (576 threads per CTA): warp 0 issues the TMA loads of its CTA (both CTAs signal
// the full barrier of CTA 0), warp 1 of CTA 0 issues the MMAs of the pair, warps 2..17
// drain (warp w: TMEM lanes 32 (w % 4) .., quarter (w - 2) / 4 of the tile's tokens).
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "launch.cuh"
#include "kernels.h"

namespace chimera {
namespace {

constexpr int BM = 128;   // features per CTA
constexpr int ATOM = 64;  // K of one 128-byte swizzle atom
constexpr int BKA = 2;    // atoms per stage
constexpr int BK = ATOM * BKA;
constexpr int UK = 16;
constexpr int A_ATOM = BM * ATOM * 2;
constexpr int A_BYTES = A_ATOM * BKA;
constexpr int A_STAGES = 3;      // weight tiles in shared memory
constexpr int MAX_B_STAGES = 8;  // token tiles
constexpr int PIPE_SMEM = 200 * 1024;
constexpr int EPI_WARPS = 16;   // four per TMEM lane quarter: a quarter of the tile's tokens each
constexpr int THREADS = (2 + EPI_WARPS) * 32;
constexpr int SEG_UNITS = 2048 / BK;  // stages per accumulation chain
constexpr int RED_PITCH = 36;   // floats per token row of a warp's transpose buffer
constexpr int MAX_TILES = 8192;
constexpr int MAX_WIDTH = 8;

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// TMA tile load whose completion is signalled to an mbarrier of either CTA of the pair
// (`bar`: a shared::cluster address).
__device__ __forceinline__ void tma_load_2d_pair(void* smem_dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair_hint(void* smem_dst, const CUtensorMap* map, int c0, int c1,
                                                      uint32_t bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar), "l"(policy)
      : "memory");
}
// D (both CTAs' tensor memory) (+)= A . B^T with 128 rows of A and N / 2 rows of B in each CTA.
__device__ __forceinline__ void tc_mma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                 uint32_t accumulate, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(elected)
      : "memory");
}
// Arrive on the barrier at this offset in both CTAs once every MMA issued so far is done.
__device__ __forceinline__ void tc_commit_pair(uint64_t* bar, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %2, 0;\n\t"
      "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}" ::"r"(
          smem_u32(bar)),
      "h"(static_cast<uint16_t>(3)), "r"(elected)
      : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// 32 lanes x 8 columns; the wait names the registers so that no use is moved above it.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait8x2(uint32_t (&a)[8], uint32_t (&b)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                 "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])::"memory");
}
__device__ __forceinline__ bool bar_any(int id, int nthreads, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred pi, po;\n\t"
      "setp.ne.u32 pi, %1, 0;\n\t"
      "bar.red.or.pred po, %2, %3, pi;\n\t"
      "selp.u32 %0, 1, 0, po;\n\t}"
      : "=r"(r)
      : "r"(static_cast<uint32_t>(pred)), "r"(id), "r"(nthreads)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ uint32_t pair_of_unit(uint32_t u, uint32_t U, uint32_t P) { return ((u + 1) * P - 1) / U; }
__device__ __forceinline__ uint32_t unit_begin(uint32_t c, uint32_t U, uint32_t P) { return c * U / P; }

constexpr int G = 4;  // 8-token groups a warp holds: its quarter of the token tile

struct Ctrl {  // at the start of the aligned dynamic shared memory
  uint64_t full_a[A_STAGES], empty_a[A_STAGES], full_b[MAX_B_STAGES], empty_b[MAX_B_STAGES];
  uint64_t tfull[2], tempty[2], drain;
  uint32_t tmem;
  int abort, last;
  uint32_t issued, issued_par;  // stages requested, their parities; bits 0..: weight tiles, 8..: token tiles
};
constexpr int CTRL_BYTES = 1024;
static_assert(sizeof(Ctrl) <= CTRL_BYTES, "control block");
__device__ __forceinline__ uint8_t* smem_base() {
  extern __shared__ uint8_t smem_raw[];
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
}
__device__ __forceinline__ int b_bytes_of(const TcPairParams& p) { return p.TT * BK * 2; }  // a token tile in shared memory

// The units of this CTA's pair: W pairs side by side (a group) take the same units for W
// token tiles.
struct Work {
  uint32_t KB, W, U, P, pair, grp, begin, end;
  __device__ __forceinline__ explicit Work(const TcPairParams& p)
      : KB(p.kblocks), W(p.width), U(p.units), P(gridDim.x / (2 * p.width)), pair(blockIdx.x / 2), grp(pair / W),
        begin(unit_begin(grp, U, P)), end(unit_begin(grp + 1, U, P)) {}
  // tile of unit u: feature tile and token tile
  __device__ __forceinline__ int ft(const TcPairParams& p, uint32_t u) const {
    return static_cast<int>(u / KB % p.feat_tiles);
  }
  __device__ __forceinline__ int tt(const TcPairParams& p, uint32_t u) const {
    return static_cast<int>(u / KB / p.feat_tiles * W + pair % W);
  }
};

// Each role derives what it needs by itself, and the epilogue is written so that nothing is
// spilled at the 96 registers that 18 warps leave: shared memory takes almost all of L1, so
// a spill goes to L2.  With values shared between the roles, the reductions and the other
// epilogues in one kernel and 148 bytes of spills: 256 rows, 22016 x 4096 67.1 us (60.6),
// 4096 x 11008 40.0 (32.5); 640 rows 141.9 (132.3) and 75.6 (67.8).
__device__ __forceinline__ void produce(const TcPairParams& p, int lane, uint32_t rank) {
  if (lane == 0) {
    uint8_t* base = smem_base();
    Ctrl* c = reinterpret_cast<Ctrl*>(base);
    uint8_t* smem = base + CTRL_BYTES;
    uint8_t* smem_b = smem + A_STAGES * A_BYTES;
    const int b_bytes = b_bytes_of(p), b_atom = b_bytes / BKA;
    const Work w(p);
    volatile int* abort = &c->abort;
    // ---------------- TMA producer (each CTA: its features, its rows of B) ----------------
    const uint64_t pol_w = policy_evict_first();
    uint32_t issued = 0, issued_par = 0;
    const CUtensorMap* bmap = rank ? &p.tmB2 : &p.tmB;
    int sa = 0, sb = 0;
    uint32_t pa = 0, pb = 0;
    auto weight_tile = [&](uint32_t u, int& k, int& row) {
      const int half = w.ft(p, u) * 2 + static_cast<int>(rank);
      const bool second = half >= p.half_split;
      k = static_cast<int>(u % w.KB) * BK;
      row = (second ? half - p.half_split : half) * BM;
      return second ? &p.tmA2 : &p.tmA;
    };
    auto prefetch_a = [&](uint32_t u) {
      int k, row;
      const CUtensorMap* map = weight_tile(u, k, row);
#pragma unroll
      for (int a = 0; a < BKA; ++a) tma_prefetch_2d(map, k + a * ATOM, row);
    };
    auto load_a = [&](uint32_t u) {
      int k, row;
      const CUtensorMap* map = weight_tile(u, k, row);
      const uint32_t bar = dsmem_addr(smem_u32(&c->full_a[sa]), 0);
      if (!rank) mbar_arrive_expect_tx(&c->full_a[sa], static_cast<uint32_t>(2 * A_BYTES));
#pragma unroll
      for (int a = 0; a < BKA; ++a) {
        if (p.tok_tiles == 1)  // read by this pair alone
          tma_load_2d_pair_hint(smem + sa * A_BYTES + a * A_ATOM, map, k + a * ATOM, row, bar, pol_w);
        else
          tma_load_2d_pair(smem + sa * A_BYTES + a * A_ATOM, map, k + a * ATOM, row, bar);
      }
      issued |= 1u << sa;
      issued_par = (issued_par & ~(1u << sa)) | (pa << sa);
      if (++sa == A_STAGES) {
        sa = 0;
        pa ^= 1u;
      }
    };
    auto load_b = [&](uint32_t u) {
      const int row = w.tt(p, u) * p.TT, k = static_cast<int>(u % w.KB) * BK;
      const uint32_t bar = dsmem_addr(smem_u32(&c->full_b[sb]), 0);
      if (!rank) mbar_arrive_expect_tx(&c->full_b[sb], static_cast<uint32_t>(2 * b_bytes));
#pragma unroll
      for (int a = 0; a < BKA; ++a)
        tma_load_2d_pair(smem_b + sb * b_bytes + a * b_atom, bmap, k + a * ATOM, row, bar);
      issued |= 256u << sb;
      issued_par = (issued_par & ~(256u << sb)) | (pb << (8 + sb));
      if (++sb == p.b_stages) {
        sb = 0;
        pb ^= 1u;
      }
    };
    // the first two units' weights are requested before the dependency wait (as in
    // linear_tc.cu), into L2 alone when an earlier kernel may still be writing them
    uint32_t ua = w.begin;
    const uint32_t pre = min(w.begin + 2, w.end);
    if (p.early_w)
      for (; ua < pre; ++ua) load_a(ua);
    else
      for (uint32_t u = ua; u < pre; ++u) prefetch_a(u);
    pdl_wait();
    pdl_trigger();
    for (; ua < pre; ++ua) load_a(ua);
    bool ok = true;
    for (uint32_t u = w.begin; ok && u < w.end && !*abort; ++u) {
      if (u == ua) {
        ok = mbar_wait(&c->empty_a[sa], pa ^ 1u, abort, p.wait_ns);
        if (ok) load_a(ua++);
      }
      ok = ok && mbar_wait(&c->empty_b[sb], pb ^ 1u, abort, p.wait_ns);
      if (ok) load_b(u);
    }
    c->issued = issued;
    c->issued_par = issued_par;
  } else {
    pdl_wait();
    pdl_trigger();
  }
}

// Some role gave up (whichever: the others may have been done before).  A CTA must not end
// before its copies have landed.  They signal CTA 0's barriers, which CTA 1 cannot wait on and
// which stay short of bytes when only one CTA requested a stage: CTA 0 waits for its stages
// within a limit, and both let 10 ms pass (a copy takes microseconds).  The MMAs end before
// tensor memory is released.
__device__ __forceinline__ void settle(const TcPairParams& p) {
  Ctrl* c = reinterpret_cast<Ctrl*>(smem_base());
  const uint32_t rank = cluster_rank();
  if (threadIdx.x == 0) {
    if (!rank)
      for (int i = 0; i < 8 + p.b_stages; ++i)
        if (c->issued >> i & 1u)
          mbar_wait_plain(i < 8 ? &c->full_a[i] : &c->full_b[i - 8], c->issued_par >> i & 1u, 20000000ull);
    for (const uint64_t t0 = global_timer_ns(); global_timer_ns() - t0 < 10000000ull;) {
    }
  } else if (threadIdx.x >> 5 == 1 && !rank) {
    tc_commit_pair(&c->drain, elect_one());  // (the lane that issued them: the election is deterministic)
    mbar_wait_plain(&c->drain, 0, 200000000ull);
  }
}

__device__ __forceinline__ void multiply(const TcPairParams& p, uint32_t rank) {
  pdl_wait();
  pdl_trigger();
  __syncwarp();
  if (!rank) {
    uint8_t* base = smem_base();
    Ctrl* c = reinterpret_cast<Ctrl*>(base);
    uint8_t* smem = base + CTRL_BYTES;
    uint8_t* smem_b = smem + A_STAGES * A_BYTES;
    const int b_bytes = b_bytes_of(p), b_atom = b_bytes / BKA;
    const Work w(p);
    volatile int* abort = &c->abort;
    const uint32_t tmem_base = c->tmem;
    // ---------------- MMA issuer of the pair (the whole warp, one elected lane issues) ----------------
    const uint32_t elected = elect_one();
    const uint32_t n = 2 * p.TT;
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | (static_cast<uint32_t>(256 >> 4) << 24);
    const uint64_t desc_a = sw128_desc(smem_u32(smem)), desc_b = sw128_desc(smem_u32(smem_b));
    int sa = 0, sb = 0, buf = 0;
    uint32_t pa = 0, pb = 0, aphase = 0;
    bool ok = true;
    for (uint32_t u = w.begin; ok && u < w.end;) {
      const uint32_t tile_end = min(w.end, (u / w.KB + 1) * w.KB);
      const uint32_t seg_end = min(tile_end, u + SEG_UNITS);
      ok = mbar_wait_warp(&c->tempty[buf], aphase ^ 1u, abort, p.wait_ns);
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + buf * 256;
      uint32_t acc = 0;
      for (; ok && u < seg_end; ++u) {
        ok = mbar_wait_warp(&c->full_a[sa], pa, abort, p.wait_ns) && mbar_wait_warp(&c->full_b[sb], pb, abort, p.wait_ns);
        if (!ok) break;
        tc_fence_after();
        const uint64_t da = desc_a + static_cast<uint64_t>((sa * A_BYTES) >> 4);
        const uint64_t db = desc_b + static_cast<uint64_t>((sb * b_bytes) >> 4);
#pragma unroll
        for (int a = 0; a < BKA; ++a)
#pragma unroll
          for (int k = 0; k < ATOM / UK; ++k) {
            tc_mma_bf16_pair(d_tmem, da + static_cast<uint64_t>((a * A_ATOM + k * 32) >> 4),
                             db + static_cast<uint64_t>((a * b_atom + k * 32) >> 4), idesc, acc, elected);
            acc = 1;
          }
        tc_commit_pair(&c->empty_a[sa], elected);
        tc_commit_pair(&c->empty_b[sb], elected);
        if (++sa == A_STAGES) {
          sa = 0;
          pa ^= 1u;
        }
        if (++sb == p.b_stages) {
          sb = 0;
          pb ^= 1u;
        }
      }
      if (ok) tc_commit_pair(&c->tfull[buf], elected);
      buf ^= 1;
      if (buf == 0) aphase ^= 1u;
    }
  }
  __syncwarp();
}

template <bool RED>
__device__ __forceinline__ void drain_tiles(const TcPairParams& p, int warp, int lane, uint32_t rank) {
  pdl_wait();  // Y, the workspace and the counters are shared with earlier kernels
  pdl_trigger();
  if (p.zero) {  // this CTA's share (float4s) of a later linear's accumulator
    const long long n4 = p.zero_floats / 4, per = (n4 + gridDim.x - 1) / gridDim.x, z0 = blockIdx.x * per;
    float4* z = reinterpret_cast<float4*>(p.zero);
    for (long long i = z0 + (threadIdx.x - 64); i < min(n4, z0 + per); i += EPI_WARPS * 32)
      z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  uint8_t* base = smem_base();
  Ctrl* c = reinterpret_cast<Ctrl*>(base);
  const Work w(p);
  volatile int* abort = &c->abort;
  const uint32_t tmem_base = c->tmem;
  const int q = warp & 3, th = (warp - 2) >> 2;
  const int row = q * 32 + lane;
  // this warp's 8-token groups: a quarter of the tile's
  const int ng = p.TT / 8, per4 = (ng + 3) / 4;
  const int g0 = min(ng, th * per4), gn = min(ng, g0 + per4) - g0;
  const uint32_t tempty0 = dsmem_addr(smem_u32(&c->tempty[0]), 0);
  float* sw = reinterpret_cast<float*>(base + CTRL_BYTES + A_STAGES * A_BYTES + p.b_stages * b_bytes_of(p)) +
              (warp - 2) * 8 * RED_PITCH;  // this warp's transpose buffer
  float acc[G][8];
  int buf = 0;
  uint32_t aphase = 0;
  // 8 tokens (this warp's group `g`) x 32 features to the transpose buffer
  auto stage_group = [&](int g) {
#pragma unroll
    for (int i = 0; i < G; ++i)
      if (i == g) {
#pragma unroll
        for (int j = 0; j < 8; ++j) sw[j * RED_PITCH + lane] = acc[i][j];
      }
    __syncwarp();
  };
  bool ok = true;
  for (uint32_t u = w.begin; u < w.end;) {
    const uint32_t t = u / w.KB, tile_end = min(w.end, (t + 1) * w.KB);
    const int half = w.ft(p, u) * 2 + static_cast<int>(rank), tt = w.tt(p, u);
    const int f0 = half * BM + q * 32, m0 = tt * p.TT + g0 * 8;
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[g][j] = 0.f;
    while (ok && u < tile_end) {
      u = min(tile_end, u + SEG_UNITS);
      ok = mbar_wait(&c->tfull[buf], aphase, abort, p.wait_ns);
      ok = !bar_any(1, EPI_WARPS * 32, !ok);
      tc_fence_after();
      const uint32_t tbase = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + buf * 256 + g0 * 8;
#pragma unroll
      for (int g = 0; g < G; ++g) {
        if (ok && g < gn) {
          uint32_t r[8];
          uint32_t lo[8];
          tmem_ld8(tbase + g * 8, r);
          tmem_ld8(tbase + p.TT + g * 8, lo);
          tmem_wait8x2(r, lo);
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[g][j] += __uint_as_float(r[j]) + __uint_as_float(lo[j]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(tempty0 + buf * 8);
      buf ^= 1;
      if (buf == 0) aphase ^= 1u;
    }
    if (!ok) break;
    if (RED) {  // float4 reductions
#pragma unroll 1
      for (int g = 0; g < gn; ++g) {
        stage_group(g);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int j = h * 4 + (lane >> 3), k = (lane & 7) * 4, m = m0 + g * 8 + j;
          if (m < p.M && f0 + k < p.N)
            red_add_v4(static_cast<float*>(p.Y) + static_cast<size_t>(m) * p.ldy + f0 + k,
                       *reinterpret_cast<const float4*>(sw + j * RED_PITCH + k));
        }
        __syncwarp();
      }
      continue;
    }
    // ---- this pair's part of tile t is complete ----
    const int f = f0 + lane;
    const uint32_t c_first = pair_of_unit(t * w.KB, w.U, w.P), c_last = pair_of_unit(t * w.KB + w.KB - 1, w.U, w.P);
    // 8 tokens of this lane's feature
    auto store8 = [&](int m, const float (&v)[8]) {
      if (f >= p.N) return;
      if (p.epi == EPI_RESID) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (m + j < p.M) red_add_f32(static_cast<float*>(p.Y) + static_cast<size_t>(m + j) * p.ldy + f, v[j]);
        return;
      }
      if (p.epi == EPI_SILU) {
        float e[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) e[j] = 1.0f + expf(-v[j]);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (m + j >= p.M) break;
          const float x = v[j] / e[j];
          const size_t idx = static_cast<size_t>(m + j) * p.ldy + f;
          if (p.out_f32)
            static_cast<float*>(p.Y)[idx] = x;
          else
            store_act(static_cast<bf16*>(p.Y), static_cast<bf16*>(p.Y2), idx, x);
        }
        return;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const size_t idx = static_cast<size_t>(m + j) * p.ldy + f;
        if (m + j < p.M) {
          if (p.out_f32)
            static_cast<float*>(p.Y)[idx] = v[j];
          else
            store_act(static_cast<bf16*>(p.Y), static_cast<bf16*>(p.Y2), idx, v[j]);
        }
      }
    };
    // slot of group c's partial of this token tile: [token][feature]
    auto slot = [&](uint32_t c) {
      const int first_slot = (unit_begin(c, w.U, w.P) / w.KB == t) ? 0 : 1;
      return p.ws + static_cast<size_t>(2 * (2 * (c * w.W + w.pair % w.W) + rank) + first_slot) * BM * p.TT +
             static_cast<size_t>(g0 * 8) * BM + row;
    };
    const bool parts = p.epi != EPI_RESID && c_first != c_last;
    float* wsp = parts ? slot(w.grp) : nullptr;
    int* counter = p.counters + 2 * (t * w.W + w.pair % w.W) + rank;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      if (g < gn) {
        if (parts) {
#pragma unroll
          for (int j = 0; j < 8; ++j) __stcg(wsp + (g * 8 + j) * BM, acc[g][j]);
        } else {
          store8(m0 + g * 8, acc[g]);
        }
      }
    }
    if (parts) {  // the last pair to arrive sums the partials in pair order
      __threadfence();
      named_bar(1, EPI_WARPS * 32);
      if (threadIdx.x == 64) c->last = atomicAdd(counter, 1) == static_cast<int>(c_last - c_first) ? 1 : 0;
      named_bar(1, EPI_WARPS * 32);
      if (c->last) {
        __threadfence();
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[g][j] = 0.f;
        for (uint32_t c = c_first; c <= c_last; ++c) {  // a part's loads are all in flight at once
          const float* src = slot(c);
#pragma unroll
          for (int g = 0; g < G; ++g)
            if (g < gn) {
#pragma unroll
              for (int j = 0; j < 8; ++j) acc[g][j] += __ldcg(src + (g * 8 + j) * BM);
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g)
          if (g < gn) store8(m0 + g * 8, acc[g]);
        if (threadIdx.x == 64) *counter = 0;
      }
      named_bar(1, EPI_WARPS * 32);
    }
  }
}

template <bool RED>
__global__ void __launch_bounds__(THREADS, 1) __cluster_dims__(2, 1, 1)
    tc_pair_kernel(const __grid_constant__ TcPairParams p) {
  if (p.skip) {  // written by the previous kernel; the same value in both CTAs
    pdl_wait();
    if (*reinterpret_cast<const volatile int*>(p.skip)) {
      pdl_trigger();
      return;
    }
  }
  Ctrl* c = reinterpret_cast<Ctrl*>(smem_base());
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();

  if (threadIdx.x == 0) {
    for (int s = 0; s < A_STAGES; ++s) {
      mbar_init(&c->full_a[s], 1);
      mbar_init(&c->empty_a[s], 1);
    }
    for (int s = 0; s < p.b_stages; ++s) {
      mbar_init(&c->full_b[s], 1);
      mbar_init(&c->empty_b[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&c->tfull[b], 1);
      mbar_init(&c->tempty[b], 2 * EPI_WARPS);
    }
    mbar_init(&c->drain, 1);
    c->abort = 0;
    c->last = 0;
    mbar_fence_init();
  }
  if (warp == 0 && lane == 0) {
    prefetch_tensormap(&p.tmA);
    if (p.half_split < p.halves) prefetch_tensormap(&p.tmA2);  // a second weight
    prefetch_tensormap(&p.tmB);
    prefetch_tensormap(&p.tmB2);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&c->tmem)), "r"(512)
                 : "memory");
    __syncwarp();
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  __syncwarp();
  cluster_sync();  // the peer's barriers and tensor memory are ready
  tc_fence_after();
  if (warp == 0)
    produce(p, lane, rank);
  else if (warp == 1)
    multiply(p, rank);
  else
    drain_tiles<RED>(p, warp, lane, rank);

  tc_fence_before();
  __syncthreads();
  if (*const_cast<volatile int*>(&c->abort)) settle(p);
  __syncwarp();
  cluster_sync();  // both CTAs are done with each other's shared and tensor memory
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(c->tmem), "r"(512) : "memory");
  }
  if (threadIdx.x == 0 && *const_cast<volatile int*>(&c->abort)) atomicOr(p.err, ERR_TIMEOUT);
}

constexpr int MAX_DEVICES = 64;
std::mutex g_pair_mu;
bool g_pair_attr[MAX_DEVICES];

}  // namespace

int tc_pair_plan(TcPairPlan* plan, int M, int N1, int N2, int K, const void* X, const void* X_lo, int ldx, const void* W,
                 const void* W2, void* Y, void* Y_lo, int ldy, int epi, int out_f32, float* ws, int* counters, int* err,
                 unsigned long long wait_ns, float* zero, long long zero_floats) {
  TcPairParams& p = plan->p;
  memset(&p, 0, sizeof(p));
  p.M = M;
  p.N = N1 + N2;
  p.halves = (p.N + BM - 1) / BM;
  // an odd number of halves leaves CTA 1 of the last tile a half past the weights (read as
  // zeros): without a second weight every half, that one too, belongs to W's tensor map
  p.half_split = W2 ? N1 / BM : p.halves + 1;
  // token tiles of equal height, at most 128; the pair's MMA takes N = 2 TT in steps of 32
  p.vec_red = (epi == EPI_RESID && (reinterpret_cast<uintptr_t>(Y) & 15) == 0 && ldy % 4 == 0 && p.N % 4 == 0) ? 1 : 0;
  p.tok_tiles = (M + 127) / 128;
  p.TT = ((M + p.tok_tiles - 1) / p.tok_tiles + 15) / 16 * 16;
  p.kblocks = (K + BK - 1) / BK;
  // groups of at most MAX_WIDTH pairs read the same weight tiles at the same time
  const int rounds = (p.tok_tiles + MAX_WIDTH - 1) / MAX_WIDTH;
  p.width = (p.tok_tiles + rounds - 1) / rounds;
  p.feat_tiles = (p.halves + 1) / 2;
  const int groups = tc_num_sms() / 2 / p.width;
  const long long units = static_cast<long long>(rounds) * p.feat_tiles * p.kblocks;
  // A pair with little work spends its time on the ramp and on adding its part of a tile.
  // The line lies at 1000 stage-tokens per pair: 862 (256 rows, 2048 x 4096) 12.5 us here
  // and in linear_tc.cu, 539 (160 rows, same) 10.5 and 9.7, 808 (80 rows, 6144 x 4096) 13.9
  // and 13.5; 1078 (160 rows, 4096 x 4096) 14.9 and 15.8, 1132 (112 rows, 6144 x 4096) 15.1
  // and 15.5, 1724 (256 rows, 4096 x 4096) 17.1 and 19.2.
  if (units * p.TT < 1000ll * groups) return -1;
  if (2ll * rounds * p.width * p.feat_tiles > MAX_TILES || groups < 1 || units * (groups + 1) >= (1ll << 32)) return -1;
  p.units = static_cast<uint32_t>(units);
  const int b_bytes = p.TT * BK * 2;
  p.b_stages = std::min(MAX_B_STAGES, (PIPE_SMEM - A_STAGES * A_BYTES) / b_bytes);
  p.epi = epi;
  p.out_f32 = out_f32;
  p.Y = Y;
  p.Y2 = out_f32 ? nullptr : Y_lo;
  p.ldy = ldy;
  p.ws = ws;
  p.counters = counters;
  p.err = err;
  p.wait_ns = wait_ns;
  p.zero = zero;
  p.zero_floats = zero ? zero_floats : 0;
  plan->grid = 2 * p.width * static_cast<int>(std::min<long long>(units, groups));
  plan->smem = 1024 + CTRL_BYTES + A_STAGES * A_BYTES + static_cast<size_t>(p.b_stages) * b_bytes + EPI_WARPS * 8 * RED_PITCH * sizeof(float);
  if (encode_2d_bf16(&p.tmA, W, K, N1, K, ATOM, BM) != 0) return -2;
  if (W2 && encode_2d_bf16(&p.tmA2, W2, K, N2, K, ATOM, BM) != 0) return -2;
  if (encode_2d_bf16(&p.tmB, X, K, M, ldx, ATOM, p.TT) != 0) return -2;
  if (encode_2d_bf16(&p.tmB2, X_lo, K, M, ldx, ATOM, p.TT) != 0) return -2;
  return 0;
}

cudaError_t tc_pair_launch(const TcPairPlan& plan, cudaStream_t s) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  {
    std::lock_guard<std::mutex> lk(g_pair_mu);
    if (!g_pair_attr[dev]) {
      for (auto k : {tc_pair_kernel<false>, tc_pair_kernel<true>}) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
      }
      g_pair_attr[dev] = true;
    }
  }
  launch_pdl(plan.p.vec_red ? tc_pair_kernel<true> : tc_pair_kernel<false>, dim3(plan.grid), dim3(THREADS), plan.smem, s, plan.p);
  return cudaGetLastError();
}

}  // namespace chimera

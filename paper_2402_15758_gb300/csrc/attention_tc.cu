// Tree-masked attention on the 5th-generation tensor cores (bf16 models, head_dim 128).
//
// One CTA per (KV split s, head h, sequence b); the S splits of a (b, h) form one
// thread-block cluster and merge their partial states through distributed shared
// memory.  Per 64-key tile of the CTA's key range:
//
//   S  = Q K^T    tcgen05.mma, M = 64 queries, N = 64 keys, K = 128 dims, fp32 in TMEM
//   P  = exp(S - m) on the softmax warps (tcgen05.ld of S, mask, online max/sum)
//   O += P V      tcgen05.mma, M = 64 queries, N = 128 dims, K = 64 keys, fp32 in TMEM
//
// Every bf16 operand is a two-term split x = hi + lo of an fp32 value (queries, keys,
// values, probabilities); each product takes hi*hi + lo*hi + hi*lo, so the result
// matches fp32 arithmetic to ~2^-16.  Q, K and V tiles sit in shared memory in the
// K-major 128-byte-swizzled layout (V is read MN-major by the PV product); P is written
// by the softmax warps in the same layout.  The running max is only raised (and O
// rescaled) when a row's maximum grows by more than a factor ~e^8 (keeping P, l and O
// finite in fp32); the final normalisation uses the same max, so the result is exact.
// Scores and maxima are kept in base-2 units (scaled by log2 e).
//
// A tile's chain (QK product, softmax, PV product and the barriers between them) is
// longer than its K and V take to stream in, so the even and the odd tiles of a CTA are
// two independent softmax streams: each has its own four warps, S accumulator, P buffer,
// running max and sum, and O accumulator, and nothing passes between them until the end.
//
// What bounds it (GB300, split planes, 4 splits of 32 heads): at a 16384-row context the K
// and V stream (85.2 us, 6.3 TB/s), at a 1000-row one the latency of the prologue and of the
// merge (64 queries 13.9 us, of which about 9 do not depend on the context).
//
// A tile of K or V takes 1.4-1.7 us to arrive under load and holds its slot for 0.5 us more
// while the tensor cores read it, so the bytes in flight decide: K and V share one ring of
// five 32 KB slots, filled in the order of use, which takes all of shared memory, and each
// product has a warp of its own that waits for nothing but its operands.  With two slots
// for K, two for V and one warp polling for both products: 90.2 us and 14.5, eight ragged
// sequences of 32-node trees 104.2 us (98.9), one query over 512 rows 10.1 (9.5), plain
// planes at 16384 rows 73.3 (63.9).  Before the two streams, with one lane issuing the MMAs
// (54 cycles each, operands moved to uniform registers): 128.4 and 18.1 us.  Also measured,
// at 16384 rows: an L2 prefetch three tiles ahead of the ring 108.9 us against 95.8
// without; QK products of 32 keys, which let a box keep a page's 16 rows together, 95.8
// against 91.5.
//
// Warps: 0..7 softmax + epilogue (warp w: stream w / 4, tensor-memory lanes 32 (w % 4)..,
// rows 16 (w % 4) .. + 15; a warp whose rows are all past nq only keeps the barriers
// going), 8 loads the KV tiles (TMA copies of 16-row page boxes, 128-byte swizzle applied
// by the copy engine), 9 issues the QK products, 10 the PV products (and owns the
// tensor-memory allocation).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "attention.cuh"
#include "common.cuh"
#include "kernels.h"

namespace chimera {
namespace {

constexpr int HD = 128;
constexpr int KT = 64;                      // keys per tile
constexpr int NQ = 64;                      // query rows (UMMA M)
constexpr int SOFT_WARPS = 8;               // softmax: warps w and w + 4 share rows, w / 4 = tile parity
constexpr int STREAM_WARPS = SOFT_WARPS / 2;
constexpr int LOAD_WARP = SOFT_WARPS, QK_WARP = LOAD_WARP + 1, PV_WARP = QK_WARP + 1;
constexpr int THREADS = (PV_WARP + 1) * 32;
constexpr int ATOM_ROWS64 = 64 * 128;       // bytes of one 64-row x 128-byte swizzle atom column
constexpr int GROUP = 8 * 128;              // 8 rows x 64 dims: one swizzle atom
constexpr int TILE64 = 2 * ATOM_ROWS64;     // 64 rows x 128 bf16 (two atoms): 16 KB
constexpr int PAGE_CACHE = 448;
constexpr float RESCALE_LOG2 = 11.5f;        // raise the running max when it grows by > 2^11.5 (~e^8)
constexpr uint32_t TMEM_COLS = 512;          // S[2] (64 cols each), O[2] (128 cols each)
constexpr uint32_t O_COL = 128;
constexpr int MAX_PARTS = 16;                // partials of a row: one or two per split
// The following linear's weights are requested into L2 by CTAs of at most this many tiles:
// at 4 a step gains 0.2-1.1 % (4096 wide, one to four sequences), at 5-6 it is even or
// loses 0.7 % and at 7-8 it loses 0.6-0.8 %, the requests competing with the KV loads.
constexpr int NEXT_W_TILES = 4, NEXT_W_CHUNK = 4096;
constexpr int MANY_NQ = 32;                  // more query rows than this take the MANY variant
constexpr int PREC = HD + 4;                 // partial record (o[128], m, l, pad)
constexpr int PART_FLOATS = (2 * MANY_NQ + 16) * PREC;  // the partial records of a CTA (<= NQ + 14 rows)
constexpr int TILE_BYTES = 224 * 1024;       // Q, P, K and V tiles (with plain planes: and 64 KB of staging)
static_assert((3 * PART_FLOATS + NQ * MAX_PARTS) * 4 <= TILE_BYTES, "partials and merge weights fit over the tiles");

// Byte offset of 16-byte chunk c (0..7) of row r inside a 128-byte-swizzled atom column.
__device__ __forceinline__ uint32_t swz(int r, int c) {
  return static_cast<uint32_t>((r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4));
}

// K-major (or, for the PV B operand, MN-major) 128-byte-swizzled smem descriptor.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((addr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}

// kind::f16 instruction descriptor: D fp32, A and B bf16, A K-major, B K-major or
// MN-major (b_mn), shape M x N.
__device__ __forceinline__ uint32_t idesc_f16(int m, int n, bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn ? (1u << 16) : 0u) | (static_cast<uint32_t>(n >> 3) << 17) |
         (static_cast<uint32_t>(m >> 4) << 24);
}

// 16x32bx2 access shape: lanes 0..15 of the warp read (write) TMEM lanes 0..15 of the
// warp's sub-partition at the addressed column, lanes 16..31 the same TMEM lanes at the
// column plus OFS; each of the 16 registers is the next column.
template <int OFS>
__device__ __forceinline__ void tmem_ld16x2(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x32bx2.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16], %17;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr), "n"(OFS));
}
template <int OFS>
__device__ __forceinline__ void tmem_st16x2(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x32bx2.x16.b32 [%0], %1, "
      "{%2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17};" ::"r"(taddr), "n"(OFS), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
// Wait for the issued TMEM loads; the registers are operands so that no use of them is
// scheduled before the wait.
__device__ __forceinline__ void tmem_wait_ld16(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
// Four 16-column pieces of a 128-column row: lanes 0..15 columns 0..63, 16..31 columns 64..127.
__device__ __forceinline__ void tmem_ld_row(uint32_t taddr, uint32_t (&r)[4][16]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) tmem_ld16x2<64>(taddr + 16 * c, r[c]);
#pragma unroll
  for (int c = 0; c < 4; ++c) tmem_wait_ld16(r[c]);
}
// 2^x on the special-function unit (inputs here are <= 0; results below 2^-126 flush to 0)
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Bulk request of `bytes` (a multiple of 16) at p into L2.
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void fence_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

// Kernel arguments: the tensor map of the pool viewed as [8-row group][plane][dim half][8
// rows][64 dims] (box: the planes of K, or of V, of one page) and the attention parameters.
struct TcArgs {
  CUtensorMap kv_map;
  AttnParams p;
};

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// (a, b) -> hi pair, lo pair (lo = rounding residual of hi)
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  const float2 hf = __bfloat1622float2(h);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = pack_bf16x2(a - hf.x, b - hf.y);
}

// Two-term bf16 split of four values: hi (4 x bf16) and lo = the rounding residual.
__device__ __forceinline__ void split4(float4 v, uint2& hi, uint2& lo) {
  split_pair(v.x, v.y, hi.x, lo.x);
  split_pair(v.z, v.w, hi.y, lo.y);
}

// Under the M = 64 data-path layout, query rows 16q .. 16q + 15 sit in TMEM lanes 0..15 of
// sub-partition q (warp w reaches sub-partition w % 4).


// MANY: more than MANY_NQ query rows.  Their rows and the local tile's are staged through
// shared memory, and a CTA merges its two streams before it sends them; with fewer rows
// each of these steps adds more latency than it saves (one query 9.9 us without, 10.6
// with them; 64 queries 15.7 and 14.5; two-slot rings), and both paths in one kernel cost each other
// (64 queries 15.3).
template <bool SPLIT, bool MANY>
__global__ void __launch_bounds__(THREADS, 1) attn_tc_kernel(const __grid_constant__ TcArgs args) {
  const AttnParams& p = args.p;
  constexpr int NP = SPLIT ? 4 : 2;
  constexpr int KP = NP / 2;                 // planes of K (and of V): hi (, lo)
  constexpr int SLOTS = SPLIT ? 5 : 6;       // ring of K and V tiles
  constexpr int HALF_BYTES = KP * TILE64;   // one slot, a tile of K or of V:
  // [page][8-row group][plane][dim half][8 rows][128 B]: one box per page, and the groups of
  // a plane and dim half lie at one stride (ROW_STRIDE) over the whole tile, as the
  // descriptors need
  constexpr int ROW_STRIDE = 2 * KP * GROUP;
  constexpr int PAGE_BYTES = 2 * ROW_STRIDE;
  constexpr int PLANE_STRIDE = 2 * GROUP;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* q_hi = smem;                     // 64 x 128 (two atoms)
  uint8_t* q_lo = q_hi + TILE64;
  uint8_t* p_buf = q_lo + TILE64;           // [2 buffers][hi, lo] 64 x 64 (one atom each, 8 KB)
  uint8_t* ring = p_buf + 4 * (NQ * 128);   // [SLOTS][KP planes] 64 keys x 128 dims
  // fp32 rows of the projections on their way into the tiles: q, and the local tile's k and v
  float* q_st = reinterpret_cast<float*>(p_buf);
  float* k_st = reinterpret_cast<float*>(ring + (SPLIT ? 3 : SLOTS) * HALF_BYTES);
  float* v_st = k_st + NQ * HD;
  static_assert(SPLIT || (SLOTS * HALF_BYTES + 8 * TILE64 <= TILE_BYTES), "staging behind the ring");
  float* part = reinterpret_cast<float*>(smem);  // partial records, over the tiles after the loop
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + TILE_BYTES);
  uint64_t* full = bars;             // [SLOTS] count 1 + transaction bytes (TMA)
  uint64_t* empty = bars + 6;        // [SLOTS] tcgen05.commit after the product
  uint64_t* s_full = bars + 12;      // [2] tcgen05.commit
  uint64_t* s_free = bars + 14;      // [2] count 4 (the stream's softmax warps)
  uint64_t* p_full = bars + 16;      // [2] count 4
  uint64_t* pv_done = bars + 18;     // [2] tcgen05.commit
  uint64_t* o_done = bars + 20;      // count 2: tcgen05.commit of the QK and of the PV warp
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 21);
  int* s_abort = reinterpret_cast<int*>(tmem_slot + 1);
  int* s_next = s_abort + 1;         // ring position after the last one requested
  int* s_pages = s_abort + 2;        // [PAGE_CACHE]
  int* s_lpages = s_pages + PAGE_CACHE;  // [8] pages of the local rows
  volatile int* abort = s_abort;

  const int s = blockIdx.x, h = blockIdx.y;
  const int S = gridDim.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  bf16* pool = static_cast<bf16*>(const_cast<void*>(p.pool)) + static_cast<size_t>(p.layer) * p.pool_layer_stride;

  if (threadIdx.x == 0) {
    for (int i = 0; i < SLOTS; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s_full[i], 1);
      mbar_init(&s_free[i], STREAM_WARPS);
      mbar_init(&p_full[i], STREAM_WARPS);
      mbar_init(&pv_done[i], 1);
    }
    mbar_init(o_done, 2);
    *s_abort = 0;
    mbar_fence_init();
  }
  if (warp == PV_WARP) tmem_alloc(tmem_slot, TMEM_COLS);

  if (!p.prewait_kv) pdl_wait();
  const QueryBlock qb(p, blockIdx.z);  // (early reads: n_ctx; the device counts are used by prompt chunks only)
  const int b = qb.b, nctx = qb.nctx;
  // Local mode (fused projections, local rows starting at row 0: verify, prefill, plain
  // decoding, the draft's first sub-step): every local row is written by this launch,
  // so the local rows form one extra tile that the CTA owning it builds in shared
  // memory from the projections (no round trip through the pool); the committed rows
  // are tiles of the pool.  The local tile is the last of the split's virtual tiles
  // (so it goes to the CTA with the fewest committed tiles) and that CTA's first tile
  // (its slots are free at start).  Otherwise the tiles cover slots [0, nctx + n_local).
  const bool lmode = p.qkv != nullptr && p.q_local0 == 0;
  // tiles of the pool (a block of prompt rows past its sequence's last row has none)
  const int ntiles = lmode              ? (nctx + KT - 1) / KT
                     : p.q_blocks <= 1 ? (nctx + p.n_local + KT - 1) / KT
                     : qb.nq > 0       ? (nctx + qb.nloc + KT - 1) / KT
                                       : 0;
  const int T = ntiles + (lmode ? 1 : 0);
  const int tps = (T + S - 1) / S;
  const int v0 = min(T, s * tps), v1 = min(T, v0 + tps);
  const int hl = (lmode && v0 < v1 && v1 == T) ? 1 : 0;  // this CTA holds the local tile (index 0)
  const int t0 = v0;                                    // pool tiles [t0, t1), tile indices hl ..
  const int t1 = hl ? T - 1 : v1;
  const int nt = hl + (t1 - t0);
  const bool cached = (t1 - t0) * 4 <= PAGE_CACHE;
  if (cached) {
    const int np = min((t1 - t0) * 4, p.max_pages - t0 * 4);
    for (int i = threadIdx.x; i < np; i += blockDim.x) s_pages[i] = p.page_table[b * p.max_pages + t0 * 4 + i];
  }
  if (hl && threadIdx.x >= THREADS - 5) {
    const int i = threadIdx.x - (THREADS - 5);
    s_lpages[i] = (nctx >> 4) + i < p.max_pages ? p.page_table[b * p.max_pages + (nctx >> 4) + i] : 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // ---- KV loads (the loader warp, all lanes together).  The tiles go through the ring in
  // the order in which they are consumed, K0 K1 V0 K2 V1 K3 ...: position 0 is K of tile 0,
  // an odd position 2 i - 1 K of tile i, an even one 2 i + 2 V of tile i (the one that K of
  // tile nt would have stays empty).  Tile index i: the local tile (i = 0 when hl; not
  // loaded) or pool tile t0 + i - hl.  A page's planes and dim halves are one box per lane
  // (4 or 8 KB); pages at or past kend are requested out of bounds (zero fill). ----
  auto k_pos = [](int i) { return i > 0 ? 2 * i - 1 : 0; };
  auto v_pos = [](int i) { return 2 * i + 2; };
  const int groups_per_layer = static_cast<int>(p.pool_layer_stride / (16 * HD));  // 16-row planes
  auto tile_of = [&](int pos, bool& is_v) {
    is_v = pos > 0 && (pos & 1) == 0;
    return is_v ? (pos - 2) >> 1 : (pos + 1) >> 1;
  };
  auto box_of = [&](int pos, int end) {  // the box this lane requests
    bool is_v;
    const int t = t0 + tile_of(pos, is_v) - hl;
    int y = static_cast<int>(p.pool_rows / 16);  // out of bounds
    if (lane < 4 && t * KT + lane * 16 < end) {
      const int page = cached ? s_pages[(t - t0) * 4 + lane] : p.page_table[b * p.max_pages + t * 4 + lane];
      y = p.layer * groups_per_layer + (page * p.H + h) * NP + (is_v ? KP : 0);
    }
    return y;
  };
  auto request = [&](int slot, int y) {
    if (lane == 0) mbar_arrive_expect_tx(&full[slot], static_cast<uint32_t>(HALF_BYTES));
    __syncwarp();
    if (lane < 4) tma_load_5d(ring + slot * HALF_BYTES + lane * PAGE_BYTES, &args.kv_map, 0, 0, 0, y, 0, &full[slot]);
  };
  // a tile to load (or nothing at this position)
  auto wanted = [&](int pos) {
    bool is_v;
    const int i = tile_of(pos, is_v);
    return i < nt && !(hl && i == 0);
  };

  int next_pos = 0;  // positions requested before the dependency wait
  if (p.prewait_kv) {
    if (warp == LOAD_WARP) {
      if (lane == 0) prefetch_tensormap(&args.kv_map);
      __syncwarp();
      // pool tiles whose rows are all committed (local mode: rows at or past nctx are
      // masked; the pool holds finite values there, the pools being cleared at set-up)
      // (with many rows and split planes the local tile's owner stages k and v in slots 3 and 4 first)
      const int lim = SPLIT && MANY && hl ? 3 : SLOTS;
      for (; next_pos < lim; ++next_pos) {
        bool is_v;
        if (!wanted(next_pos)) continue;
        if (!lmode && (t0 + tile_of(next_pos, is_v) + 1) * KT > nctx) break;
        request(next_pos, box_of(next_pos, nctx));
      }
    }
    __syncwarp();
  }
  // The angles of this thread's two query items (item it: row it / 8, dims 8j .. and 64 + 8j
  // .., j = it % 8): neither they nor the positions depend on the kernel before, and their
  // two dependent loads, after the wait, outlast the copy of the rows (1.2 us of 2.8)
  constexpr int ITEMS = MANY ? 2 : 1;
  float2 cs[ITEMS][8];
  if (p.qkv) {
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      const int it = threadIdx.x + k * THREADS, r = it >> 3;
      if (r < p.nq) {
        const int pos = min(max(nctx + p.pos_base + (p.pos_off ? p.pos_off[r] : r), 0), p.max_pos - 1);
        const float4* tab = reinterpret_cast<const float4*>(p.rope + static_cast<size_t>(pos) * (HD / 2) + 8 * (it & 7));
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float4 t = tab[e];
          cs[k][2 * e] = make_float2(t.x, t.y);
          cs[k][2 * e + 1] = make_float2(t.z, t.w);
        }
      }
    }
  }

  if (p.prewait_kv) pdl_wait();
  pdl_trigger();

  const int nloc = p.q_blocks > 1 ? qb.nloc : min(p.n_local_dev ? p.n_local_dev[b] : p.n_local, p.n_local);
  const int nq = p.q_blocks > 1 ? qb.nq : p.nq_dev ? p.nq_dev[b] : p.nq;
  const int total = nctx + nloc;
  const int dm = p.H * HD;

  const float* q_src = p.qkv ? p.qkv + static_cast<size_t>(qb.row0) * p.ldqkv + h * HD
                             : p.q + static_cast<size_t>(qb.row0) * p.ldq + h * HD;
  const float* k_src = hl ? p.qkv + static_cast<size_t>(qb.row0) * p.ldqkv + dm + h * HD : nullptr;
  const float* v_src = hl ? k_src + dm : nullptr;
  int q_ld = p.qkv ? p.ldqkv : p.ldq, kv_ld = p.ldqkv;
  if constexpr (MANY) {
    // fp32 rows into shared memory, every copy of a thread in flight at once (loaded item by
    // item, q took 2.8 us and the local tile another 4.3)
    auto stage_rows = [&](float* dst, const float* src, int ld) {
      for (int it = threadIdx.x; it < nq * (HD / 4); it += THREADS)
        cp_async16(dst + it * 4, src + static_cast<size_t>(it / (HD / 4)) * ld + it % (HD / 4) * 4);
    };
    stage_rows(q_st, q_src, q_ld);
    if (hl) {
      stage_rows(k_st, k_src, kv_ld);
      stage_rows(v_st, v_src, kv_ld);
    }
    q_src = q_st;
    k_src = k_st;
    v_src = v_st;
    q_ld = kv_ld = HD;
    cp_async_wait_all();
    __syncthreads();
  }

  // ---- queries: rotate (fused mode), split, write the swizzled Q tiles ----
  static_assert(NQ * 8 <= 2 * THREADS && MANY_NQ * 8 <= THREADS, "two items per thread, or one");
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int it = threadIdx.x + k * THREADS;
    if (it >= NQ * 8) break;
    const int r = it >> 3, j = it & 7;
    float lo_half[8], hi_half[8];
    if (k < ITEMS && r < nq) {  // (up to MANY_NQ rows: a thread's second item is past them)
      const float* src = q_src + static_cast<size_t>(r) * q_ld + 8 * j;
      const float4 a0 = *reinterpret_cast<const float4*>(src), a1 = *reinterpret_cast<const float4*>(src + 4);
      const float4 b0 = *reinterpret_cast<const float4*>(src + HD / 2),
                   b1 = *reinterpret_cast<const float4*>(src + HD / 2 + 4);
      const float x1[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float x2[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
      if (p.qkv) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          lo_half[e] = x1[e] * cs[k < ITEMS ? k : 0][e].x - x2[e] * cs[k < ITEMS ? k : 0][e].y;
          hi_half[e] = x2[e] * cs[k < ITEMS ? k : 0][e].x + x1[e] * cs[k < ITEMS ? k : 0][e].y;
        }
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          lo_half[e] = x1[e];
          hi_half[e] = x2[e];
        }
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) lo_half[e] = hi_half[e] = 0.f;
    }
    uint4 h0, l0, h1, l1;
    split_pair(lo_half[0], lo_half[1], h0.x, l0.x);
    split_pair(lo_half[2], lo_half[3], h0.y, l0.y);
    split_pair(lo_half[4], lo_half[5], h0.z, l0.z);
    split_pair(lo_half[6], lo_half[7], h0.w, l0.w);
    split_pair(hi_half[0], hi_half[1], h1.x, l1.x);
    split_pair(hi_half[2], hi_half[3], h1.y, l1.y);
    split_pair(hi_half[4], hi_half[5], h1.z, l1.z);
    split_pair(hi_half[6], hi_half[7], h1.w, l1.w);
    *reinterpret_cast<uint4*>(q_hi + swz(r, j)) = h0;
    *reinterpret_cast<uint4*>(q_lo + swz(r, j)) = l0;
    *reinterpret_cast<uint4*>(q_hi + ATOM_ROWS64 + swz(r, j)) = h1;
    *reinterpret_cast<uint4*>(q_lo + ATOM_ROWS64 + swz(r, j)) = l1;
  }
  // the P tiles' rows are all rewritten every tile; nothing else to clear

  // ---- local mode: the owner of the local tile rotates k, writes k and v of the fresh
  // rows to the pool (for later steps) and into the slots of its first K and V tile; rows past the
  // fresh ones are zero there ----
  if (hl) {
    for (int it = threadIdx.x; it < KT * 16; it += THREADS) {
      const int i = it >> 4, j = (it & 15) * 4;  // local row, pair index j .. j + 3 of the first half
      uint2 kh0 = make_uint2(0u, 0u), kl0 = kh0, kh1 = kh0, kl1 = kh0, vh0 = kh0, vl0 = kh0, vh1 = kh0, vl1 = kh0;
      if (i < nq) {
        const int slot = nctx + i;
        const int pos = nctx + p.pos_base + (p.pos_off ? p.pos_off[i] : i);
        if (pos < 0 || pos >= p.max_pos || (slot >> 4) >= p.max_pages) {
          if (p.err) atomicOr(p.err, ERR_CAPACITY);
        } else {
          const size_t o = static_cast<size_t>(i) * kv_ld + j;
          const float4 k1 = *reinterpret_cast<const float4*>(k_src + o);
          const float4 k2 = *reinterpret_cast<const float4*>(k_src + o + HD / 2);
          const float4 v1 = *reinterpret_cast<const float4*>(v_src + o);
          const float4 v2 = *reinterpret_cast<const float4*>(v_src + o + HD / 2);
          const float2* tab = p.rope + static_cast<size_t>(pos) * (HD / 2) + j;
          const float4 cs01 = *reinterpret_cast<const float4*>(tab);
          const float4 cs23 = *reinterpret_cast<const float4*>(tab + 2);
          const float4 c = make_float4(cs01.x, cs01.z, cs23.x, cs23.z);
          const float4 sn = make_float4(cs01.y, cs01.w, cs23.y, cs23.w);
          split4(rot_lo(k1, k2, c, sn), kh0, kl0);
          split4(rot_hi(k1, k2, c, sn), kh1, kl1);
          split4(v1, vh0, vl0);
          split4(v2, vh1, vl1);
          const int page = s_lpages[(slot >> 4) - (nctx >> 4)];
          bf16* base = pool + (static_cast<size_t>(page) * p.H + h) * NP * 16 * HD + (slot & 15) * HD + j;
          constexpr size_t plane = 16 * HD;
          if (SPLIT) {
            *reinterpret_cast<uint2*>(base) = kh0;
            *reinterpret_cast<uint2*>(base + plane) = kl0;
            *reinterpret_cast<uint2*>(base + HD / 2) = kh1;
            *reinterpret_cast<uint2*>(base + plane + HD / 2) = kl1;
            *reinterpret_cast<uint2*>(base + 2 * plane) = vh0;
            *reinterpret_cast<uint2*>(base + 3 * plane) = vl0;
            *reinterpret_cast<uint2*>(base + 2 * plane + HD / 2) = vh1;
            *reinterpret_cast<uint2*>(base + 3 * plane + HD / 2) = vl1;
          } else {
            *reinterpret_cast<uint2*>(base) = kh0;
            *reinterpret_cast<uint2*>(base + HD / 2) = kh1;
            *reinterpret_cast<uint2*>(base + plane) = vh0;
            *reinterpret_cast<uint2*>(base + plane + HD / 2) = vh1;
          }
        }
      }
      // row i, dims j .. j + 3 (half 0) and 64 + j .. (half 1): half of chunk j / 8
      const uint32_t o0 = (i >> 3) * ROW_STRIDE + swz(i & 7, j >> 3) + ((j & 7) << 1);
      const uint32_t o1 = GROUP + o0;
      uint8_t* kt = ring + k_pos(0) * HALF_BYTES;
      uint8_t* vt = ring + v_pos(0) * HALF_BYTES;
      *reinterpret_cast<uint2*>(kt + o0) = kh0;
      *reinterpret_cast<uint2*>(kt + o1) = kh1;
      *reinterpret_cast<uint2*>(vt + o0) = vh0;
      *reinterpret_cast<uint2*>(vt + o1) = vh1;
      if (SPLIT) {
        *reinterpret_cast<uint2*>(kt + PLANE_STRIDE + o0) = kl0;
        *reinterpret_cast<uint2*>(kt + PLANE_STRIDE + o1) = kl1;
        *reinterpret_cast<uint2*>(vt + PLANE_STRIDE + o0) = vl0;
        *reinterpret_cast<uint2*>(vt + PLANE_STRIDE + o1) = vl1;
      }
    }
  }
  // ---- otherwise: fresh local rows of this CTA's key range: rotate k, write k and v to
  // the pool, read back by TMA ----
  if (p.qkv && !lmode) {
    const int fresh0 = nctx + p.q_local0;
    const int f0 = max(0, t0 * KT - fresh0), f1 = min(nq, t1 * KT - fresh0);
    for (int it = threadIdx.x; it < (f1 - f0) * 16; it += blockDim.x) {
      const int i = f0 + (it >> 4), j = (it & 15) * 4;
      const int slot = fresh0 + i;
      const int pos = nctx + p.pos_base + (p.pos_off ? p.pos_off[i] : i);
      if (pos < 0 || pos >= p.max_pos || (slot >> 4) >= p.max_pages) {
        if (p.err) atomicOr(p.err, ERR_CAPACITY);
        continue;
      }
      const int page = p.page_table[b * p.max_pages + (slot >> 4)];
      const float* src = p.qkv + static_cast<size_t>(b * p.q_rows + i) * p.ldqkv + h * HD + j;
      const float4 k1 = *reinterpret_cast<const float4*>(src + dm);
      const float4 k2 = *reinterpret_cast<const float4*>(src + dm + HD / 2);
      const float4 v1 = *reinterpret_cast<const float4*>(src + 2 * dm);
      const float4 v2 = *reinterpret_cast<const float4*>(src + 2 * dm + HD / 2);
      const float2* tab = p.rope + static_cast<size_t>(pos) * (HD / 2) + j;
      const float4 cs01 = *reinterpret_cast<const float4*>(tab);
      const float4 cs23 = *reinterpret_cast<const float4*>(tab + 2);
      const float4 c = make_float4(cs01.x, cs01.z, cs23.x, cs23.z);
      const float4 sn = make_float4(cs01.y, cs01.w, cs23.y, cs23.w);
      const float4 ka = rot_lo(k1, k2, c, sn), kb = rot_hi(k1, k2, c, sn);
      bf16* base = pool + (static_cast<size_t>(page) * p.H + h) * NP * 16 * HD + (slot & 15) * HD + j;
      constexpr size_t plane = 16 * HD;
      if (SPLIT) {
        store4_split(base, base + plane, ka);
        store4_split(base + HD / 2, base + plane + HD / 2, kb);
        store4_split(base + 2 * plane, base + 3 * plane, v1);
        store4_split(base + 2 * plane + HD / 2, base + 3 * plane + HD / 2, v2);
      } else {
        store4<bf16>(base, ka);
        store4<bf16>(base + HD / 2, kb);
        store4<bf16>(base + plane, v1);
        store4<bf16>(base + plane + HD / 2, v2);
      }
    }
    fence_async_global();  // the rows are read back by TMA (async proxy)
  }
  fence_async_smem();  // the Q tiles (and the local K, V tile) are read by the tensor cores (async proxy)
  __threadfence_block();
  __syncthreads();
  if (hl && threadIdx.x == 0) {  // the local tile is in place: the slots of K and V of tile 0 are full
    mbar_arrive(&full[k_pos(0)]);
    mbar_arrive(&full[v_pos(0)]);
  }

  // softmax state of this lane's row (softmax warps)
  const int strm = (warp >> 2) & 1, quad = warp & 3, sub = lane >> 4;
  const int r = quad * 16 + (lane & 15);
  const uint32_t tlane = static_cast<uint32_t>(quad * 32) << 16;
  float m_used = -INFINITY, l = 0.f;

  if (warp == LOAD_WARP) {
    // ---------------- KV loader (the whole warp) ----------------
    if (!p.prewait_kv && lane == 0) prefetch_tensormap(&args.kv_map);
    __syncwarp();
    const int end = lmode ? nctx : total;
    const int last_pos = nt > 0 ? v_pos(nt - 1) : -1;
    int slot = next_pos % SLOTS;
    uint32_t phase = static_cast<uint32_t>(next_pos / SLOTS) & 1u;
    for (; next_pos <= last_pos; ++next_pos) {
      if (wanted(next_pos)) {
        const int y = box_of(next_pos, end);
        if (next_pos >= SLOTS && !mbar_wait_warp(&empty[slot], phase ^ 1u, abort)) break;
        request(slot, y);
      }
      if (++slot == SLOTS) {
        slot = 0;
        phase ^= 1u;
      }
    }
    if (p.next_w && nt <= NEXT_W_TILES) {  // (all of this CTA's KV is requested)
      const long long ctas = static_cast<long long>(gridDim.x) * gridDim.y * gridDim.z;
      const long long cta = (static_cast<long long>(blockIdx.z) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
      const char* w = static_cast<const char*>(p.next_w);
      for (long long o = (cta * 32 + lane) * NEXT_W_CHUNK; o < p.next_w_bytes; o += ctas * 32 * NEXT_W_CHUNK)
        prefetch_l2(w + o, static_cast<uint32_t>(min(static_cast<long long>(NEXT_W_CHUNK), p.next_w_bytes - o)));
      __syncwarp();
    }
    if (lane == 0) *s_next = next_pos;
    __syncwarp();
  } else if (warp == QK_WARP || warp == PV_WARP) {
    // ---------------- MMA issuers (a warp for each product, one elected lane issues) ----------------
    const int ntu = __shfl_sync(0xffffffffu, nt, 0);
    if (ntu > 0) {
      const uint32_t elected = elect_one();
      constexpr uint64_t LO_OFS = PLANE_STRIDE >> 4;  // hi plane -> lo plane
      // descriptors are made once; advancing an operand by b bytes adds b >> 4 to its
      // start-address field (all operands lie below 256 KB of shared memory)
      if (warp == QK_WARP) {  // S_i = Q K_i^T into S buffer i & 1, once the softmax has read S_(i - 2)
        const uint32_t id_qk = idesc_f16(NQ, KT, false);
        const uint64_t dq_h = desc_sw128(smem_u32(q_hi), 16, 1024), dq_l = desc_sw128(smem_u32(q_lo), 16, 1024);
        const uint64_t dk = desc_sw128(smem_u32(ring), 16, ROW_STRIDE);
        for (int i = 0; i < ntu; ++i) {
          const int pos = k_pos(i), slot = pos % SLOTS, st = i & 1;
          if (i >= 2 && !mbar_wait_warp(&s_free[st], ((i - 2) >> 1) & 1, abort)) break;
          // (K of tile i may follow V of tile i - 4 in its slot, whose load need not have landed
          // yet: a wait two phases ahead would pass on the parity of the phase before)
          if (pos >= SLOTS && !mbar_wait_warp(&empty[slot], (pos / SLOTS - 1) & 1, abort)) break;
          if (!mbar_wait_warp(&full[slot], (pos / SLOTS) & 1, abort)) break;
          tc_fence_after();
          const uint32_t s_t = tmem + st * 64;
          const uint64_t b0 = dk + static_cast<uint64_t>(slot * (HALF_BYTES >> 4));
#pragma unroll
          for (int ks = 0; ks < HD / 16; ++ks) {
            const uint64_t a_ofs = static_cast<uint64_t>(((ks >> 2) * ATOM_ROWS64 + (ks & 3) * 32) >> 4);
            const uint64_t b_h = b0 + static_cast<uint64_t>(((ks >> 2) * GROUP + (ks & 3) * 32) >> 4);
            tc_mma_bf16(s_t, dq_h + a_ofs, b_h, id_qk, ks > 0 ? 1u : 0u, elected);
            tc_mma_bf16(s_t, dq_l + a_ofs, b_h, id_qk, 1u, elected);
            if (SPLIT) tc_mma_bf16(s_t, dq_h + a_ofs, b_h + LO_OFS, id_qk, 1u, elected);
          }
          tc_commit(&empty[slot], elected);
          tc_commit(&s_full[st], elected);
        }
      } else {  // O[i & 1] += P_i V_i
        const uint32_t id_pv = idesc_f16(NQ, HD, true);
        const uint64_t dp = desc_sw128(smem_u32(p_buf), 16, 1024);
        // V as MN-major B: 64-dim atoms GROUP apart (leading), 8-key groups ROW_STRIDE apart
        const uint64_t dv = desc_sw128(smem_u32(ring), GROUP, ROW_STRIDE);
        constexpr uint64_t P_LO_OFS = (NQ * 128) >> 4;  // P hi -> P lo (8 KB)
        for (int i = 0; i < ntu; ++i) {
          const int pos = v_pos(i), slot = pos % SLOTS, st = i & 1;
          if (!mbar_wait_warp(&full[slot], (pos / SLOTS) & 1, abort)) break;
          if (!mbar_wait_warp(&p_full[st], (i >> 1) & 1, abort)) break;
          tc_fence_after();
          const uint32_t o_t = tmem + O_COL + st * 128;
          const uint64_t a0 = dp + static_cast<uint64_t>(st * (2 * NQ * 128 >> 4));
          const uint64_t b0 = dv + static_cast<uint64_t>(slot * (HALF_BYTES >> 4));
          uint32_t acc = i > 1 ? 1u : 0u;
#pragma unroll
          for (int ks = 0; ks < KT / 16; ++ks) {
            const uint64_t a_h = a0 + static_cast<uint64_t>(ks * 2);                   // 32 bytes per K step
            const uint64_t b_h = b0 + static_cast<uint64_t>(ks * (PAGE_BYTES >> 4));  // 16 keys: a page
            tc_mma_bf16(o_t, a_h, b_h, id_pv, acc, elected);
            acc = 1;
            tc_mma_bf16(o_t, a_h + P_LO_OFS, b_h, id_pv, 1u, elected);
            if (SPLIT) tc_mma_bf16(o_t, a_h, b_h + LO_OFS, id_pv, 1u, elected);
          }
          tc_commit(&empty[slot], elected);
          tc_commit(&pv_done[st], elected);
        }
      }
      tc_commit(o_done, elected);  // all MMAs issued by this lane, including any after an abort
      // tensor memory and the KV slots are released only after every MMA completed
      mbar_wait_plain(o_done, 0, 200000000ull);
    }
  } else {
    // ---------------- softmax (warps 0..7) ----------------
    // Warp w owns the 16 rows of TMEM sub-partition w % 4 in every second tile (w / 4: even
    // or odd); lanes l and l + 16 share row l % 16 and take 32 keys each (the 16x32bx2
    // access shape) and combine by a shuffle.
    const bool any = quad * 16 < nq;
    const bool live = r < nq;
    const unsigned long long anc = live ? p.anc[p.q_local0 + r] : 0ull;
    const float scale2 = p.scale * 1.4426950408889634f;  // softmax in base 2: exp(x) = 2^(x log2 e)
    uint8_t* ph = p_buf + (2 * strm) * (NQ * 128);
    uint8_t* pl = ph + NQ * 128;
    for (int i = strm; i < nt; i += 2) {
      const bool loc = hl && i == 0;
      const int t = t0 + i - hl;
      if (!__all_sync(0xffffffffu, mbar_wait(&s_full[strm], (i >> 1) & 1, abort))) break;
      tc_fence_after();
      float sv[32];
      if (any) {
        uint32_t ra[16], rb[16];
        tmem_ld16x2<32>(tmem + tlane + strm * 64, ra);
        tmem_ld16x2<32>(tmem + tlane + strm * 64 + 16, rb);
        tmem_wait_ld16(ra);
        tmem_wait_ld16(rb);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          sv[j] = __uint_as_float(ra[j]);
          sv[16 + j] = __uint_as_float(rb[j]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&s_free[strm]);
      // this stream's P buffer and O accumulator are used by the PV product of tile i - 2:
      // waited for when one of them is first written, after the arithmetic
      bool pv_ok = i < 2;
      auto wait_pv = [&] {
        if (!pv_ok) {
          pv_ok = __all_sync(0xffffffffu, mbar_wait(&pv_done[strm], ((i - 2) >> 1) & 1, abort));
          tc_fence_after();
        }
        return pv_ok;
      };
      uint4 hh[4], ll[4];
      if (any) {
        // visibility of this lane's 32 keys (bit j: key 32 sub + j of the tile): the local
        // tile's keys are local rows (ancestor mask), a pool tile's keys are slots 64 t ..
        uint32_t vbits = 0u;
        if (live) {
          unsigned long long vis;
          if (loc) {
            vis = anc & (nloc >= 64 ? ~0ull : ((1ull << nloc) - 1ull));
          } else {
            const int base = t * KT;
            const int nc = nctx - base, nv = total - base, off = base - nctx;
            const unsigned long long cm = nc >= 64 ? ~0ull : (nc <= 0 ? 0ull : ((1ull << nc) - 1ull));
            const unsigned long long lm =
                lmode ? 0ull : (off >= 0 ? (off < 64 ? (anc >> off) : 0ull) : (-off < 64 ? (anc << -off) : 0ull));
            const unsigned long long vm = nv >= 64 ? ~0ull : (nv <= 0 ? 0ull : ((1ull << nv) - 1ull));
            vis = (cm | lm) & vm;
          }
          vbits = static_cast<uint32_t>(vis >> (32 * sub));
        }
        if (__any_sync(0xffffffffu, vbits != 0xffffffffu)) {
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (!((vbits >> j) & 1u)) sv[j] = -INFINITY;
        }
        float t4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};  // four chains of maxima
#pragma unroll
        for (int j = 0; j < 32; ++j) t4[j & 3] = fmaxf(t4[j & 3], sv[j]);
        float tmax = fmaxf(fmaxf(t4[0], t4[1]), fmaxf(t4[2], t4[3]));
        tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 16)) * scale2;  // over the row's 64 keys
        // m moves only when the tile's maximum exceeds it by more than 2^RESCALE_LOG2; O then
        // holds products of earlier tiles exactly when m was already finite.  Both lanes of a
        // row decide alike.
        const bool raise = tmax > m_used + RESCALE_LOG2 || (m_used == -INFINITY && tmax > -INFINITY);
        const bool rescale = raise && m_used != -INFINITY;
        float corr = 1.f;
        if (raise) {
          corr = rescale ? exp2f(m_used - tmax) : 0.f;
          m_used = tmax;
        }
        if (__any_sync(0xffffffffu, rescale)) {  // factor 1 for rows that kept m
          if (!wait_pv()) break;
          const float f = rescale ? corr : 1.f;
          const uint32_t oa = tmem + tlane + O_COL + strm * 128;
          uint32_t rr[4][16];
          tmem_ld_row(oa, rr);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
#pragma unroll
            for (int j = 0; j < 16; ++j) rr[c][j] = __float_as_uint(__uint_as_float(rr[c][j]) * f);
            tmem_st16x2<64>(oa + 16 * c, rr[c]);
          }
          tmem_wait_st();
        }
        l *= corr;
        // P = 2^(S - m), two-term split into the swizzled P tile (this lane's 4 chunks of 8);
        // a row with no visible key yet has m = -inf and scores -inf: P = 0
        const float mm = m_used == -INFINITY ? 0.f : m_used;
        float l4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float e[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            e[j] = ex2_approx(fmaf(sv[8 * c + j], scale2, -mm));
            l4[j & 3] += e[j];
          }
          split_pair(e[0], e[1], hh[c].x, ll[c].x);
          split_pair(e[2], e[3], hh[c].y, ll[c].y);
          split_pair(e[4], e[5], hh[c].z, ll[c].z);
          split_pair(e[6], e[7], hh[c].w, ll[c].w);
        }
        l += (l4[0] + l4[1]) + (l4[2] + l4[3]);
      }
      if (!wait_pv()) break;
      if (any) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          *reinterpret_cast<uint4*>(ph + swz(r, 4 * sub + c)) = hh[c];
          *reinterpret_cast<uint4*>(pl + swz(r, 4 * sub + c)) = ll[c];
        }
        fence_async_smem();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_full[strm]);
    }
    l += __shfl_xor_sync(0xffffffffu, l, 16);  // the row's sum over the stream's tiles
  }

  // ---- epilogue: a CTA's partial rows (O, m, l) go to the cluster CTA that finishes them
  // (rows [r * ceil(nq / S), ...) belong to rank r) once every CTA of the cluster is past
  // its main loop; everything lies over the tiles.  Few rows: each stream pushes its own from
  // the registers.  Many: that is bound by the traffic (64 rows: 3.3 us), so the streams are
  // merged first, while the cluster gathers, and whole records are pushed (1.1 us). ----
  if (warp < SOFT_WARPS) {
    if (nt > 0) {
      mbar_wait(o_done, 0, abort);
      tc_fence_after();
    }
    __syncwarp();
  }
  __syncthreads();  // this CTA's tiles are idle: every load landed and every MMA completed
  if (*abort) {     // (but if some wait gave up: copies may still be in flight)
    if (warp == LOAD_WARP)
      for (int n = *s_next, j = max(0, n - SLOTS); j < n; ++j)
        if (wanted(j)) mbar_wait_plain(&full[j % SLOTS], (j / SLOTS) & 1, 200000000ull);
    __syncthreads();
  }
  __syncwarp();
  if (S > 1) cluster_arrive();
  const int rpc = (nq + S - 1) / S;
  constexpr int ps = MANY ? 1 : 2;              // partials per CTA
  const int blk = ps * rpc * PREC;            // what a CTA sends to an owner: [ps][rpc][PREC]
  float* recv = part + PART_FLOATS;           // [S] blocks
  float* other = recv + PART_FLOATS;          // [64][PREC] the odd tiles' rows
  float* s_w = other + PART_FLOATS;           // [rpc][MAX_PARTS] merge weights
  if (warp < SOFT_WARPS) {
    const bool mine = r < nq;
    const bool have = quad * 16 < nq && nt > strm && !*abort;
    const int owner = mine ? r / rpc : 0, orow = r - owner * rpc;
    uint32_t rr[4][16];
    if (have) tmem_ld_row(tmem + tlane + O_COL + strm * 128, rr);  // this lane's 64 columns
    auto piece = [&](int c, int j) {
      return make_float4(__uint_as_float(rr[c][j]), __uint_as_float(rr[c][j + 1]), __uint_as_float(rr[c][j + 2]),
                         __uint_as_float(rr[c][j + 3]));
    };
    __syncwarp();
    if constexpr (!MANY) {
      if (S > 1) cluster_wait();  // every CTA's tiles are idle
      if (mine) {
        const uint32_t slot = smem_u32(recv + s * blk + (strm * rpc + orow) * PREC);
        const uint32_t dst = S > 1 ? dsmem_addr(slot, owner) : slot;
        const bool keep = have && l > 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int j = 0; j < 16; j += 4)
            st_dsmem4(dst + static_cast<uint32_t>((64 * sub + 16 * c + j) * 4),
                      keep ? piece(c, j) : make_float4(0.f, 0.f, 0.f, 0.f));
        if (sub == 0)
          st_dsmem4(dst + HD * 4, make_float4(have ? m_used : -INFINITY, have ? l : 0.f, 0.f, 0.f));
      }
    } else {
      float* o1 = other + r * PREC;
      if (strm == 1 && have && mine) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int j = 0; j < 16; j += 4) *reinterpret_cast<float4*>(o1 + 64 * sub + 16 * c + j) = piece(c, j);
        if (sub == 0) {
          o1[HD] = m_used;
          o1[HD + 1] = l;
        }
      }
      named_bar(1 + quad, 64);  // the two warps of these rows
      if (strm == 0 && mine) {
        const bool have1 = nt > 1 && !*abort;
        const float m0 = have ? m_used : -INFINITY, l0 = have ? l : 0.f;
        const float m1 = have1 ? o1[HD] : -INFINITY, l1 = have1 ? o1[HD + 1] : 0.f;
        const float m = fmaxf(m0, m1);
        const float w0 = l0 > 0.f ? exp2f(m0 - m) : 0.f, w1 = l1 > 0.f ? exp2f(m1 - m) : 0.f;
        float* dst = (owner == s ? recv + s * blk : part + owner * blk) + orow * PREC;
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int j = 0; j < 16; j += 4) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (l0 > 0.f) {
              const float4 t = piece(c, j);
              v = make_float4(w0 * t.x, w0 * t.y, w0 * t.z, w0 * t.w);
            }
            if (l1 > 0.f) {
              const float4 t = *reinterpret_cast<const float4*>(o1 + 64 * sub + 16 * c + j);
              v.x += w1 * t.x; v.y += w1 * t.y; v.z += w1 * t.z; v.w += w1 * t.w;
            }
            *reinterpret_cast<float4*>(dst + 64 * sub + 16 * c + j) = v;
          }
        if (sub == 0) {
          dst[HD] = m;
          dst[HD + 1] = w0 * l0 + w1 * l1;
        }
      }
    }
  } else if (!MANY && S > 1) {
    cluster_wait();
  }
  tc_fence_before();
  __syncthreads();
  __syncwarp();
  if (MANY && S > 1) {
    cluster_wait();
    for (int it = threadIdx.x; it < nq * (PREC / 4); it += THREADS) {  // 512 contiguous bytes per warp
      const int row = it / (PREC / 4), c = it % (PREC / 4) * 4, owner = row / rpc;
      const int o = owner * blk + (row - owner * rpc) * PREC + c;
      if (owner != s)
        st_dsmem4(dsmem_addr(smem_u32(recv + o + (s - owner) * blk), owner), *reinterpret_cast<const float4*>(part + o));
    }
    __syncwarp();
  }
  if (S > 1) cluster_arrive();
  if (warp == PV_WARP) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
  if (threadIdx.x == 0 && *abort && p.err) atomicOr(p.err, ERR_TIMEOUT);
  __syncwarp();
  if (S > 1) cluster_wait();  // the peers' partials are in

  // ---- merge the partials of this CTA's rows (local shared memory) ----
  bf16* out = static_cast<bf16*>(p.out);
  bf16* out_lo = static_cast<bf16*>(p.out_lo);
  const int q0 = s * rpc, nrows = max(0, min(nq, q0 + rpc) - q0), parts = ps * S;
  constexpr int LPR = 8 * ps;  // lanes per row, one partial each
  for (int r0 = warp * (32 / LPR); r0 < nrows; r0 += 32 / LPR * (THREADS / 32)) {
    const int rl = r0 + lane / LPR, k = lane % LPR;
    const bool on = rl < nrows && k < parts;
    const float* rec = recv + (k * rpc + rl) * PREC;
    const float m = on ? rec[HD] : -INFINITY, ls = on ? rec[HD + 1] : 0.f;
    float M = m;
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    const float e = m == -INFINITY ? 0.f : exp2f(m - M);
    float L = e * ls;
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
    if (on) s_w[rl * MAX_PARTS + k] = L > 0.f ? e / L : 0.f;
  }
  __syncthreads();
  for (int it = threadIdx.x; it < nrows * (HD / 4); it += blockDim.x) {
    const int rl = it / (HD / 4), c = (it % (HD / 4)) * 4;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < LPR; ++k) {
      if (k < parts) {
        const float w = s_w[rl * MAX_PARTS + k];
        const float4 v = *reinterpret_cast<const float4*>(recv + (k * rpc + rl) * PREC + c);
        acc.x += w * v.x; acc.y += w * v.y; acc.z += w * v.z; acc.w += w * v.w;
      }
    }
    const size_t o_idx = static_cast<size_t>(qb.row0 + q0 + rl) * p.ldo + h * HD + c;
    store_act4(out, out_lo, o_idx, acc);
  }
}

constexpr size_t TC_SMEM = 1024 + TILE_BYTES + 22 * 8 + 16 + (PAGE_CACHE + 8) * 4;

// The dynamic shared memory limit is an attribute of the device that is current when it
// is set: raised once per device (and kernel variant), the return code checked.
constexpr int ATT_MAX_DEVICES = 64;
std::mutex g_att_attr_mu;
bool g_att_attr[4][ATT_MAX_DEVICES];

template <bool SPLIT, bool MANY>
cudaError_t tc_attr() {
  constexpr int variant = (SPLIT ? 2 : 0) + (MANY ? 1 : 0);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= ATT_MAX_DEVICES) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_att_attr_mu);
  if (!g_att_attr[variant][dev]) {
    e = cudaFuncSetAttribute(attn_tc_kernel<SPLIT, MANY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(TC_SMEM));
    if (e != cudaSuccess) return e;
    g_att_attr[variant][dev] = true;
  }
  return cudaSuccess;
}

template <bool SPLIT, bool MANY>
cudaError_t launch_tc(const AttnParams& p, cudaStream_t s) {
  cudaError_t ae = tc_attr<SPLIT, MANY>();
  if (ae != cudaSuccess) return ae;
  TcArgs args;
  memset(&args, 0, sizeof(args));
  args.p = p;
  const uint64_t dims[5] = {64, 8, 2, static_cast<uint64_t>(p.pool_rows / 16), 2};
  const uint64_t strides[4] = {HD * 2, 128, 16 * HD * 2, 8 * HD * 2};
  const uint32_t box[5] = {64, 8, 2, SPLIT ? 2u : 1u, 2};
  if (encode_5d_bf16(&args.kv_map, p.pool, dims, strides, box) != 0) return cudaErrorInvalidValue;
  cudaLaunchAttribute at[2];
  int na = 0;
  at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[na].val.programmaticStreamSerializationAllowed = 1;
  ++na;
  if (p.splits > 1) {
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = p.splits;
    at[na].val.clusterDim.y = 1;
    at[na].val.clusterDim.z = 1;
    ++na;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.splits, p.H, p.B * std::max(1, p.q_blocks));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = TC_SMEM;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = na;
  cudaLaunchKernelEx(&cfg, attn_tc_kernel<SPLIT, MANY>, args);
  return cudaGetLastError();
}

template <bool SPLIT>
int tc_splits(int BH, int want) {
  if (tc_attr<SPLIT, true>() != cudaSuccess) return 1;  // both row variants have the same footprint
  int S = std::max(1, std::min(8, want));
  for (; S > 1; --S) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = S;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S, BH, 1);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = TC_SMEM;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, attn_tc_kernel<SPLIT, true>, &cfg) == cudaSuccess && n >= BH) break;
    cudaGetLastError();
  }
  return S;
}

}  // namespace


cudaError_t attention_tc(const AttnParams& p, cudaStream_t s) {
  if (p.hd != HD || p.nq_max > NQ || p.n_local > 64 || p.splits < 1 || p.splits > 8) return cudaErrorInvalidValue;
  // the TMA row coordinate is a 32-bit integer; the pool base must be 16-byte aligned
  if (p.pool_rows < 16 || p.pool_rows >= (1ll << 31) || (reinterpret_cast<uintptr_t>(p.pool) & 15))
    return cudaErrorInvalidValue;
  if (p.planes != 2 && p.planes != 4) return cudaErrorInvalidValue;
  if (p.qkv && (!p.rope || !p.err || p.max_pos < 1 || (p.ldqkv & 3))) return cudaErrorInvalidValue;
  if (!p.qkv && (p.ldq & 3)) return cudaErrorInvalidValue;
  if (p.nq_max > MANY_NQ) return p.planes == 4 ? launch_tc<true, true>(p, s) : launch_tc<false, true>(p, s);
  return p.planes == 4 ? launch_tc<true, false>(p, s) : launch_tc<false, false>(p, s);
}

int attention_tc_splits(int planes, int BH, int want) {
  return planes == 4 ? tc_splits<true>(BH, want) : tc_splits<false>(BH, want);
}

}  // namespace chimera

// Causal (or bidirectional) grouped-query attention, Eq. 1, on the sm_103a
// tensor cores: two query tiles per CTA whose softmaxes take turns, so each
// tile's exponentials run while the tensor core works on the other tile.
//
// A work item is two tiles of 128 queries that read the same keys and values,
// so each K/V block is loaded once for both: two query heads of a KV group
// (an even number of heads per group), or two neighbouring query blocks of one
// head (an odd number; with the causal mask the first tile has fewer key
// blocks, and the last block of a sequence may have no partner).  Per key block
// j of 128 keys (causal: up to the diagonal):
//   S_x = Q_x K_j^T                      (tcgen05, M = 128, N = 128, K = hd)
//   softmax warps of tile x (one query row per thread, TMEM lane = row):
//     pass 1: the block's row maximum (masked keys excluded), log2 domain;
//       the running maximum m moves only when the block's exceeds it by more
//       than 2^8 (until then P entries may reach 256, exact in fp32 and in the
//       bf16 pair), and then O is rescaled in TMEM by 2^(m_old - m_new);
//     pass 2: P = 2^(s*scale - m) as a bf16 pair P_hi + P_lo (P_lo is the
//       rounding remainder, so P is carried to ~16 bits), written back over
//       the S columns it came from, and the running row sum l.
//   O_x += P_hi V_j + P_lo V_j           (A = P from TMEM, B = V straight from
//                                         the packed qkv rows, MN-major)
// O stays in TMEM across the key blocks; the epilogue divides by l, rounds to
// bf16 and writes the row normaliser lse2 = m + log2(l).
//
// Tensor-core order (one issuing thread; tcgen05.mma executes in issue order):
//   S_A(0) S_B(0) | PV_A(0) S_A(1) PV_B(0) S_B(1) | PV_A(1) S_A(2) PV_B(1) ...
// so tile A's softmax of block j+1 runs under PV_B(j) and S_B(j+1), and tile
// B's under PV_A(j+1) and S_A(j+2).  An item's last P V is followed by the next
// item's first S in the same way, and its epilogue runs under the next item's
// first P V (with heads of 64 dims O has two buffers per tile for that).
//
// What bounds it: on long sequences the MMA stream (24 MMAs per tile and key
// block, 16 of them P V), on short ones the chain softmax -> P V -> epilogue of
// an item and the fetches of code that runs only once or twice per CTA.  So 32-
// column chunks with no visible key are skipped (only their P is zeroed), MMAs
// cover the live keys alone, and the code has one copy of each part: two copies
// of the conversion (an unrolled pair of chunks, or masked and unmasked) cost
// 5-25% at one or two key blocks.  Measured before and after (causal, 32 heads
// over 8 groups): 4 x 2048 rows of 128 dims 201 -> 185 us, 64 x 256 of 64 dims
// 84 -> 77, 64 x 30 34 -> 25; 16 x 501, 16 heads without groups, no mask: 75
// (one tile per CTA and a transposed V) -> 52; 1 x 2048, 32 such heads of 128
// dims, causal: 121 -> 55.
//
// Roles (384 threads): warp 0 TMA producer (both Q tiles per item; K and V of
// every key block through a ring), warp 1 MMA issuer, warps 4-7 tile A's
// softmax and epilogue, warps 8-11 tile B's (warp w reads TMEM lanes
// 32*(w%4)..+31).  TMEM: S_A | O_A | S_B | O_B, 128 columns each.  Every wait
// is bounded; after a timeout every role skips its remaining work, copies in
// flight are drained, and TMEM is freed.
#include "common.cuh"
#include "kernels.h"

namespace zsaa {
namespace {

constexpr int PP_BM = 128;  // queries per tile
constexpr int PP_BN = 128;  // keys per block
constexpr int PP_THREADS = 384;
constexpr uint32_t PP_TMEM_COLS = 512;
constexpr float PP_RESCALE_LOG2 = 8.0f;  // lazy rescale threshold (factor 256)

template <int HD>
struct PpCfg {
  static constexpr int CH = HD / 64;                 // 64-dim (128-byte) chunks
  static constexpr int TILE = PP_BM * HD * 2;        // one Q tile, K block or V block
  static constexpr int STAGES = HD == 128 ? 2 : 4;   // K/V ring
  static constexpr int O_BUFS = 128 / HD;            // O accumulators per tile
  static constexpr size_t SMEM = 2 * static_cast<size_t>(TILE) + 2 * STAGES * static_cast<size_t>(TILE) + 256 + 1024;
};
static_assert(PpCfg<64>::SMEM <= 227 * 1024 && PpCfg<128>::SMEM <= 227 * 1024, "shared memory");

__host__ __device__ constexpr uint32_t s_col(int x) { return 256u * x; }
template <int HD>
__host__ __device__ constexpr uint32_t o_col(int x, uint32_t buf) {
  return 256u * x + 128u + HD * buf;
}

struct PpArgs {
  float* lse2;  // [B, Hq, N], log2 domain
  bf16* out;    // [B*N (or the packed rows), Hq*hd]
  int B, N, Hq, Hkv, n_qb, causal, total;
  int by_head;   // 1: the two tiles are neighbouring heads, 0: neighbouring query blocks of one head
  int wide_out;  // out allows 32-byte stores
  FastDiv inner, units, groups;  // items per query position, heads (or pairs) per group, groups
  const int* cu;  // packed sequences of different lengths: rows [cu[b], cu[b+1]); N = the longest
  float scale_log2;
  int* status;
};

struct PpItem {
  int b, g, row0, n;         // sequence, KV group, first row and length of the sequence
  int h[2], qb[2], nk[2];    // per tile: head, query block, key blocks (0: no such tile)
  int n_kb;                  // key blocks of the item
};

// Work item t, longest query blocks first; false when its sequence has no such queries.
__device__ __forceinline__ bool pp_item(int t, const PpArgs& a, PpItem& it) {
  int r, u;
  const int qp = (a.by_head ? a.n_qb : (a.n_qb + 1) / 2) - 1 - a.inner.div(t, r);
  r = a.units.div(r, u);
  it.b = a.groups.div(r, it.g);
  if (a.cu) {
    it.row0 = a.cu[it.b];
    it.n = a.cu[it.b + 1] - it.row0;
  } else {
    it.row0 = it.b * a.N;
    it.n = a.N;
  }
  const int h0 = it.g * (a.by_head ? 2 * a.units.d : a.units.d) + (a.by_head ? 2 * u : u);
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    it.h[x] = a.by_head ? h0 + x : h0;
    it.qb[x] = a.by_head ? qp : 2 * qp + x;
    const int keys = a.causal ? min(it.n, (it.qb[x] + 1) * PP_BM) : it.n;
    it.nk[x] = it.qb[x] * PP_BM < it.n ? (keys + PP_BN - 1) / PP_BN : 0;
  }
  it.n_kb = max(it.nk[0], it.nk[1]);
  return it.nk[0] > 0;  // tile 0's queries come first
}

// This CTA's items: numbered longest query blocks first and dealt to the CTAs
// in a snake order (0..G-1, then G-1..0, ...), so the causal triangle's long
// and short items even out across CTAs.  Advances r to the next live item;
// false once there is none.
__device__ __forceinline__ bool pp_next(int& r, const PpArgs& a, PpItem& it) {
  const int G = gridDim.x, i = blockIdx.x;
  while (true) {
    if (r * G >= a.total) return false;
    const int t = r * G + ((r & 1) ? G - 1 - i : i);
    ++r;
    if (t < a.total && pp_item(t, a, it)) return true;
  }
}

__device__ __forceinline__ float ex2_fast(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// max of three in one instruction (the rate of a two-operand maximum)
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}

// Shared-memory descriptor of an MN-major operand with the 128-byte swizzle:
// rows of 64 bf16 along N (128 B) for consecutive K, 8-row atoms 1024 B apart
// along K (stride byte offset), 64-element N chunks `chunk_bytes` apart
// (leading byte offset).
__device__ __forceinline__ uint64_t sdesc_sw128_mn(uint32_t saddr, uint32_t chunk_bytes) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((chunk_bytes >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>(1024 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}

// D[tmem] (+)= A[tmem] * B[smem]: A (M x K) read from tensor memory, lane =
// row, two bf16 per 32-bit column in K order (lower K in the low half).
__device__ __forceinline__ void tc_mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc,
                                               uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Warp-collective: lane i writes TMEM lane (base + i), 32 consecutive columns.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  tmem_st16(taddr, *reinterpret_cast<const uint32_t(*)[16]>(r));
  tmem_st16(taddr + 16, *reinterpret_cast<const uint32_t(*)[16]>(r + 16));
}


// The two products of a key block, issued by one thread.  Not inlined: a CTA
// with one or two short items runs this code cold, and its instruction fetches
// are then a good part of its time.
template <int HD>
__device__ __noinline__ void pp_issue_s(uint32_t qa, uint32_t ka, uint32_t d_tmem, int keys, uint64_t* done) {
  const uint32_t idesc = idesc_bf16_f32(PP_BM, (keys + 15) & ~15);  // the block's live keys
#pragma unroll
  for (int kk = 0; kk < HD / 16; ++kk)
    tc_mma_bf16(d_tmem, sdesc_sw128(qa + (kk / 4) * (PP_BM * 128) + (kk % 4) * 32),
                sdesc_sw128(ka + (kk / 4) * (PP_BN * 128) + (kk % 4) * 32), idesc, kk > 0 ? 1u : 0u);
  tc_commit(done);
}
// O (+)= P_hi V + P_lo V over the 16-key steps that hold a key.
template <int HD>
__device__ __noinline__ void pp_issue_pv(uint32_t va, uint32_t p_tmem, uint32_t o_tmem, bool first, int keys) {
  constexpr uint32_t idesc = idesc_bf16_f32(PP_BM, HD) | (1u << 16);  // B (V) MN-major
  // V's 64-dim chunks are PP_BN * 128 bytes apart; with one chunk (hd 64) the
  // stride is never used and is set to the 8-row atom stride, so the
  // descriptor addresses only the 16 keys of each MMA either way.
  constexpr uint32_t kVChunkStride = HD > 64 ? PP_BN * 128 : 1024;
  auto mma = [&](int part, int kk) {
    tc_mma_bf16_ts(o_tmem, p_tmem + 32 * (kk / 2) + 16 * part + 8 * (kk % 2),
                   sdesc_sw128_mn(va + kk * 16 * 128, kVChunkStride), idesc, (first && part == 0 && kk == 0) ? 0u : 1u);
  };
  if (keys == PP_BN) {  // (no test between the issues: they bound the long sequences)
#pragma unroll
    for (int part = 0; part < 2; ++part)
#pragma unroll
      for (int kk = 0; kk < PP_BN / 16; ++kk) mma(part, kk);
  } else {
#pragma unroll 2
    for (int i = 0; i < 2 * ((keys + 15) / 16); ++i) mma(i & 1, i >> 1);
  }
}

template <int HD>
__global__ void __launch_bounds__(PP_THREADS, 1)
    attn_pp_kernel(const __grid_constant__ CUtensorMap tm, const PpArgs a) {
  using C = PpCfg<HD>;
  constexpr int CH = C::CH, TILE = C::TILE, ST = C::STAGES, NB = C::O_BUFS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* sQ = smem;                   // [2 tiles]
  uint8_t* sK = sQ + 2 * TILE;          // [ST]
  uint8_t* sV = sK + ST * TILE;         // [ST]
  uint64_t* bars = reinterpret_cast<uint64_t*>(sV + ST * TILE);
  uint64_t* q_full = bars;              // [1]
  uint64_t* q_empty = bars + 1;         // [1]
  uint64_t* s_full = bars + 2;          // [2] per tile
  uint64_t* p_full = bars + 4;          // [2]
  uint64_t* o_full = bars + 6;          // [2][NB]
  uint64_t* o_empty = bars + 10;        // [2][NB]
  uint64_t* mma_done = bars + 14;       // [1]
  uint64_t* kv_full = bars + 15;        // [ST]
  uint64_t* kv_empty = bars + 15 + ST;  // [ST]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 15 + 2 * ST);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_trigger();
  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    mbar_init(q_empty, 1);
    for (int x = 0; x < 2; ++x) {
      mbar_init(&s_full[x], 1);
      mbar_init(&p_full[x], 4);
    }
    for (int i = 0; i < 2 * NB; ++i) {
      mbar_init(&o_full[i], 1);
      mbar_init(&o_empty[i], 4);
    }
    mbar_init(mma_done, 1);
    for (int i = 0; i < ST; ++i) {
      mbar_init(&kv_full[i], 1);
      mbar_init(&kv_empty[i], 1);
    }
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 0 && lane == 0) prefetch_tmap(&tm);
  if (warp == 1) tmem_alloc(tmem_slot, PP_TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      bool ok = true;
      uint32_t J = 0, items = 0, q_issued = 0;
      PpItem it;
      for (int r = 0; ok && pp_next(r, a, it); ++items) {
        if (!mbar_wait_ab(q_empty, (items & 1) ^ 1, a.status, abort_flag)) {
          ok = false;
          break;
        }
        ++q_issued;
        mbar_arrive_expect_tx(q_full, (it.nk[1] > 0 ? 2 : 1) * TILE);
        for (int x = 0; x < 2; ++x)
          if (it.nk[x] > 0)
            for (int c = 0; c < CH; ++c)
              tma_load_2d(sQ + x * TILE + c * (PP_BM * 128), &tm, it.h[x] * HD + c * 64,
                          it.row0 + it.qb[x] * PP_BM, q_full);
        for (int j = 0; j < it.n_kb; ++j, ++J) {
          const int st = J % ST;
          if (!mbar_wait_ab(&kv_empty[st], ((J / ST) & 1) ^ 1, a.status, abort_flag)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&kv_full[st], 2 * TILE);
          for (int c = 0; c < CH; ++c) {
            tma_load_2d(sK + st * TILE + c * (PP_BN * 128), &tm, (a.Hq + it.g) * HD + c * 64,
                        it.row0 + j * PP_BN, &kv_full[st]);
            tma_load_2d(sV + st * TILE + c * (PP_BN * 128), &tm, (a.Hq + a.Hkv + it.g) * HD + c * 64,
                        it.row0 + j * PP_BN, &kv_full[st]);
          }
        }
      }
      if (!ok) {  // let the copies already issued land before the CTA's memory goes away
        for (uint32_t k = J; k > 0 && k + ST > J; --k)
          mbar_wait(&kv_full[(k - 1) % ST], ((k - 1) / ST) & 1, nullptr);
        if (q_issued > 0) mbar_wait(q_full, (q_issued - 1) & 1, nullptr);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      bool ok = true;
      uint32_t J = 0, items = 0;  // key blocks before this item, items begun
      uint32_t n_p[2] = {0, 0}, n_o[2] = {0, 0};  // per tile: P blocks taken, items
      auto issue_s = [&](int x, int st, int keys) {  // S_x = Q_x K^T over the block's `keys` live keys
        pp_issue_s<HD>(smem_u32(sQ + x * TILE), smem_u32(sK + st * TILE), tmem + s_col(x), keys, &s_full[x]);
      };
      // The S of an item's first block are issued under the item before it, each
      // as soon as its tile's last P V is (s_left: S products of the item after
      // this one not issued yet).
      PpItem it, nx;
      int r = 0;
      bool have = pp_next(r, a, nx), begun = false;  // begun: nx's Q and first keys are there
      int s_left = have ? nx.nk[0] + nx.nk[1] : 0;
      auto first_s = [&](int x, uint32_t Jn) {
        if (!begun) {
          if (!mbar_wait_ab(q_full, items & 1, a.status, abort_flag) ||
              !mbar_wait_ab(&kv_full[Jn % ST], (Jn / ST) & 1, a.status, abort_flag)) {
            ok = false;
            return;
          }
          tc_fence_after();
          begun = true;
        }
        issue_s(x, Jn % ST, min(PP_BN, nx.n));
        if (--s_left == 0) tc_commit(q_empty);  // Q read for the last time
      };
      if (have) {
        first_s(0, 0);
        if (ok && nx.nk[1] > 0) first_s(1, 0);
      }
      while (have && ok) {
        it = nx;
        int left = s_left;  // this item's S products not issued yet
        have = pp_next(r, a, nx);
        s_left = have ? nx.nk[0] + nx.nk[1] : 0;
        begun = false;
        ++items;
        bool early[2] = {false, false};  // the next item's first S issued
        const uint32_t Jn = J + it.n_kb;
        for (int j = 0; j < it.n_kb && ok; ++j) {
          const uint32_t Jj = J + j;
          const int st = Jj % ST, st1 = (Jj + 1) % ST;
          const int keys = min(PP_BN, it.n - j * PP_BN);
          bool next_kv = false;  // K_{j+1} waited for
          for (int x = 0; x < 2 && ok; ++x) {
            if (j >= it.nk[x]) continue;
            const uint32_t buf = n_o[x] % NB;
            // the epilogue of the item that used this O last has read it out
            if ((j == 0 && n_o[x] >= NB &&
                 !mbar_wait_ab(&o_empty[x * NB + buf], (n_o[x] / NB - 1) & 1, a.status, abort_flag)) ||
                !mbar_wait_ab(&p_full[x], n_p[x] & 1, a.status, abort_flag)) {
              ok = false;
              break;
            }
            ++n_p[x];
            tc_fence_after();
            pp_issue_pv<HD>(smem_u32(sV + st * TILE), tmem + s_col(x), tmem + o_col<HD>(x, buf), j == 0, keys);
            if (x == 1 || j >= it.nk[1]) tc_commit(&kv_empty[st]);  // K_j and V_j read for the last time
            if (j + 1 < it.nk[x]) {
              if (!next_kv) {
                if (!mbar_wait_ab(&kv_full[st1], ((Jj + 1) / ST) & 1, a.status, abort_flag)) {
                  ok = false;
                  break;
                }
                tc_fence_after();
                next_kv = true;
              }
              issue_s(x, st1, min(PP_BN, it.n - (j + 1) * PP_BN));
              if (--left == 0) tc_commit(q_empty);
            } else {
              tc_commit(&o_full[x * NB + buf]);
              ++n_o[x];
              // (while this item's S are outstanding its Q buffers are, too)
              if (have && nx.nk[x] > 0 && left == 0) {
                first_s(x, Jn);
                early[x] = true;
              }
            }
          }
        }
        for (int x = 0; x < 2 && ok && have; ++x)
          if (nx.nk[x] > 0 && !early[x]) first_s(x, Jn);
        J = Jn;
      }
      // every MMA issued has finished before the CTA frees TMEM
      tc_commit(mma_done);
      mbar_wait(mma_done, 0, a.status);
    }
    __syncwarp();
  } else if (warp >= 4) {
    // ---------------------------------------------------------------- softmax + epilogue
    const int x = (warp - 4) / 4;  // tile
    const int quad = warp & 3;
    const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
    const uint32_t s_addr = tmem + lane_off + s_col(x);
    bool ok = true;
    uint32_t J = 0;                      // key blocks of the items before this one
    uint32_t n_s = 0, n_o = 0, n_e = 0;  // S blocks taken, items begun, epilogues done
    auto arrive = [&](uint64_t* bar) {
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
    };
    // the item whose epilogue is still to do: its row's output, normaliser and sums
    bf16* e_out = nullptr;  // nullptr: the row is past the sequence's end
    float* e_lse = nullptr;
    float e_m = 0.f, e_l = 0.f;
    // O / l in bf16, and the row normaliser
    auto epilogue = [&]() {
      const int buf = static_cast<int>(n_e % NB);
      const uint32_t o_addr = tmem + lane_off + o_col<HD>(x, buf);
      ok = ok && __all_sync(0xffffffffu, mbar_wait_ab(&o_full[x * NB + buf], (n_e / NB) & 1, a.status, abort_flag));
      tc_fence_after();
      if (ok && __any_sync(0xffffffffu, e_out != nullptr)) {
        const float inv = e_l > 0.f ? 1.f / e_l : 0.f;
#pragma unroll 1
        for (int c = 0; c < HD / 32; ++c) {
          uint32_t r[32];
          tmem_ld32(o_addr + 32 * c, r);
          tmem_ld_wait();
          if (e_out != nullptr) {
            uint32_t w[16];
#pragma unroll
            for (int v = 0; v < 16; ++v)
              w[v] = pack_bf16x2(__uint_as_float(r[2 * v]) * inv, __uint_as_float(r[2 * v + 1]) * inv);
            bf16* o = e_out + 32 * c;
            if (a.wide_out) {  // whole 32-byte sectors
              st_global_v8(o, w);
              st_global_v8(o + 16, w + 8);
            } else {
#pragma unroll
              for (int v = 0; v < 4; ++v)
                *reinterpret_cast<uint4*>(o + 8 * v) = make_uint4(w[4 * v], w[4 * v + 1], w[4 * v + 2], w[4 * v + 3]);
            }
          }
        }
        if (e_out != nullptr) *e_lse = e_m + log2f(e_l);
      }
      tc_fence_before();
      arrive(&o_empty[x * NB + buf]);
      ++n_e;
    };
    // The loop runs once more after the last item, for its epilogue.
    PpItem it;
    int r = 0;
    while (true) {
      int nk = 0;
      while (nk == 0 && pp_next(r, a, it)) {
        nk = x == 0 ? it.nk[0] : it.nk[1];
        if (nk == 0) J += it.n_kb;
      }
      if (nk == 0 && n_e == n_o) break;
      const int h = x == 0 ? it.h[0] : it.h[1];
      const int w0 = (x == 0 ? it.qb[0] : it.qb[1]) * PP_BM + quad * 32;  // the warp's first query
      const int q = w0 + lane;
      const uint32_t o_addr = tmem + lane_off + o_col<HD>(x, n_o % NB);
      float m = -INFINITY, l = 0.f;
      int j = 0;
      do {
        if (nk > 0) {
          ok = ok && __all_sync(0xffffffffu, mbar_wait_ab(&s_full[x], n_s & 1, a.status, abort_flag));
          ++n_s;
          tc_fence_after();
          // keys k0 + e with e >= lim are hidden (causal diagonal, sequence end):
          // lim grows with the row, so 32-column chunks below the first row's
          // limit need no mask and chunks past the last row's hold no key
          const int k0 = j * PP_BN;
          const int keys = min(PP_BN, it.n - k0);
          const int lim = a.causal ? min(keys, q - k0 + 1) : keys;
          const int lim_first = a.causal ? min(keys, w0 - k0 + 1) : keys;
          const int n_ch = ((a.causal ? min(keys, w0 + 32 - k0) : keys) + 31) / 32;
          auto mask = [&](uint32_t (&v)[32], int c) {  // hidden scores become -inf
            if (32 * c + 32 > lim_first) {
#pragma unroll
              for (int e = 0; e < 32; ++e) v[e] = 32 * c + e < lim ? v[e] : 0xff800000u;
            }
          };
          if (keys & 15) {
            // P is zero past the last key, but V's rows there belong to another
            // sequence (or are zero-filled): keep a non-finite one out of 0 * V
            const uint32_t va = smem_u32(sV + (J + j) % ST * TILE);
            const int t = static_cast<int>(threadIdx.x) & 127, per = (-keys & 15) * 8;
            for (int i = t; i < per * CH; i += 128)
              asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(va + (i / per) * (PP_BN * 128) +
                                                                          keys * 128 + (i % per) * 16),
                           "r"(0)
                           : "memory");
            fence_proxy_async_smem();
          }
          if (ok && w0 < it.n) {  // some row of the warp is a query
            // pass 1: the block's row maximum
            float mx = -INFINITY;
            int c1 = 0;
#pragma unroll 1
            for (; 32 * c1 + 64 <= lim_first; c1 += 2) {  // two whole chunks per TMEM round trip
              uint32_t u[64];
              tmem_ld32(s_addr + 32 * c1, *reinterpret_cast<uint32_t(*)[32]>(u));
              tmem_ld32(s_addr + 32 * c1 + 32, *reinterpret_cast<uint32_t(*)[32]>(u + 32));
              tmem_ld_wait();
              float m4[4] = {mx, mx, mx, mx};
#pragma unroll
              for (int e = 0; e < 64; e += 8)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                  m4[k] = fmax3(m4[k], __uint_as_float(u[e + 2 * k]), __uint_as_float(u[e + 2 * k + 1]));
              mx = fmaxf(fmax3(m4[0], m4[1], m4[2]), m4[3]);
            }
#pragma unroll 1
            for (int c = c1; c < n_ch; ++c) {
              uint32_t u[32];
              tmem_ld32(s_addr + 32 * c, u);
              tmem_ld_wait();
              mask(u, c);
              float m4[4] = {mx, mx, mx, mx};
#pragma unroll
              for (int e = 0; e < 32; e += 8)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                  m4[k] = fmax3(m4[k], __uint_as_float(u[e + 2 * k]), __uint_as_float(u[e + 2 * k + 1]));
              mx = fmaxf(fmax3(m4[0], m4[1], m4[2]), m4[3]);
            }
            const float mb = mx == -INFINITY ? -INFINITY : mx * a.scale_log2;
            const bool need = mb > m + PP_RESCALE_LOG2;
            if (__any_sync(0xffffffffu, need)) {
              const float mn = need ? mb : m;
              const float f = need ? (m == -INFINITY ? 0.f : exp2f(m - mn)) : 1.f;
              if (j > 0) {  // O holds blocks 0..j-1 (PV_x(j-1) finished before S_x(j) was signalled)
#pragma unroll 1
                for (int c = 0; c < HD / 32; ++c) {
                  uint32_t v[32];
                  tmem_ld32(o_addr + 32 * c, v);
                  tmem_ld_wait();
#pragma unroll
                  for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) * f);
                  tmem_st32(o_addr + 32 * c, v);
                }
              }
              l *= f;
              m = mn;
            }
            // pass 2: P as a bf16 pair over the S columns just read; the next
            // chunk's load is in flight while this one is converted
            // P = 2^(s*scale - m) split as hi = P rounded to bf16 and lo = P - hi
            // (exact in fp32, then rounded to bf16), so hi + lo carries P to
            // about 17 bits
            const uint64_t scale2 = f2pack(a.scale_log2, a.scale_log2);
            const uint64_t nm2 = f2pack(-m, -m);
            uint32_t v[32];
            tmem_ld32(s_addr, v);
            tmem_ld_wait();
#pragma unroll 1
            for (int c = 0; c < n_ch; ++c) {
              mask(v, c);
              uint64_t t[16];
#pragma unroll
              for (int e = 0; e < 16; ++e)
                t[e] = ffma2(f2pack(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1])), scale2, nm2);
              if (c + 1 < n_ch) tmem_ld32(s_addr + 32 * (c + 1), v);
              uint32_t hi[16], lo[16];
              uint64_t lsum = f2pack(0.f, 0.f);
#pragma unroll
              for (int e = 0; e < 16; ++e) {
                float p0, p1, r0, r1;
                f2unpack(t[e], p0, p1);
                p0 = ex2_fast(p0);
                p1 = ex2_fast(p1);
                const uint64_t pp = f2pack(p0, p1);
                lsum = fadd2(lsum, pp);
                hi[e] = pack_bf16x2(p0, p1);
                f2unpack(fsub2(pp, f2pack(bf16lo(hi[e]), bf16hi(hi[e]))), r0, r1);
                lo[e] = pack_bf16x2(r0, r1);
              }
              float l0, l1;
              f2unpack(lsum, l0, l1);
              l += l0 + l1;
              tmem_st16(s_addr + 32 * c, hi);
              tmem_st16(s_addr + 32 * c + 16, lo);
              tmem_ld_wait();
            }
            // P of the chunks that hold no key of this warp but some of the tile
#pragma unroll 1
            for (int c = n_ch; 32 * c < keys; ++c) {
              const uint32_t z[16] = {};
              tmem_st16(s_addr + 32 * c, z);
              tmem_st16(s_addr + 32 * c + 16, z);
            }
            tmem_st_wait();
          }
          tc_fence_before();
          arrive(&p_full[x]);
        }
        // the previous item's output, under this one's first P V
        if (j == 0 && n_e < n_o) epilogue();
      } while (++j < nk);
      if (nk == 0) break;
      const bool live = q < it.n;
      e_out = live ? a.out + (static_cast<size_t>(it.row0) + q) * (static_cast<size_t>(a.Hq) * HD) + h * HD : nullptr;
      e_lse = a.lse2 + (static_cast<size_t>(it.b) * a.Hq + h) * a.N + q;
      e_m = m;
      e_l = l;
      ++n_o;
      J += it.n_kb;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, PP_TMEM_COLS);
  }
}

int pp_sms() {
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  if (cached[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
    cached[dev] = n;
  }
  return cached[dev];
}

bool encode_rows(CUtensorMap* m, const void* base, uint64_t cols, uint64_t rows) {
  EncodeTiledFn enc = get_encode_tiled();
  if (enc == nullptr) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, 128};
  cuuint32_t es[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int HD>
cudaError_t run_pp(const void* qkv, int B, int N, int Hq, int Hkv, void* out, float* lse, int causal, int* status,
                   cudaStream_t s, const int* cu, int rows) {
  using C = PpCfg<HD>;
  const int ld = (Hq + 2 * Hkv) * HD;
  CUtensorMap tm;
  if (!encode_rows(&tm, qkv, static_cast<uint64_t>(ld), cu ? static_cast<uint64_t>(rows) : static_cast<uint64_t>(B) * N))
    return cudaErrorInvalidValue;
  static OncePerDevice once;
  const cudaError_t attr = set_smem_limit_once(once, attn_pp_kernel<HD>, static_cast<int>(C::SMEM));
  if (attr != cudaSuccess) return attr;
  PpArgs a;
  a.lse2 = lse;
  a.out = static_cast<bf16*>(out);
  a.B = B;
  a.N = N;
  a.Hq = Hq;
  a.Hkv = Hkv;
  a.n_qb = (N + PP_BM - 1) / PP_BM;
  a.causal = causal;
  // an even number of heads per group: two heads a tile pair (equal key blocks);
  // otherwise two query blocks of one head
  const int per = Hq / Hkv;
  a.by_head = per % 2 == 0;
  a.wide_out = (reinterpret_cast<uintptr_t>(out) & 31) == 0;
  a.units = fast_div(a.by_head ? per / 2 : per);
  a.groups = fast_div(Hkv);
  a.inner = fast_div(B * Hkv * a.units.d);
  a.total = (a.by_head ? a.n_qb : (a.n_qb + 1) / 2) * a.inner.d;
  a.cu = cu;
  a.scale_log2 = 1.4426950408889634f / sqrtf(static_cast<float>(HD));
  a.status = status;
  const int grid = a.total < pp_sms() ? a.total : pp_sms();
  ZSAA_LAUNCH(attn_pp_kernel<HD>, dim3(grid), dim3(PP_THREADS), C::SMEM, s, tm, a);
  return cudaGetLastError();
}

}  // namespace

bool attention_pp_supported(int dtype, int hd, int Hq, int Hkv, const uint8_t* key_alive, int* status) {
  return dtype == ZSAA_BF16 && (hd == 64 || hd == 128) && Hkv > 0 && Hq % Hkv == 0 && key_alive == nullptr &&
         status != nullptr;
}

cudaError_t launch_attention_pp(const void* qkv, int B, int N, int Hq, int Hkv, int hd, void* out, float* lse,
                                int causal, int* status, cudaStream_t s, const int* cu, int rows) {
  if (B < 1 || N < 1) return cudaSuccess;
  if (hd == 64) return run_pp<64>(qkv, B, N, Hq, Hkv, out, lse, causal, status, s, cu, rows);
  if (hd == 128) return run_pp<128>(qkv, B, N, Hq, Hkv, out, lse, causal, status, s, cu, rows);
  return cudaErrorInvalidValue;
}

}  // namespace zsaa

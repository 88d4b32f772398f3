// Soft-score column mass on the sm_103a tensor cores (Sec. 3.2: soft-score
// times V gives each V row's contribution).
//
// S^T = K Q^T puts keys on the MMA's rows: a tile is (sequence b, KV group g,
// some query heads of g, up to 256 keys), held as one or two 128-key blocks
// (the M = 128 operands), and the queries of each head stream past it in stages
// (only queries at or after the keys when the mask is causal).  Epilogue
// warps -- one TMEM lane, i.e. one key, per thread -- accumulate
// exp2(s * c - lse2[q]) over the queries q >= key: the column sum of the
// normalised soft-score P (the row normalisers lse2 come from the attention
// kernel).  Each head writes its own partial, optionally times ||v_key|| of
// group g (the position score of R1 is linear in the column mass; the norms
// come from the QKV projection's epilogue):   parts[head][b][g][key]
// and the select / reduce kernels sum a group's heads in a fixed order.
//
// What bounds it: per 128 x 256 scores, the tensor pipe needs hd/16 N = 256
// MMAs of 128 clocks (which also take most of the shared-memory bandwidth at
// hd 128), the exponentials 1024 clocks of MUFU.  So:
//  - two key blocks per query stage, so a stage's copy is used twice, and N = 256:
//    the issuing thread needs about 100 clocks an MMA whatever its width, and a
//    narrower one re-reads the keys more often (N = 192 and N = 160 with three
//    stages or accumulators ran at 1.1x the time; sharing the copies of two CTAs
//    by multicast did not help either);
//  - two TMEM accumulators, each with its own group of eight epilogue warps, so
//    one group's exponentials run under the other's MMAs and both share the
//    MUFU; no barrier between warps inside a head;
//  - a warp of its own copies the normalisers, several stages ahead;
//  - several heads per tile where there are tiles enough: they share its keys.
// One key block and N = 128 per step with eight epilogue warps and a barrier a
// step took 116 us at 4 x 2048 rows, 32 heads of 128 (causal), and 49 us at
// 64 x 256 rows, 32 heads of 64; this takes 82
// and 37 (the reduce kernel of the stand-alone call included in all four).
//
// Work is counted in substeps, one accumulator each: with two key blocks a
// query stage is two substeps (block 0, block 1), with one key block its two
// halves are.  Substep i belongs to accumulator and epilogue
// group i mod 2.
//
// Roles (608 threads): warp 0 TMA producer (key blocks through KS slots, the
// queries through QS stages), warp 1 MMA issuer, warp 2 normaliser loader, warps
// 3..18 epilogue (group (warp-3)/8; warp w reads TMEM lanes 32*(w%4)..+32 and
// every other 32-column chunk).  All waits are bounded; epilogue warps never
// leave the step loops early, so their named barriers cannot strand the others.
#include "common.cuh"
#include "kernels.h"

namespace zsaa {
namespace {

constexpr int CM_KB = 128;   // keys per block (MMA M)
constexpr int CM_TQ = 256;      // queries per stage (MMA N)
constexpr int CM_THREADS = 608;
constexpr int CM_GROUP_WARPS = 8;
constexpr int CM_LS = 4;     // normaliser slots

template <int HD>
struct CmCfg {
  static constexpr int CHUNKS = HD / 64;                 // 64-wide swizzled K chunks
  static constexpr int K_BYTES = CM_KB * HD * 2;          // one key block
  static constexpr int Q_BYTES = CM_TQ * HD * 2;             // one query stage
  static constexpr int KS = HD == 128 ? 2 : 4;            // key-block slots
  static constexpr int QS = HD == 128 ? 2 : 4;            // query stages
  // operands, 512 B of barriers, normalisers, partial sums (2 x 2 x 128 within a group, 3 x 128 across)
  static constexpr size_t SMEM = static_cast<size_t>(K_BYTES) * KS + static_cast<size_t>(Q_BYTES) * QS + 512 +
                                 CM_LS * CM_TQ * 4 + 7 * CM_KB * 4 + 1024;
};
static_assert(CmCfg<64>::SMEM <= 227 * 1024 && CmCfg<128>::SMEM <= 227 * 1024, "shared memory");

struct CmArgs {
  const float* lse2;   // [B, Hq, N]
  const float* vnorm;  // [B*N, Hkv] ||v|| per row and group (used when weight_vnorm)
  float* parts;        // [per * nsplit][B][G][N]
  int B, N, Hq, Hkv, total, weight_vnorm;
  int tk;      // keys per tile: CM_KB or 2 CM_KB
  int hpt;     // query heads of one group per tile
  int nsplit;  // parts of a head's queries, each a tile of its own
  FastDiv inner, chunks, groups;  // tiles per key position, head chunks (times nsplit) per group, groups
  int causal;  // 0: bidirectional (every query, no causal mask)
  const int* cu;  // packed sequences of different lengths: rows [cu[b], cu[b+1]); N = the longest
  const uint8_t* q_alive;  // masked mode: [B, N] flags, queries with 0 add nothing
  float scale_log2;
  int* status;
};

// 2^x with the MUFU approximation (flush-to-zero: soft-score terms below
// 2^-126 are negligible next to the column sums).
__device__ __forceinline__ float ex2_ftz(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

struct CmTile {
  int b, g, hh0, h0;  // sequence, group, first query head within the group and overall
  int row0, n;        // first packed row and length of the sequence
  int key0, nk;       // first key, live key blocks (1 or 2)
  int split;          // which part of the queries
  int q_first, n_st;  // its first query, query stages per head
};

// Tile t; false when its sequence has no such keys (it is shorter than the longest).
__device__ __forceinline__ bool cm_tile(int t, const CmArgs& a, CmTile& c) {
  int r, hc;
  const int kp = a.inner.div(t, r);  // early keys first: they have the most queries
  r = a.chunks.div(r, hc);
  c.b = a.groups.div(r, c.g);
  c.split = 0;
  if (a.nsplit > 1) {  // hpt is 1
    c.split = hc % a.nsplit;
    hc /= a.nsplit;
  }
  c.hh0 = hc * a.hpt;
  c.h0 = c.g * (a.Hq / a.Hkv) + c.hh0;
  if (a.cu) {
    c.row0 = a.cu[c.b];
    c.n = a.cu[c.b + 1] - c.row0;
  } else {
    c.row0 = c.b * a.N;
    c.n = a.N;
  }
  c.key0 = kp * a.tk;
  c.nk = min(a.tk, c.n - c.key0) > CM_KB ? 2 : 1;
  c.q_first = a.causal ? c.key0 : 0;
  c.n_st = (c.n - c.q_first + CM_TQ - 1) / CM_TQ;
  if (a.nsplit > 1) {
    const int s0 = c.split * c.n_st / a.nsplit, s1 = (c.split + 1) * c.n_st / a.nsplit;
    c.q_first += s0 * CM_TQ;
    c.n_st = s1 - s0;
  }
  return c.key0 < c.n;
}

// This CTA's tiles: dealt in a snake order (0..G-1, then G-1..0, ...), so the
// causal triangle's long and short tiles even out.  Advances r to the next
// live tile; false when there is none.
__device__ __forceinline__ bool cm_next(int& r, const CmArgs& a, CmTile& c) {
  const int G = gridDim.x, i = blockIdx.x;
  while (true) {
    const int t = r * G + ((r & 1) ? G - 1 - i : i);
    ++r;
    if (r > (a.total + G - 1) / G) return false;
    if (t < a.total && cm_tile(t, a, c)) return true;
  }
}

// Substeps of the stage whose first query is q0.
__device__ __forceinline__ int cm_subs(const CmTile& c, int q0) {
  return c.nk == 2 || q0 + CM_TQ / 2 < c.n ? 2 : 1;
}

template <int HD>
__global__ void __launch_bounds__(CM_THREADS, 1)
    colmass_tc_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_q,
                      const CmArgs a) {
  using C = CmCfg<HD>;
  constexpr int KS = C::KS, QS = C::QS;
  constexpr int KCH = CM_KB * 128, QCH = CM_TQ * 128, QHCH = QCH / 2;  // bytes of one 64-dim chunk; half a query stage
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* sK = smem;                       // [KS] key blocks
  uint8_t* sQ = sK + KS * C::K_BYTES;       // [QS] query stages
  uint8_t* tail = sQ + QS * C::Q_BYTES;
  uint64_t* qfull = reinterpret_cast<uint64_t*>(tail);  // [QS]
  uint64_t* qempty = qfull + QS;                        // [QS]
  uint64_t* kfull = qempty + QS;                        // [KS]
  uint64_t* kempty = kfull + KS;                        // [KS]
  uint64_t* acc_full = kempty + KS;                     // [2]
  uint64_t* acc_empty = acc_full + 2;                   // [2]
  uint64_t* lfull = acc_empty + 2;                      // [LS]
  uint64_t* lempty = lfull + CM_LS;                     // [LS]
  uint64_t* mma_done = lempty + CM_LS;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* s_lse = reinterpret_cast<float*>(tail + 512);  // [LS][CM_TQ]
  float* s_own = s_lse + CM_LS * CM_TQ;                 // [2 groups][2][CM_KB] half 1's sums
  float* s_all = s_own + 4 * CM_KB;                     // [3][CM_KB] all but group 0 half 0's sums

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < QS; ++s) {
      mbar_init(&qfull[s], 1);
      mbar_init(&qempty[s], 1);
    }
    for (int s = 0; s < KS; ++s) {
      mbar_init(&kfull[s], 1);
      mbar_init(&kempty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&acc_full[s], 1);
      mbar_init(&acc_empty[s], CM_GROUP_WARPS);
    }
    for (int s = 0; s < CM_LS; ++s) {
      mbar_init(&lfull[s], 32);
      mbar_init(&lempty[s], 2 * CM_GROUP_WARPS);
    }
    mbar_init(mma_done, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 0 && lane < 2) prefetch_tmap(lane == 0 ? &tm_k : &tm_q);
  if (warp == 1) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      bool ok = true;
      uint32_t it = 0, kc = 0;  // query stages and key blocks issued
      CmTile c;
      for (int r = 0; ok && cm_next(r, a, c);) {
        for (int x = 0; x < c.nk && ok; ++x) {
          const int s = kc % KS;
          if (!mbar_wait_ab(&kempty[s], ((kc / KS) & 1) ^ 1, a.status, abort_flag)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&kfull[s], C::K_BYTES);
          for (int ch = 0; ch < C::CHUNKS; ++ch)
            tma_load_2d(sK + s * C::K_BYTES + ch * KCH, &tm_k, (a.Hq + c.g) * HD + ch * 64,
                        c.row0 + c.key0 + x * CM_KB, &kfull[s]);
          ++kc;
        }
        for (int hh = 0; hh < a.hpt && ok; ++hh)
          for (int st = 0; st < c.n_st; ++st, ++it) {
            const int s = it % QS, q0 = c.q_first + st * CM_TQ;
            if (!mbar_wait_ab(&qempty[s], ((it / QS) & 1) ^ 1, a.status, abort_flag)) {
              ok = false;
              break;
            }
            const int boxes = q0 + CM_TQ / 2 < c.n ? 2 : 1;  // halves with a live query
            mbar_arrive_expect_tx(&qfull[s], boxes * (C::Q_BYTES / 2));
            for (int ch = 0; ch < C::CHUNKS; ++ch)
              for (int y = 0; y < boxes; ++y)
                tma_load_2d(sQ + s * C::Q_BYTES + ch * QCH + y * QHCH, &tm_q, (c.h0 + hh) * HD + ch * 64,
                            c.row0 + q0 + y * (CM_TQ / 2), &qfull[s]);
          }
      }
      if (!ok || *abort_flag) {  // let the copies already issued land before the CTA's memory goes away
        for (uint32_t j = it; j > 0 && j + QS > it; --j)
          mbar_wait(&qfull[(j - 1) % QS], ((j - 1) / QS) & 1, nullptr);
        for (uint32_t j = kc; j > 0 && j + KS > kc; --j)
          mbar_wait(&kfull[(j - 1) % KS], ((j - 1) / KS) & 1, nullptr);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      uint32_t it = 0, kc = 0, i = 0;  // query stages, key blocks, substeps
      bool ok = true;
      CmTile c;
      for (int r = 0; ok && cm_next(r, a, c); kc += c.nk) {
        uint32_t kseen = 0;  // key blocks of this tile already waited for
        for (int hh = 0; hh < a.hpt && ok; ++hh)
          for (int st = 0; st < c.n_st && ok; ++st, ++it) {
            const int s = it % QS, q0 = c.q_first + st * CM_TQ;
            const bool last = hh == a.hpt - 1 && st == c.n_st - 1;
            if (!mbar_wait_ab(&qfull[s], (it / QS) & 1, a.status, abort_flag)) {
              ok = false;
              break;
            }
            const int subs = cm_subs(c, q0);
            for (int x = 0; x < subs; ++x, ++i) {
              const int ab = i & 1;
              const uint32_t kb = kc + (c.nk == 2 ? x : 0);
              if (!mbar_wait_ab(&acc_empty[ab], ((i >> 1) & 1) ^ 1, a.status, abort_flag) ||
                  (!(kseen >> (kb - kc) & 1) && !mbar_wait_ab(&kfull[kb % KS], (kb / KS) & 1, a.status, abort_flag))) {
                ok = false;
                break;
              }
              kseen |= 1u << (kb - kc);
              tc_fence_after();
              const uint32_t k_base = smem_u32(sK + (kb % KS) * C::K_BYTES);
              const uint32_t q_base = smem_u32(sQ + s * C::Q_BYTES) + (c.nk == 2 ? 0 : x * QHCH);
              const uint32_t idesc = idesc_bf16_f32(CM_KB, c.nk == 2 && q0 + CM_TQ / 2 < c.n ? CM_TQ : CM_TQ / 2);
              const uint32_t d_tmem = tmem + static_cast<uint32_t>(ab * 256);
#pragma unroll
              for (int kk = 0; kk < HD / 16; ++kk)
                tc_mma_bf16(d_tmem, sdesc_sw128(k_base + (kk / 4) * KCH + (kk % 4) * 32),
                            sdesc_sw128(q_base + (kk / 4) * QCH + (kk % 4) * 32), idesc, kk > 0 ? 1u : 0u);
              tc_commit(&acc_full[ab]);
              if (last && (c.nk == 2 || x == subs - 1)) tc_commit(&kempty[kb % KS]);
            }
            if (ok) tc_commit(&qempty[s]);
          }
      }
      // every MMA issued has finished before the CTA frees TMEM
      tc_commit(mma_done);
      mbar_wait(mma_done, 0, a.status);
    }
    __syncwarp();
  } else if (warp == 2) {
    // ---------------------------------------------------------------- normaliser loader
    uint32_t it = 0;
    bool ok = true;
    CmTile c;
    for (int r = 0; ok && cm_next(r, a, c);)
      for (int hh = 0; hh < a.hpt && ok; ++hh)
        for (int st = 0; st < c.n_st; ++st, ++it) {
          const int s = it % CM_LS, q0 = c.q_first + st * CM_TQ;
          const float* src = a.lse2 + (static_cast<size_t>(c.b) * a.Hq + c.h0 + hh) * a.N;
          ok = __all_sync(0xffffffffu, mbar_wait_ab(&lempty[s], ((it / CM_LS) & 1) ^ 1, a.status, abort_flag));
          if (!ok) break;
          if (a.q_alive == nullptr) {  // asynchronous copies; they arrive on the barrier by themselves
#pragma unroll
            for (int e = 0; e < CM_TQ / 32; ++e) {
              const int q = q0 + e * 32 + lane;
              asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                               smem_u32(s_lse + s * CM_TQ + e * 32 + lane)),
                           "l"(q < c.n ? src + q : src), "r"(q < c.n ? 4 : 0)
                           : "memory");
            }
            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&lfull[s])) : "memory");
          } else {
#pragma unroll
            for (int e = 0; e < CM_TQ / 32; ++e) {
              const int q = q0 + e * 32 + lane;
              float v = q < c.n ? src[q] : 0.f;
              // exp2(s * c - inf) = 0: a hidden query contributes nothing
              if (q < c.n && a.q_alive[static_cast<size_t>(c.b) * a.N + q] == 0) v = INFINITY;
              s_lse[s * CM_TQ + e * 32 + lane] = v;
            }
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&lfull[s])) : "memory");
          }
        }
    cp_async_wait<0>();
  } else {
    // ---------------------------------------------------------------- epilogue
    const int grp = (warp - 3) / CM_GROUP_WARPS;  // accumulator
    const int quad = warp & 3, half = ((warp - 3) >> 2) & 1;
    const int krow = quad * 32 + lane;  // key within its block
    const uint32_t t_addr = tmem + static_cast<uint32_t>(grp * 256) + (static_cast<uint32_t>(quad * 32) << 16);
    auto arrive = [&](uint64_t* bar) {
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
    };
    const uint64_t nc2 = f2pack(-a.scale_log2, -a.scale_log2);
    uint32_t it = 0, i = 0, own = 0;  // query stages, substeps, heads finished by this group alone
    bool ok = true;
    CmTile c;
    for (int r = 0; cm_next(r, a, c);) {
      for (int hh = 0; hh < a.hpt; ++hh) {
        const uint32_t i0 = i;
        const int x0 = static_cast<int>((grp ^ i0) & 1);  // this group's first substep of the head
        const int key = c.key0 + (c.nk == 2 ? x0 * CM_KB : 0) + krow;
        float acc = 0.f, vn = 1.f;
        if (a.weight_vnorm && half == 0 && key < c.n)
          vn = a.vnorm[(static_cast<size_t>(c.row0) + key) * a.Hkv + c.g];
        for (int st = 0; st < c.n_st; ++st, ++it) {
          const int q0 = c.q_first + st * CM_TQ;
          const int subs = cm_subs(c, q0);
          ok = ok && __all_sync(0xffffffffu, mbar_wait_ab(&lfull[it % CM_LS], (it / CM_LS) & 1, a.status, abort_flag));
          for (int x = 0; x < subs; ++x, ++i) {
            if ((i & 1) != static_cast<uint32_t>(grp)) continue;
            ok = ok && __all_sync(0xffffffffu, mbar_wait_ab(&acc_full[grp], (i >> 1) & 1, a.status, abort_flag));
            tc_fence_after();
            if (ok) {
              const int kmin = c.key0 + (c.nk == 2 ? x * CM_KB : 0) + quad * 32;  // the warp's first key
              const int qs = q0 + (c.nk == 2 ? 0 : x * (CM_TQ / 2));  // the substep's first query
              const int ncol = min(c.nk == 2 ? CM_TQ : CM_TQ / 2, c.n - qs);
              const float* L = s_lse + (it % CM_LS) * CM_TQ + (qs - q0);
              // chunks of 32 queries, every other one; those wholly before the warp's keys are skipped
              int ch = half * 32;
              ch += (max(0, a.causal ? kmin - qs - 31 : 0) - ch + 63) / 64 * 64;
#pragma unroll 1
              for (; ch < ncol; ch += 64) {
                uint32_t v[32];
                tmem_ld32(t_addr + ch, v);
                tmem_ld_wait();
                // lse - s c for two columns in one packed FMA, then exp2 of its
                // negation (the same rounding as s c - lse), summed in pairs
                const int qc = qs + ch;
                uint64_t sum = 0ull;
                auto add4 = [&](int e, uint32_t mask) {  // bits of mask: columns inside the mask
                  const ulonglong2 l2 = *reinterpret_cast<const ulonglong2*>(L + ch + e);
                  float u[4];
                  f2unpack(ffma2(f2pack(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), nc2, l2.x), u[0], u[1]);
                  f2unpack(ffma2(f2pack(__uint_as_float(v[e + 2]), __uint_as_float(v[e + 3])), nc2, l2.y), u[2], u[3]);
#pragma unroll
                  for (int k = 0; k < 4; ++k) u[k] = (mask >> (e + k)) & 1u ? ex2_ftz(-u[k]) : 0.f;
                  sum = fadd2(fadd2(sum, f2pack(u[0], u[1])), f2pack(u[2], u[3]));
                };
                if ((!a.causal || qc >= kmin + 31) && qc + 32 <= c.n) {  // the warp's whole chunk is visible
#pragma unroll
                  for (int e = 0; e < 32; e += 4) add4(e, 0xffffffffu);
                } else {
                  const int lo = a.causal ? max(0, key - qc) : 0, hi = c.n - qc;  // columns [lo, hi)
                  const uint32_t mask = (lo > 31 ? 0u : 0xffffffffu << lo) & (hi > 31 ? 0xffffffffu : (1u << hi) - 1u);
#pragma unroll
                  for (int e = 0; e < 32; e += 4) add4(e, mask);
                }
                float a0, a1;
                f2unpack(sum, a0, a1);
                acc += a0 + a1;
              }
            }
            tc_fence_before();
            arrive(&acc_empty[grp]);
          }
          arrive(&lempty[it % CM_LS]);
        }
        // Add the partial sums of a key in a fixed order.  A group that has its
        // keys to itself (two key blocks, or one substep in all) adds its two
        // halves; one key block in several substeps is shared by both groups.
        const int subs_done = static_cast<int>(i - i0);
        const bool alone = c.nk == 2 || subs_done == 1;
        if (alone && x0 < subs_done) {
          float* sp = s_own + (grp * 2 + (own++ & 1)) * CM_KB;
          if (half == 1) sp[krow] = acc;
          if (grp == 0)
            asm volatile("bar.sync 1, %0;" ::"n"(CM_GROUP_WARPS * 32) : "memory");
          else
            asm volatile("bar.sync 2, %0;" ::"n"(CM_GROUP_WARPS * 32) : "memory");
          if (half == 0) acc += sp[krow];
          // this buffer is rewritten two heads of the group later, after the next one's barrier
        } else if (!alone) {
          if (grp + half > 0) s_all[(grp * 2 + half - 1) * CM_KB + krow] = acc;
          asm volatile("bar.sync 3, %0;" ::"n"(2 * CM_GROUP_WARPS * 32) : "memory");
          if (grp + half == 0) acc = ((acc + s_all[krow]) + s_all[CM_KB + krow]) + s_all[2 * CM_KB + krow];
          asm volatile("bar.sync 3, %0;" ::"n"(2 * CM_GROUP_WARPS * 32) : "memory");
        }
        if (half == 0 && (alone ? x0 < subs_done : grp == 0) && key < c.n)
          a.parts[((static_cast<size_t>((c.hh0 + hh) * a.nsplit + c.split) * a.B + c.b) * a.Hkv + c.g) * a.N + key] = acc * vn;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

int cm_num_sms() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 148;
  return n;
}

// Tensor map of the packed qkv rows, boxes of 64 columns (128 bytes, swizzled) by box_rows.
bool cm_map(CUtensorMap* m, const void* qkv, uint64_t cols, uint64_t rows, int box_rows) {
  EncodeTiledFn enc = get_encode_tiled();
  if (enc == nullptr) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, static_cast<cuuint32_t>(box_rows)};
  cuuint32_t es[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(qkv), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Query heads per tile (they share its key blocks): the most that still give
// every SM six tiles.
int cm_heads_per_tile(int per, long long key_tiles, int sms) {
  int best = 1;
  for (int h = 1; h <= per; ++h)
    if (per % h == 0 && key_tiles * (per / h) >= 6LL * sms) best = h;
  return best;
}

template <int HD>
cudaError_t run_cm(const void* qkv, uint64_t cols, uint64_t rows, const CmArgs& a, int sms, cudaStream_t s) {
  using C = CmCfg<HD>;
  CUtensorMap tm_k, tm_q;
  if (!cm_map(&tm_k, qkv, cols, rows, CM_KB) || !cm_map(&tm_q, qkv, cols, rows, CM_TQ / 2))
    return cudaErrorInvalidValue;
  static OncePerDevice once;
  const cudaError_t attr_err = set_smem_limit_once(once, colmass_tc_kernel<HD>, static_cast<int>(C::SMEM));
  if (attr_err != cudaSuccess) return attr_err;
  const int grid = a.total < sms ? a.total : sms;
  ZSAA_LAUNCH(colmass_tc_kernel<HD>, dim3(grid), dim3(CM_THREADS), C::SMEM, s, tm_k, tm_q, a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_colmass_tc(const void* qkv, const float* lse, const float* vnorm, int B, int N,
                              int Hq, int Hkv, int hd, float* parts, int* status, int* n_chunks,
                              int causal, cudaStream_t s, const int* cu, int rows,
                              const uint8_t* q_alive) {
  if (hd != 64 && hd != 128) return cudaErrorInvalidValue;
  const int ld = (Hq + 2 * Hkv) * hd;
  CmArgs a;
  a.lse2 = lse;
  a.vnorm = vnorm;
  a.parts = parts;
  a.B = B;
  a.N = N;
  a.Hq = Hq;
  a.Hkv = Hkv;
  const int per = Hq / Hkv, sms = cm_num_sms();
  // Tiles of two key blocks, of one where pairs would not give every SM a tile
  // (1 x 4096 rows, 8 heads of 128: 43 -> 30 us), and of half the queries where
  // even those end in a ragged second wave of equal tiles (no causal mask, so
  // no short tiles to fill it; 1 x 1500 rows, 16 heads of 64: 22.8 -> 20.5 us).
  auto tiles = [&](int tk) { return static_cast<long long>((N + tk - 1) / tk) * B * Hq; };
  a.tk = tiles(2 * CM_KB) < sms ? CM_KB : 2 * CM_KB;
  a.nsplit = !causal && cu == nullptr && a.tk == CM_KB && tiles(CM_KB) > sms && tiles(CM_KB) < 2 * sms && N > 2 * CM_TQ ? 2 : 1;
  const int n_kp = (N + a.tk - 1) / a.tk;
  a.hpt = a.nsplit > 1 ? 1 : cm_heads_per_tile(per, static_cast<long long>(n_kp) * B * Hkv, sms);
  a.chunks = fast_div(per / a.hpt * a.nsplit);
  a.groups = fast_div(Hkv);
  a.inner = fast_div(B * Hkv * a.chunks.d);
  a.total = n_kp * a.inner.d;
  a.weight_vnorm = vnorm != nullptr;
  a.causal = causal;
  a.cu = cu;
  a.q_alive = q_alive;
  a.scale_log2 = 1.4426950408889634f / sqrtf(static_cast<float>(hd));
  a.status = status;
  *n_chunks = per * a.nsplit;
  const uint64_t all = cu ? static_cast<uint64_t>(rows) : static_cast<uint64_t>(B) * N;
  return hd == 64 ? run_cm<64>(qkv, ld, all, a, sms, s) : run_cm<128>(qkv, ld, all, a, sms, s);
}

}  // namespace zsaa

// fp32 CUDA-core GEMM for models stored in float32: out = epi(A[M,K] W[N,K]^T).
// True fp32 FMA (no TF32).  Epilogues: store, residual add, SwiGLU (two weight
// matrices, gate and up), RoPE (the QKV projection, read from its three
// weight matrices).
//
// What bounds it: the FMA pipe (about 76 TFLOP/s) once there are enough tiles,
// and the length of one tile's K chain when there are few.  So:
//  - 64 x 64 tiles of two groups of 64 threads, each group half of the tile's K
//    with its own stages and barrier: a CTA loads all four schedulers (one of
//    two warps leaves two idle, and two such CTAs can meet on the same two).
//  - 8 x 8 outputs a thread, as packed pairs of neighbouring columns
//    (fma.rn.f32x2 with the row's value in both halves; an output is one FMA
//    chain per part of K).  That wants a k's columns side by side, so a thread
//    moves its weights from the place they were copied to into [16 k][64
//    columns]; A stays K-major (rows of 16 k, padded to 20 floats), four k of a
//    row read at once.  Copies, moves and reads hit distinct banks.  From shared
//    memory alone this loop runs at 62 TFLOP/s in 134 registers; with pairs of k
//    and no transpose it needs twice the accumulators and runs at 55.
//  - Three stages of 16-byte cp.async, weights too: loaded through registers one
//    block ahead, the few-tile shapes waited on them (24 rows, N 2048, K 1024:
//    37 us against 33 for a whole tile).
//  - Few tiles: K is also split over a thread-block cluster of S <= 8 CTAs,
//    whose partial tiles meet in distributed shared memory and are added in the
//    order of their parts (deterministic).
//    Measured, d 1024, ffn 4096, 324-1536 rows, a launch: gate/up 206 us (43
//    TFLOP/s on average, 53 at 1536 rows), down 113, QKV with RoPE 70, O 54;
//    with pairs of k, one group and the earlier split rule 247, 138, 89, 59;
//    with 4 x 4 outputs a thread, 4-byte staging and one stage 399, 570, 437 (QKV
//    and its RoPE), 6-22 TFLOP/s.
#include "common.cuh"
#include "kernels.h"

namespace zsaa {
namespace {

constexpr int FB = 64;       // tile edge: rows of A, weight rows
constexpr int FK = 16;       // k per stage
constexpr int FLD = FK + 4;  // A: shared-memory row stride, floats
constexpr int FWLD = FB + 4;  // weights: stride of one k's columns, floats
constexpr int FST = 3;       // stages of copies
constexpr int FG = 2;        // groups of two warps, each with its part of K
constexpr int FGT = 64;      // threads of a group
constexpr int FTHREADS = FG * FGT;
constexpr int FRED = FB + 4;  // row stride of the partial tile
constexpr int FA_STAGE = FB * FLD, FC_STAGE = FB * FK, FW_STAGE = FK * FWLD;
// a group's shared memory: stages of A, of the weights as copied (each thread's
// chunks side by side), two of the weights transposed
constexpr int F_COPY = FST * FA_STAGE, F_TRANS = F_COPY + FST * FC_STAGE, F_SMEM = F_TRANS + 2 * FW_STAGE;
static_assert(F_SMEM >= FB * FRED, "the partial tile reuses the stages");

struct F32Args {
  const float* A;
  int lda;
  TcWeights W;
  GemmParams p;
};

// cp.async of `bytes` valid ones out of SZ, the rest zero-filled.
template <int SZ>
__device__ __forceinline__ void cp_async_zfill(uint32_t dst, const float* src, bool valid) {
  const int n = valid ? SZ : 0;
  if constexpr (SZ == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// One group's barrier.
__device__ __forceinline__ void group_sync(int grp) { asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(FGT) : "memory"); }

// VEC: K, lda and every base allow 16-byte copies of A and W (else 4-byte ones).
template <int EPI, bool VEC>
__global__ void __launch_bounds__(FTHREADS, 3) gemm_f32_kernel(const F32Args a) {
  constexpr bool DUAL = EPI == kEpiSwiGLU;
  constexpr int NOUT = DUAL ? FB / 2 : FB;  // output columns of a tile
  extern __shared__ __align__(16) float smem[];
  pdl_trigger();
  const GemmParams& p = a.p;
  const int grp = threadIdx.x / FGT, tid = threadIdx.x % FGT, tx = tid & 7, ty = tid >> 3;
  float* sm = smem + grp * F_SMEM;
  const int S = static_cast<int>(cluster_size()), rank = static_cast<int>(cluster_rank());
  const int tn = blockIdx.x / S, m0 = blockIdx.y * FB;
  // Output column of tile column j.  RoPE pairs dims c and c + hd/2 of a head:
  // a tile holds whole heads (hd <= 64) or matching quarters of one (hd 128).
  auto col = [&](int j) {
    if (EPI == kEpiRope && p.hd == 128) return (tn >> 1) * 128 + (tn & 1) * 32 + (j & 31) + (j >> 5) * 64;
    return tn * NOUT + j;
  };
  // weight row of tile row r (nullptr past the last column)
  auto wrow = [&](int r) -> const float* {
    const int n = DUAL ? tn * NOUT + (r & (NOUT - 1)) : col(r);
    if (n >= p.N) return nullptr;
    const void* w;
    int nn = n;
    if (DUAL) {
      w = r < NOUT ? a.W.w0 : a.W.w1;
    } else if (n >= a.W.n2) {
      w = a.W.w2, nn = n - a.W.n2;
    } else if (n >= a.W.n1) {
      w = a.W.w1, nn = n - a.W.n1;
    } else {
      w = a.W.w0;
    }
    return static_cast<const float*>(w) + static_cast<size_t>(nn) * p.K;
  };

  const int KB = (p.K + FK - 1) / FK;
  const int part = rank * FG + grp, parts = S * FG;
  const int kb0 = static_cast<int>(static_cast<long long>(part) * KB / parts);
  const int kb1 = static_cast<int>(static_cast<long long>(part + 1) * KB / parts);
  // VEC: a thread copies 16-byte chunks: of A, chunk tid%4 of rows tid/4 + 16 i;
  // of the weights, chunk tid%2 + 2 warp of rows (tid%32)/2 + 16 i (whole
  // sectors, and the transposed stores of a warp hit 32 banks).  A row past the
  // matrix reads a valid one instead: its outputs are not stored.
  constexpr int RPT = 4;
  const int wr = (tid & 31) >> 1, wk = ((tid & 1) + 2 * (tid >> 5)) * 4;
  const float* srcA[RPT];
  const float* srcW[RPT];
  if (VEC) {
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      srcA[i] = a.A + static_cast<size_t>(min(m0 + (tid >> 2) + 16 * i, p.M - 1)) * a.lda + kb0 * FK + (tid & 3) * 4;
      const float* w = wrow(wr + 16 * i);
      srcW[i] = (w != nullptr ? w : static_cast<const float*>(a.W.w0)) + kb0 * FK + wk;
    }
  }
  const uint32_t sbase = smem_u32(sm), dA = sbase + (VEC ? ((tid >> 2) * FLD + (tid & 3) * 4) * 4 : 0);
  // A's block kb -> stage st; blocks are loaded in order, each advancing the pointers
  auto load_a = [&](int kb, int st) {
    if (VEC) {
      const bool kin = kb * FK + (tid & 3) * 4 < p.K;
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        cp_async_zfill<16>(dA + (st * FA_STAGE + 16 * i * FLD) * 4, srcA[i], kin);
        srcA[i] += FK;
      }
    } else {
      for (int i = tid; i < FB * FK; i += FGT) {
        const int r = i / FK, k = kb * FK + i % FK;
        const bool va = k < p.K && m0 + r < p.M;
        cp_async_zfill<4>(dA + (st * FA_STAGE + r * FLD + i % FK) * 4,
                          va ? a.A + static_cast<size_t>(m0 + r) * a.lda + k : a.A, va);
      }
    }
  };
  // VEC: the weights' block kb -> stage st as copied; later each thread moves its
  // own chunks to their transposed place.  Else straight to that place.
  auto copy_w = [&](int kb, int st) {
    if (VEC) {
      const bool kin = kb * FK + wk < p.K;
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        cp_async_zfill<16>(sbase + (F_COPY + st * FC_STAGE + (i * FGT + tid) * 4) * 4, srcW[i], kin);
        srcW[i] += FK;
      }
    } else {
      for (int i = tid; i < FB * FK; i += FGT) {
        const int r = i / FK, k = kb * FK + i % FK;
        const float* w = wrow(r);
        const bool vw = k < p.K && w != nullptr;
        cp_async_zfill<4>(sbase + (F_TRANS + st * FW_STAGE + (i % FK) * FWLD + r) * 4,
                          vw ? w + k : static_cast<const float*>(a.W.w0), vw);
      }
    }
  };
  auto transpose_w = [&](int st, int sw) {
    const float* c = sm + F_COPY + st * FC_STAGE + tid * 4;
    float* d = sm + F_TRANS + sw * FW_STAGE + wk * FWLD + wr;
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const float4 v = *reinterpret_cast<const float4*>(c + i * FGT * 4);
      float* q = d + 16 * i;
      q[0] = v.x, q[FWLD] = v.y, q[2 * FWLD] = v.z, q[3 * FWLD] = v.w;
    }
  };

  // a model's weights, which no kernel writes: the first blocks before waiting
  // for the previous kernel, their activations after
  auto first_w = [&] {
#pragma unroll
    for (int s = 0; s < (VEC ? FST - 1 : 1); ++s)
      if (kb0 + s < kb1) copy_w(kb0 + s, s);
  };
  if (p.w_const) first_w();
  pdl_wait();
  if (!p.w_const) first_w();
#pragma unroll
  for (int s = 0; s < FST - 1; ++s) {
    if (kb0 + s < kb1) load_a(kb0 + s, s);
    cp_async_commit();  // the first group holds the weights too
  }
  cp_async_wait<FST - 2>();
  if (VEC && kb0 < kb1) transpose_w(0, 0);
  uint64_t acc[8][4];  // rows ty + 8 i; columns 4 tx + {0, 1}, {2, 3}, 32 + 4 tx + {0, 1}, {2, 3}
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  int st = 0, sw = 0;
  for (int kb = kb0; kb < kb1; ++kb) {
    group_sync(grp);  // block kb is in place; every thread is done with the stages filled next
    const int nx = kb + FST - 1, nst = st == 0 ? FST - 1 : st - 1;
    if (nx < kb1) {
      load_a(nx, nst);
      if (VEC) copy_w(nx, nst);
    }
    if (!VEC && kb + 1 < kb1) copy_w(kb + 1, sw ^ 1);
    cp_async_commit();
    const float* pa = sm + st * FA_STAGE + ty * FLD;
    const float* pw = sm + F_TRANS + sw * FW_STAGE + 4 * tx;
#pragma unroll
    for (int k = 0; k < FK; k += 4) {
      float4 av[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) av[i] = *reinterpret_cast<const float4*>(pa + 8 * i * FLD + k);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(pw + (k + e) * FWLD);
        const ulonglong2 w1 = *reinterpret_cast<const ulonglong2*>(pw + (k + e) * FWLD + FB / 2);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float x = e == 0 ? av[i].x : e == 1 ? av[i].y : e == 2 ? av[i].z : av[i].w;
          const uint64_t xx = f2pack(x, x);
          acc[i][0] = ffma2(xx, w0.x, acc[i][0]);
          acc[i][1] = ffma2(xx, w0.y, acc[i][1]);
          acc[i][2] = ffma2(xx, w1.x, acc[i][2]);
          acc[i][3] = ffma2(xx, w1.y, acc[i][3]);
        }
      }
    }
    st = st == FST - 1 ? 0 : st + 1;
    sw ^= 1;
    cp_async_wait<VEC ? FST - 2 : 0>();
    if (VEC && kb + 1 < kb1) transpose_w(st, sw);
  }
  cp_async_wait<0>();
  group_sync(grp);
  // the group's partial tile -> its shared memory
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; j += 2)
      *reinterpret_cast<ulonglong2*>(sm + (ty + 8 * i) * FRED + 4 * tx + 16 * j) = make_ulonglong2(acc[i][j], acc[i][j + 1]);
  if (S > 1)
    cluster_sync_all();
  else
    __syncthreads();

  // CTA `rank` finishes rows [rank*64/S, (rank+1)*64/S): four columns a thread
  const int r0 = rank * FB / S, r1 = (rank + 1) * FB / S;
  const bool vec_out = (p.ldo & 3) == 0 && (p.N & 3) == 0 && (reinterpret_cast<uintptr_t>(p.out) & 15) == 0 &&
                       (EPI != kEpiResid || (reinterpret_cast<uintptr_t>(p.resid) & 15) == 0);
  auto sum4 = [&](int r, int c) {  // the partials of four neighbouring columns, in the order of their parts of K
    float4 v = *reinterpret_cast<const float4*>(smem + r * FRED + c);
    const float4 v1 = *reinterpret_cast<const float4*>(smem + F_SMEM + r * FRED + c);
    v.x += v1.x, v.y += v1.y, v.z += v1.z, v.w += v1.w;
    if (S > 1) {
      const uint32_t local = smem_u32(smem + r * FRED + c);
      v = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int q = 0; q < S * FG; ++q) {
        float4 t;
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w)
                     : "r"(map_rank(local + (q % FG) * F_SMEM * 4, q / FG))
                     : "memory");
        v.x += t.x, v.y += t.y, v.z += t.z, v.w += t.w;
      }
    }
    return v;
  };
  constexpr int C4 = NOUT / 4;  // column groups of a row
  for (int t = threadIdx.x; t < (r1 - r0) * C4; t += FTHREADS) {
    const int r = r0 + t / C4, c = (t % C4) * 4, m = m0 + r, n = col(c);
    if (m >= p.M || n >= p.N) continue;
    const float4 v4 = sum4(r, c);
    float v[4] = {v4.x, v4.y, v4.z, v4.w};
    if (DUAL) {
      const float4 u4 = sum4(r, c + NOUT);
      const float u[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = v[e] / (1.f + expf(-v[e])) * u[e];
    }
    if (EPI == kEpiRope && n < p.rope_cols) {  // hd is a power of two from 8 to 128
      const int half = p.hd == 128 ? 32 : p.hd / 2;  // distance of a pair within the tile
      const float4 o4 = sum4(r, c ^ half);
      const float o[4] = {o4.x, o4.y, o4.z, o4.w};
      const bool second = (c & half) != 0;
      const size_t tb = static_cast<size_t>(p.pos[m]) * (p.hd / 2) + (n & (p.hd / 2 - 1));
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float cs = p.cos_t[tb + e], sn = p.sin_t[tb + e];
        v[e] = second ? v[e] * cs + o[e] * sn : v[e] * cs - o[e] * sn;
      }
    }
    const size_t o = static_cast<size_t>(m) * p.ldo + n;
    float* out = static_cast<float*>(p.out) + o;
    if (vec_out) {
      if (EPI == kEpiResid) {
        const float4 r4 = *reinterpret_cast<const float4*>(static_cast<const float*>(p.resid) + o);
        v[0] += r4.x, v[1] += r4.y, v[2] += r4.z, v[3] += r4.w;
      }
      *reinterpret_cast<float4*>(out) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (n + e < p.N) out[e] = EPI == kEpiResid ? v[e] + static_cast<const float*>(p.resid)[o + e] : v[e];
    }
  }
  if (S > 1) cluster_sync_all();  // every CTA's partial has been read
}

int f32_sms() {
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

// Cluster size.  Measured over 67 shapes (d 64-4096, 24-5000 rows): a k-block of
// a tile takes about 1 us with up to three CTAs on an SM (0.5 us for a CTA with
// neighbouring SMs idle), three more double it, and a cluster of 2, 4, 8 adds
// 0.85, 1.75, 4 us to each round of CTAs for its reduction and its smaller
// parts' ramp.  The split this picks is within 2% of the best of the four on
// average.  The earlier rule took two CTAs for a full SM and no cost per round:
// it split 1536 x 4096 x 1024 eightfold (750 us for gate and up against 482) and
// left 1100 x 1024 x 4096 whole (283 us against 194).
int f32_split(long long tiles, int KB) {
  static const double extra[4] = {0.0, 0.85, 1.75, 4.0};
  int best = 1;
  double best_cost = 0.0;
  for (int i = 0, S = 1; i < 4 && S <= KB; ++i, S *= 2) {
    const long long per_sm = (tiles * S + f32_sms() - 1) / f32_sms();
    const double rounds = per_sm > 3 ? static_cast<double>(per_sm) / 3.0 : 1.0;
    const double cost = rounds * ((KB + S - 1) / S + extra[i] + 0.5);
    if (S == 1 || cost < best_cost) best = S, best_cost = cost;
  }
  return best;
}

template <int EPI, bool VEC>
cudaError_t run_f32(const F32Args& a, int tiles_n, int tiles_m, int S, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(tiles_n) * S, tiles_m);
  cfg.blockDim = dim3(FTHREADS);
  cfg.dynamicSmemBytes = FG * F_SMEM * sizeof(float);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = S;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  static OncePerDevice once;
  const cudaError_t e =
      set_smem_limit_once(once, gemm_f32_kernel<EPI, VEC>, static_cast<int>(cfg.dynamicSmemBytes));
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, gemm_f32_kernel<EPI, VEC>, a);
}

}  // namespace

bool gemm_f32_rope_supported(int hd) { return hd >= 8 && hd <= 128 && (hd & (hd - 1)) == 0; }

cudaError_t launch_gemm_f32(const float* A, int lda, const TcWeights& W, int epi, const GemmParams& p,
                            cudaStream_t s) {
  if (epi == kEpiRope && !gemm_f32_rope_supported(p.hd)) return cudaErrorInvalidValue;
  if (p.launches) *p.launches += 1;
  F32Args a{A, lda, W, p};
  const int nout = epi == kEpiSwiGLU ? FB / 2 : FB;
  const int tiles_n = (p.N + nout - 1) / nout, tiles_m = (p.M + FB - 1) / FB;
  const int S = f32_split(static_cast<long long>(tiles_n) * tiles_m, (p.K + FK - 1) / FK);
  bool vec = p.K % 4 == 0 && lda % 4 == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  for (const void* w : {W.w0, W.w1, W.w2}) vec = vec && (reinterpret_cast<uintptr_t>(w) & 15) == 0;
  switch (epi) {
    case kEpiSwiGLU: return vec ? run_f32<kEpiSwiGLU, true>(a, tiles_n, tiles_m, S, s) : run_f32<kEpiSwiGLU, false>(a, tiles_n, tiles_m, S, s);
    case kEpiResid: return vec ? run_f32<kEpiResid, true>(a, tiles_n, tiles_m, S, s) : run_f32<kEpiResid, false>(a, tiles_n, tiles_m, S, s);
    case kEpiRope: return vec ? run_f32<kEpiRope, true>(a, tiles_n, tiles_m, S, s) : run_f32<kEpiRope, false>(a, tiles_n, tiles_m, S, s);
    default: return vec ? run_f32<kEpiStore, true>(a, tiles_n, tiles_m, S, s) : run_f32<kEpiStore, false>(a, tiles_n, tiles_m, S, s);
  }
}

}  // namespace zsaa

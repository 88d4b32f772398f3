// fp32 CUDA-core GEMM for models stored in float32: out = epi(A[M,K] W[N,K]^T).
// True fp32 FMA (no TF32).  Epilogues: store, residual add, SwiGLU (two weight
// matrices, gate and up), RoPE (the QKV projection, read from its three
// weight matrices).
//
// What bounds it: the FMA pipe (about 76 TFLOP/s) once there are enough tiles,
// and the length of one tile's K chain when there are few.  So:
//  - 64 x 64 tiles of 64 threads, 8 x 8 outputs a thread.  Both operands stay
//    K-major in shared memory (rows of 16 k, padded to 20 floats: 16-byte
//    copies in, and a quarter warp's 16-byte reads hit distinct banks), so a
//    thread reads four k of a row at once and multiplies them as two packed
//    pairs (fma.rn.f32x2): an output's even and odd k accumulate separately
//    and are added at the end, which is no less exact than one chain.
//  - A three-stage cp.async ring per CTA; four CTAs share an SM.
//    A 4 x 4 output tile per thread, 4-byte staging and one stage at a time ran
//    at 6-22 TFLOP/s; this runs at 28-36 (d 1024, ffn 4096, 324-1536 rows: down
//    570 -> 145 us, gate/up 399 -> 247 us, QKV with RoPE 437 -> 91 us a launch).
//  - Few tiles: K is split over a thread-block cluster of S <= 8 CTAs, whose
//    partial tiles meet in distributed shared memory and are added in rank
//    order (deterministic).  S minimises CTAs per SM x k-blocks per CTA.
#include "common.cuh"
#include "kernels.h"

namespace zsaa {
namespace {

constexpr int FB = 64;       // tile edge: rows of A, weight rows
constexpr int FK = 16;       // k per stage
constexpr int FLD = FK + 4;  // shared-memory row stride, floats
constexpr int FST = 3;       // stages
constexpr int FTHREADS = 64;
constexpr int FRED = FB + 4;  // row stride of the partial tile
constexpr int F_STAGE = 2 * FB * FLD;
static_assert(FST * F_STAGE >= FB * FRED, "the partial tile reuses the ring");

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

// VEC: K, lda and every base allow 16-byte copies of A and W (else 4-byte ones).
template <int EPI, bool VEC>
__global__ void __launch_bounds__(FTHREADS, 4) gemm_f32_kernel(const F32Args a) {
  constexpr bool DUAL = EPI == kEpiSwiGLU;
  constexpr int NOUT = DUAL ? FB / 2 : FB;  // output columns of a tile
  __shared__ __align__(16) float sm[FST * F_STAGE];
  pdl_trigger();
  const GemmParams& p = a.p;
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
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
  const int kb0 = static_cast<int>(static_cast<long long>(rank) * KB / S);
  const int kb1 = static_cast<int>(static_cast<long long>(rank + 1) * KB / S);
  // VEC: a thread copies 16-byte chunk tid%4 of rows tid/4 + 16 i of both operands
  constexpr int RPT = 4;
  const float* srcA[RPT];
  const float* srcW[RPT];
  if (VEC) {
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int r = (tid >> 2) + 16 * i;
      srcA[i] = m0 + r < p.M ? a.A + static_cast<size_t>(m0 + r) * a.lda + (tid & 3) * 4 : nullptr;
      const float* w = wrow(r);
      srcW[i] = w != nullptr ? w + (tid & 3) * 4 : nullptr;
    }
  }
  const uint32_t sbase = smem_u32(sm);
  auto load = [&](int kb, int st, bool first, bool second) {  // first: the weights, second: A
    const uint32_t dA = sbase + st * F_STAGE * 4, dW = dA + FB * FLD * 4;
    if (VEC) {
      const int k = kb * FK;
      const bool kin = k + (tid & 3) * 4 < p.K;
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const uint32_t o = (((tid >> 2) + 16 * i) * FLD + (tid & 3) * 4) * 4;
        const bool va = kin && srcA[i] != nullptr, vw = kin && srcW[i] != nullptr;
        if (second) cp_async_zfill<16>(dA + o, va ? srcA[i] + k : a.A, va);
        if (first) cp_async_zfill<16>(dW + o, vw ? srcW[i] + k : static_cast<const float*>(a.W.w0), vw);
      }
    } else {
      for (int i = tid; i < FB * FK; i += FTHREADS) {
        const int r = i / FK, k = kb * FK + i % FK;
        const uint32_t o = (r * FLD + i % FK) * 4;
        const float* w = wrow(r);
        const bool va = k < p.K && m0 + r < p.M, vw = k < p.K && w != nullptr;
        if (second) cp_async_zfill<4>(dA + o, va ? a.A + static_cast<size_t>(m0 + r) * a.lda + k : a.A, va);
        if (first) cp_async_zfill<4>(dW + o, vw ? w + k : static_cast<const float*>(a.W.w0), vw);
      }
    }
  };

  // a model's weights, which no kernel writes: the first stages' rows before
  // waiting for the previous kernel, their activations after
  if (p.w_const) {
#pragma unroll
    for (int s = 0; s < FST - 1; ++s)
      if (kb0 + s < kb1) load(kb0 + s, s, true, false);
  }
  pdl_wait();
#pragma unroll
  for (int s = 0; s < FST - 1; ++s) {
    if (kb0 + s < kb1) load(kb0 + s, s, !p.w_const, true);
    cp_async_commit();  // group s holds stage s's activations (and, for s = 0, the weights)
  }
  uint64_t acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
  int st = 0;
  for (int kb = kb0; kb < kb1; ++kb) {
    cp_async_wait<FST - 2>();
    __syncthreads();  // stage st has landed; every thread is done with the stage filled next
    const int nx = kb + FST - 1;
    if (nx < kb1) load(nx, st == 0 ? FST - 1 : st - 1, true, true);
    cp_async_commit();
    const float* sa = sm + st * F_STAGE + ty * FLD;
    const float* sw = sm + st * F_STAGE + FB * FLD + tx * FLD;
#pragma unroll
    for (int k = 0; k < FK; k += 4) {
      ulonglong2 av[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) av[i] = *reinterpret_cast<const ulonglong2*>(sa + 8 * i * FLD + k);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const ulonglong2 wv = *reinterpret_cast<const ulonglong2*>(sw + 8 * j * FLD + k);
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i][j] = ffma2(av[i].y, wv.y, ffma2(av[i].x, wv.x, acc[i][j]));
      }
    }
    st = st == FST - 1 ? 0 : st + 1;
  }
  cp_async_wait<0>();
  __syncthreads();
  // this CTA's partial tile -> its shared memory
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float e, o;
      f2unpack(acc[i][j], e, o);
      sm[(ty + 8 * i) * FRED + tx + 8 * j] = e + o;
    }
  if (S > 1)
    cluster_sync_all();
  else
    __syncthreads();

  // CTA `rank` finishes rows [rank*64/S, (rank+1)*64/S): four columns a thread
  const int r0 = rank * FB / S, r1 = (rank + 1) * FB / S;
  const bool vec_out = (p.ldo & 3) == 0 && (p.N & 3) == 0 && (reinterpret_cast<uintptr_t>(p.out) & 15) == 0 &&
                       (EPI != kEpiResid || (reinterpret_cast<uintptr_t>(p.resid) & 15) == 0);
  auto sum4 = [&](int r, int c) {  // the S partials of four neighbouring columns, in rank order
    float4 v = *reinterpret_cast<const float4*>(sm + r * FRED + c);
    if (S > 1) {
      const uint32_t local = smem_u32(sm + r * FRED + c);
      v = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int q = 0; q < S; ++q) {
        float4 t;
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w)
                     : "r"(map_rank(local, q))
                     : "memory");
        v.x += t.x, v.y += t.y, v.z += t.z, v.w += t.w;
      }
    }
    return v;
  };
  constexpr int C4 = NOUT / 4;  // column groups of a row
  for (int t = tid; t < (r1 - r0) * C4; t += FTHREADS) {
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

// Cluster size: an SM runs two CTAs at full FMA rate (a lone one uses half of
// it), so the time is about max(1, CTAs per SM / 2) x k-blocks per CTA
// (0.5 us each), plus about 1 us for a cluster's reduction.
int f32_split(long long tiles, int KB) {
  int best = 1;
  double best_cost = 0.0;
  for (int S = 1; S <= 8 && S <= KB; S *= 2) {
    const long long per_sm = (tiles * S + f32_sms() - 1) / f32_sms();
    const double waves = per_sm > 2 ? 0.5 * static_cast<double>(per_sm) : 1.0;
    const double cost = waves * ((KB + S - 1) / S) * 0.5 + (S > 1 ? 1.0 : 0.0);
    if (S == 1 || cost < best_cost) best = S, best_cost = cost;
  }
  return best;
}

template <int EPI, bool VEC>
cudaError_t run_f32(const F32Args& a, int tiles_n, int tiles_m, int S, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(tiles_n) * S, tiles_m);
  cfg.blockDim = dim3(FTHREADS);
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

// fp32 attention (Eq. 1) and soft-score column mass (Sec. 3.2) on the CUDA
// cores, for models stored in float32 with heads of 32, 64 or 128 dims.
//
// Both are bound by the FMA pipe, so both are register-tiled: 128 threads hold
// a tile of 8 R rows by 64 columns of S (R x 4 scores a thread), operands stay
// dim-major in shared memory (rows padded by 4 floats: a quarter warp's
// 16-byte reads hit distinct banks) and the products run as packed pairs of
// dims (fma.rn.f32x2).
//   attention: rows are queries, columns the keys of one block; online softmax
//     in the log2 domain, O in registers (R rows x HD/16 dims a thread).  The
//     next key block's copy runs under the softmax and P V, the next value
//     block's under the next scores.
//   column mass: rows are keys, columns the queries of one block; one CTA per
//     key tile and query head writes that head's partial column sums
//     (optionally times ||v_key||), and the reader adds a group's heads in order.
// One warp per row, reading every key from L2 for each query, ran at about
// 0.5 TFLOP/s: 953 us of attention and 353 us of column mass a layer (B 4, 16
// heads of 64, 81-384 rows); the tiles take 35 and 31 us.
// R is the largest of 8, 4, 2 that still gives two CTAs per SM: short
// sequences take smaller tiles instead of leaving most SMs idle.
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace zsaa {
namespace {

constexpr int AF_THREADS = 128;
constexpr int AF_COLS = 64;  // keys (attention) or queries (column mass) per block

template <int HD>
constexpr int af_ld() { return HD + 4; }
constexpr int AF_PLD = AF_COLS + 4;

template <int HD, int R>
constexpr size_t af_attn_smem() {
  return sizeof(float) * ((8 * R + 2 * AF_COLS) * static_cast<size_t>(af_ld<HD>()) + 8 * R * AF_PLD);
}
template <int HD, int R>
constexpr size_t af_mass_smem() {
  return sizeof(float) * ((8 * R + 2 * AF_COLS) * static_cast<size_t>(af_ld<HD>()) + 2 * AF_COLS);
}

// cp.async rows [row0, row0 + rows) of one head (HD floats each, ld apart) into
// a padded tile; rows at or past n are zero-filled.
template <int HD>
__device__ __forceinline__ void af_load(float* tile, const float* g, size_t ld, int row0, int rows, int n) {
  constexpr int CH = HD / 4;
  for (int i = threadIdx.x; i < rows * CH; i += AF_THREADS) {
    const int r = i / CH, c = (i % CH) * 4;
    const bool v = row0 + r < n;
    cp_async16(smem_u32(tile + r * af_ld<HD>() + c), g + (v ? static_cast<size_t>(row0 + r) * ld : 0) + c, v);
  }
}

// s[i][j] = <row ty + 8 i of X, row tx + 16 j of Y>
template <int HD, int R>
__device__ __forceinline__ void af_scores(const float* X, const float* Y, int tx, int ty, float (&s)[R][4]) {
  uint64_t acc[R][4];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  const float* x = X + ty * af_ld<HD>();
  const float* y = Y + tx * af_ld<HD>();
#pragma unroll 4
  for (int d = 0; d < HD; d += 4) {
    ulonglong2 yv[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) yv[j] = *reinterpret_cast<const ulonglong2*>(y + 16 * j * af_ld<HD>() + d);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(x + 8 * i * af_ld<HD>() + d);
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = ffma2(xv.y, yv[j].y, ffma2(xv.x, yv[j].x, acc[i][j]));
    }
  }
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float e, o;
      f2unpack(acc[i][j], e, o);
      s[i][j] = e + o;
    }
}

template <int HD, int R>
__global__ void __launch_bounds__(AF_THREADS)
    attn_f32_tile_kernel(const float* __restrict__ qkv, int N, int Hq, int Hkv, float* __restrict__ out,
                         float* __restrict__ lse2, float scale_log2, int causal) {
  pdl_trigger();
  pdl_wait();
  qkv = after_wait(qkv);
  constexpr int BQ = 8 * R, LD = af_ld<HD>();
  constexpr int NP = HD / 32;  // pairs of output dims a thread owns per row
  extern __shared__ __align__(16) float sm[];
  float* sQ = sm;
  float* sK = sQ + BQ * LD;
  float* sV = sK + AF_COLS * LD;
  float* sP = sV + AF_COLS * LD;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int qb = gridDim.x - 1 - blockIdx.x;  // the longest causal rows first
  const int h = blockIdx.y, b = blockIdx.z, g = h / (Hq / Hkv);
  const size_t ld = static_cast<size_t>(Hq + 2 * Hkv) * HD;
  const float* base = qkv + static_cast<size_t>(b) * N * ld;
  const float* Kg = base + (Hq + g) * HD;
  const float* Vg = base + (Hq + Hkv + g) * HD;
  const int q0 = qb * BQ;
  const int n_keys = causal ? min(N, q0 + BQ) : N;
  const int n_kb = (n_keys + AF_COLS - 1) / AF_COLS;
  af_load<HD>(sQ, base + h * HD, ld, q0, BQ, N);
  af_load<HD>(sK, Kg, ld, 0, AF_COLS, N);
  cp_async_commit();
  af_load<HD>(sV, Vg, ld, 0, AF_COLS, N);
  cp_async_commit();

  uint64_t o[R][NP];
  float m[R], l[R];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
#pragma unroll
    for (int c = 0; c < NP; ++c) o[i][c] = 0ull;
  }
  for (int kb = 0; kb < n_kb; ++kb) {
    const int k0 = kb * AF_COLS;
    cp_async_wait<1>();
    __syncthreads();  // K of this block has landed
    float s[R][4];
    af_scores<HD, R>(sQ, sK, tx, ty, s);
    __syncthreads();  // every thread is done with K
    if (kb + 1 < n_kb) af_load<HD>(sK, Kg, ld, k0 + AF_COLS, AF_COLS, N);
    cp_async_commit();
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int q = q0 + ty + 8 * i;
      const int lim = causal ? min(N, q + 1) : N;  // keys [0, lim) are visible
      float mx = m[i];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        s[i][j] = k0 + tx + 16 * j < lim ? s[i][j] * scale_log2 : -INFINITY;
        mx = fmaxf(mx, s[i][j]);
      }
#pragma unroll
      for (int x = 8; x > 0; x >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
      const float f = exp2f(m[i] - mx);  // 0 on the first block: key 0 is visible to every row
      m[i] = mx;
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float p = exp2f(s[i][j] - mx);
        sum += p;
        sP[(ty + 8 * i) * AF_PLD + tx + 16 * j] = p;
      }
#pragma unroll
      for (int x = 8; x > 0; x >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, x);
      l[i] = fmaf(l[i], f, sum);
      const uint64_t f2 = f2pack(f, f);
#pragma unroll
      for (int c = 0; c < NP; ++c) o[i][c] = ffma2(o[i][c], f2, 0ull);
    }
    cp_async_wait<1>();
    __syncthreads();  // V of this block has landed (and this block's P rows are written)
    // O += P V of keys k..k+3, of row i the first vis + 8 i keys of the block
    auto add4 = [&](int k, int vis, auto edge) {
      uint64_t v[4][NP];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float* vr = sV + (k + e) * LD;
        if constexpr (NP == 1) {
          v[e][0] = *reinterpret_cast<const uint64_t*>(vr + 2 * tx);
        } else {
#pragma unroll
          for (int c = 0; c < NP; c += 2) {
            const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(vr + 32 * c + 4 * tx);
            v[e][c] = t.x;
            v[e][c + 1] = t.y;
          }
        }
      }
#pragma unroll
      for (int i = 0; i < R; ++i) {
        if (edge && k >= vis + 8 * i) continue;
        const float4 p4 = *reinterpret_cast<const float4*>(sP + (ty + 8 * i) * AF_PLD + k);
        const uint64_t p2[4] = {f2pack(p4.x, p4.x), f2pack(p4.y, p4.y), f2pack(p4.z, p4.z), f2pack(p4.w, p4.w)};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (edge && k + e >= vis + 8 * i) continue;
#pragma unroll
          for (int c = 0; c < NP; ++c) o[i][c] = ffma2(p2[e], v[e][c], o[i][c]);
        }
      }
    };
    // keys that every row sees (V past the sequence's end is zero), then those on
    // the diagonal: a hidden key's P is 0, but its V need not be finite, so its
    // products are left out
    const int all = causal ? max(0, min(AF_COLS, q0 + 1 - k0)) & ~3 : AF_COLS;
#pragma unroll 2
    for (int k = 0; k < all; k += 4) add4(k, 0, std::false_type());
#pragma unroll 2
    for (int k = all; k < min(AF_COLS, q0 + BQ - k0); k += 4) add4(k, q0 + ty + 1 - k0, std::true_type());
    __syncthreads();  // every thread is done with V and P
    if (kb + 1 < n_kb) af_load<HD>(sV, Vg, ld, k0 + AF_COLS, AF_COLS, N);
    cp_async_commit();
  }
  cp_async_wait<0>();
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int q = q0 + ty + 8 * i;
    if (q >= N) continue;
    float* orow = out + (static_cast<size_t>(b) * N + q) * Hq * HD + h * HD;
    const float inv = 1.f / l[i];
    float v[2 * NP];
#pragma unroll
    for (int c = 0; c < NP; ++c) {
      f2unpack(o[i][c], v[2 * c], v[2 * c + 1]);
      v[2 * c] *= inv;
      v[2 * c + 1] *= inv;
    }
    if constexpr (NP == 1) {
      orow[2 * tx] = v[0];
      orow[2 * tx + 1] = v[1];
    } else {
#pragma unroll
      for (int c = 0; c < NP; c += 2)
#pragma unroll
        for (int e = 0; e < 4; ++e) orow[32 * c + 4 * tx + e] = v[2 * c + e];
    }
    if (tx == 0) lse2[(static_cast<size_t>(b) * Hq + h) * N + q] = m[i] + log2f(l[i]);
  }
}

template <int HD, int R>
__global__ void __launch_bounds__(AF_THREADS)
    colmass_f32_tile_kernel(const float* __restrict__ qkv, const float* __restrict__ lse2, int N, int Hq,
                            int Hkv, int B, int weight_vnorm, float* __restrict__ parts, float scale_log2,
                            int causal) {
  pdl_trigger();
  pdl_wait();
  qkv = after_wait(qkv);
  lse2 = after_wait(lse2);
  constexpr int BK = 8 * R, LD = af_ld<HD>();
  extern __shared__ __align__(16) float sm[];
  float* sK = sm;
  float* sQ = sK + BK * LD;                // [2] query blocks
  float* sL = sQ + 2 * AF_COLS * LD;       // [2] their normalisers
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int kb = blockIdx.x, h = blockIdx.y, b = blockIdx.z;  // early keys (most queries) first
  const int per = Hq / Hkv, g = h / per, hh = h % per;
  const size_t ld = static_cast<size_t>(Hq + 2 * Hkv) * HD;
  const float* base = qkv + static_cast<size_t>(b) * N * ld;
  const float* L = lse2 + (static_cast<size_t>(b) * Hq + h) * N;
  const int j0 = kb * BK;
  const int qb0 = causal ? j0 / AF_COLS : 0, n_qb = (N + AF_COLS - 1) / AF_COLS;
  auto issue = [&](int qb, int buf) {
    af_load<HD>(sQ + buf * AF_COLS * LD, base + h * HD, ld, qb * AF_COLS, AF_COLS, N);
    if (tid < AF_COLS) {
      const int q = qb * AF_COLS + tid;
      sL[buf * AF_COLS + tid] = q < N ? L[q] : 0.f;
    }
  };
  af_load<HD>(sK, base + (Hq + g) * HD, ld, j0, BK, N);
  issue(qb0, 0);
  cp_async_commit();
  float acc[R];
#pragma unroll
  for (int i = 0; i < R; ++i) acc[i] = 0.f;
  for (int qb = qb0; qb < n_qb; ++qb) {
    const int buf = (qb - qb0) & 1;
    if (qb + 1 < n_qb) issue(qb + 1, buf ^ 1);  // its last readers passed the barrier below
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    float s[R][4];
    af_scores<HD, R>(sK, sQ + buf * AF_COLS * LD, tx, ty, s);
    const int q0 = qb * AF_COLS;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int q = q0 + tx + 16 * j;
      const float lq = sL[buf * AF_COLS + tx + 16 * j];
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (q < N && (!causal || q >= j0 + ty + 8 * i)) acc[i] += exp2f(fmaf(s[i][j], scale_log2, -lq));
    }
    __syncthreads();
  }
  cp_async_wait<0>();
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int j = j0 + ty + 8 * i;
    float v = acc[i], ss = 0.f;
    if (weight_vnorm && j < N) {
      const float* vr = base + static_cast<size_t>(j) * ld + (Hq + Hkv + g) * HD;
      for (int e = tx; e < HD; e += 16) ss = fmaf(vr[e], vr[e], ss);
    }
#pragma unroll
    for (int x = 8; x > 0; x >>= 1) {
      v += __shfl_xor_sync(0xffffffffu, v, x);
      ss += __shfl_xor_sync(0xffffffffu, ss, x);
    }
    if (weight_vnorm) v *= sqrtf(ss);
    if (tx == 0 && j < N) parts[((static_cast<size_t>(hh) * B + b) * Hkv + g) * N + j] = v;
  }
}

int af_sms() {
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

// Rows per thread: the largest tile that still gives two CTAs per SM.
int af_rows(int N, int heads) {
  for (int R = 8; R > 2; R /= 2)
    if (static_cast<long long>((N + 8 * R - 1) / (8 * R)) * heads >= 2LL * af_sms()) return R;
  return 2;
}

template <int HD, int R>
cudaError_t run_attn(const float* qkv, int B, int N, int Hq, int Hkv, float* out, float* lse, float scale,
                     int causal, cudaStream_t s) {
  static OncePerDevice once;
  const cudaError_t e = set_smem_limit_once(once, attn_f32_tile_kernel<HD, R>, static_cast<int>(af_attn_smem<HD, R>()));
  if (e != cudaSuccess) return e;
  ZSAA_LAUNCH(attn_f32_tile_kernel<HD, R>, dim3((N + 8 * R - 1) / (8 * R), Hq, B), dim3(AF_THREADS),
              (af_attn_smem<HD, R>()), s, qkv, N, Hq, Hkv, out, lse, scale, causal);
  return cudaGetLastError();
}

template <int HD, int R>
cudaError_t run_mass(const float* qkv, const float* lse, int B, int N, int Hq, int Hkv, int weight_vnorm,
                     float* parts, float scale, int causal, cudaStream_t s) {
  static OncePerDevice once;
  const cudaError_t e = set_smem_limit_once(once, colmass_f32_tile_kernel<HD, R>, static_cast<int>(af_mass_smem<HD, R>()));
  if (e != cudaSuccess) return e;
  ZSAA_LAUNCH(colmass_f32_tile_kernel<HD, R>, dim3((N + 8 * R - 1) / (8 * R), Hq, B), dim3(AF_THREADS),
              (af_mass_smem<HD, R>()), s, qkv, lse, N, Hq, Hkv, B, weight_vnorm, parts, scale, causal);
  return cudaGetLastError();
}

template <int HD>
cudaError_t attn_rows(int R, const float* qkv, int B, int N, int Hq, int Hkv, float* out, float* lse, float scale,
                      int causal, cudaStream_t s) {
  switch (R) {
    case 8: return run_attn<HD, 8>(qkv, B, N, Hq, Hkv, out, lse, scale, causal, s);
    case 4: return run_attn<HD, 4>(qkv, B, N, Hq, Hkv, out, lse, scale, causal, s);
    default: return run_attn<HD, 2>(qkv, B, N, Hq, Hkv, out, lse, scale, causal, s);
  }
}

template <int HD>
cudaError_t mass_rows(int R, const float* qkv, const float* lse, int B, int N, int Hq, int Hkv, int wv,
                      float* parts, float scale, int causal, cudaStream_t s) {
  switch (R) {
    case 8: return run_mass<HD, 8>(qkv, lse, B, N, Hq, Hkv, wv, parts, scale, causal, s);
    case 4: return run_mass<HD, 4>(qkv, lse, B, N, Hq, Hkv, wv, parts, scale, causal, s);
    default: return run_mass<HD, 2>(qkv, lse, B, N, Hq, Hkv, wv, parts, scale, causal, s);
  }
}

}  // namespace

bool attention_f32_tiled(const void* qkv, int hd) {
  return (hd == 32 || hd == 64 || hd == 128) && (reinterpret_cast<uintptr_t>(qkv) & 15) == 0;
}

cudaError_t launch_attention_f32_tiled(const float* qkv, int B, int N, int Hq, int Hkv, int hd, float* out,
                                       float* lse, float scale_log2, int causal, cudaStream_t s) {
  const int R = af_rows(N, Hq * B);
  switch (hd) {
    case 32: return attn_rows<32>(R, qkv, B, N, Hq, Hkv, out, lse, scale_log2, causal, s);
    case 64: return attn_rows<64>(R, qkv, B, N, Hq, Hkv, out, lse, scale_log2, causal, s);
    case 128: return attn_rows<128>(R, qkv, B, N, Hq, Hkv, out, lse, scale_log2, causal, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_colmass_f32_tiled(const float* qkv, const float* lse, int B, int N, int Hq, int Hkv, int hd,
                                     int weight_vnorm, float* parts, int* n_chunks, float scale_log2, int causal,
                                     cudaStream_t s) {
  *n_chunks = Hq / Hkv;
  const int R = af_rows(N, Hq * B);
  switch (hd) {
    case 32: return mass_rows<32>(R, qkv, lse, B, N, Hq, Hkv, weight_vnorm, parts, scale_log2, causal, s);
    case 64: return mass_rows<64>(R, qkv, lse, B, N, Hq, Hkv, weight_vnorm, parts, scale_log2, causal, s);
    case 128: return mass_rows<128>(R, qkv, lse, B, N, Hq, Hkv, weight_vnorm, parts, scale_log2, causal, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace zsaa

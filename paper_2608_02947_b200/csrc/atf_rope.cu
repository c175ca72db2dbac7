// atf_rope: half-split rotary embedding in place (Sec. 3.1).  Memory-bound elementwise pass;
// the angle pos*theta_r, its sine/cosine and the rotation are evaluated in fp64 so that the
// result is the correctly rounded bf16 of the exact rotation even at positions ~2^20.
#include <algorithm>

#include "atf_common.cuh"

struct RopeTheta {
  double t[ATF_MAX_PAIRS];
};

// Eight consecutive elements of a row as fp64, and back with one rounding.
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&v)[8]) {
  const uint4 w = *reinterpret_cast<const uint4*>(p);
  const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = bf16lo_to_f32(u[i]);
    v[2 * i + 1] = bf16hi_to_f32(u[i]);
  }
}
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(p);
  *reinterpret_cast<float4*>(v + 4) = *reinterpret_cast<const float4*>(p + 4);
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const double (&v)[8]) {
  uint4 w;
  __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(&w);
#pragma unroll
  for (int i = 0; i < 8; ++i) o[i] = __double2bfloat16(v[i]);
  *reinterpret_cast<uint4*>(p) = w;
}
__device__ __forceinline__ void store8(float* p, const double (&v)[8]) {
  float o[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) o[i] = (float)v[i];
  *reinterpret_cast<float4*>(p) = *reinterpret_cast<const float4*>(o);
  *reinterpret_cast<float4*>(p + 4) = *reinterpret_cast<const float4*>(o + 4);
}

// In place, X bf16 or (for the split-precision prefill, whose point is that the rotated values are never rounded to
// bf16) fp32.  A block owns a few rows of every head and HL threads walk the heads of a row segment (eight pairs: 16
// bytes of each half row), every HL-th each.  The angles of a segment are evaluated once, in fp64: by its thread (HL = 1)
// or spread over the block's threads into shared memory.  For long rows memory bounds the pass (24 heads x 131072 x
// 128: 276 us, 5.8 TB/s).  For short ones HL fills the GPU; spreading the heads over blocks instead, each with the
// angles evaluated again, made the fp64 pipe the bound: 24 heads x 8192 x 128 23.2 -> 18.0 us, 8 heads 15.3 -> 8.5 us,
// 24 heads x 2048 12.8 -> 7.1 us.
// SPREAD: the heads are dealt over gridDim.y blocks as well, for rows too few to fill the GPU.
// PRE: the next head's segment is loaded before this one is stored, for fp32 data that L2 does not hold.
constexpr int ROPE_THREADS = 256;
template <int D, int HL, typename T, bool SPREAD = false, bool PRE = false>
__global__ void __launch_bounds__(ROPE_THREADS) atf_rope_kernel(T* X, int BH, int64_t N, int64_t pos0,
                                                                const __grid_constant__ RopeTheta theta) {
  constexpr int H = D / 2;
  constexpr int CHUNKS = H / 8;                         // segments of 8 pairs per row
  constexpr int SEGS = ROPE_THREADS / HL;               // (row, segment) pairs of the block
  constexpr int ROWS = SEGS / CHUNKS;
  const int64_t row0 = (int64_t)blockIdx.x * ROWS;
  grid_dependency_launch();
  const int sg = threadIdx.x % SEGS, c = sg % CHUNKS;
  const int64_t n = row0 + sg / CHUNKS;
  double cs[8], sn[8];
  if constexpr (HL == 1) {  // every thread has a segment of its own: no detour
    if (n >= N) return;
#pragma unroll
    for (int i = 0; i < 8; ++i) sincos((double)(pos0 + n) * theta.t[c * 8 + i], &sn[i], &cs[i]);
  } else {
    __shared__ double2 cs_sh[8 * SEGS];  // (cos, sin) of pair i of segment s at i * SEGS + s
#pragma unroll 1
    for (int k = threadIdx.x; k < 8 * SEGS; k += ROPE_THREADS) {
      const int i = k / SEGS, s = k % SEGS;
      double2 v;
      sincos((double)(pos0 + row0 + s / CHUNKS) * theta.t[(s % CHUNKS) * 8 + i], &v.y, &v.x);
      cs_sh[k] = v;
    }
    __syncthreads();
    if (n >= N) return;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const double2 v = cs_sh[i * SEGS + sg];
      cs[i] = v.x;
      sn[i] = v.y;
    }
  }
  auto rotate = [&](T* row, const float (&lo)[8], const float (&hi)[8]) {
    double olo[8], ohi[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const double a = (double)lo[i], b = (double)hi[i];
      olo[i] = a * cs[i] - b * sn[i];
      ohi[i] = b * cs[i] + a * sn[i];
    }
    store8(row, olo);
    store8(row + H, ohi);
  };
  grid_dependency_wait();  // the angles need nothing of the kernel before; X, not __restrict__, is touched behind this alone
  const int64_t head = N * D;
  const int lane = threadIdx.x / SEGS;
  const int first = SPREAD ? (int)blockIdx.y * HL + lane : lane, step = SPREAD ? HL * (int)gridDim.y : HL;
  T* row = X + ((int64_t)first * N + n) * D + c * 8;
  float lo[8], hi[8];
  if constexpr (PRE) {
    if (first >= BH) return;
    load8(row, lo);
    load8(row + H, hi);
  }
  for (int bh = first; bh < BH; bh += step, row += step * head) {
    if constexpr (PRE) {
      float lo2[8], hi2[8];
      if (bh + step < BH) {
        load8(row + step * head, lo2);
        load8(row + step * head + H, hi2);
      }
      rotate(row, lo, hi);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        lo[i] = lo2[i];
        hi[i] = hi2[i];
      }
    } else {
      load8(row, lo);
      load8(row + H, hi);
      rotate(row, lo, hi);
    }
  }
}

// Threads per row segment: one as long as that gives four blocks (fp32: eight, its rows are twice as long) for each SM, more
// for shorter rows; more threads than heads (they share the angles' evaluation only) below two blocks.  Eight threads walk
// at least every eighth head, one round trip to memory each; rows that do not give three blocks for each SM then have
// their heads dealt over blocks too, each with the angles evaluated again (d = 128, bf16, us, without -> with: 192 heads x 1 row, the queries of a decode step, 13.2 -> 2.4; 1536 x 1 91 -> 2.9; 2048 x 33
// 127 -> 9.3; 192 x 128 14.5 -> 4.4; 192 x 512 14.7 -> 10.5; 24 x 128 3.6 -> 2.6).
// fp32 moves twice the bytes an angle and is bound by the loads in flight: the heads are dealt over twelve blocks for each SM
// (192 heads x 512 20.6 -> 18, 100 x 1500 29 -> 26).  Past the 126 MB of L2 a thread waits for DRAM between its heads unless
// the next one is on its way (192 heads x 2048 96 -> 69 us, 24 x 32768 200 -> 132, 24 x 131072 603 -> 504); smaller
// data is slower so (24 x 8192 31.6 -> 33.0), and so is bf16 (24 x 131072 272 -> 306).
template <int D, typename T>
static cudaError_t launch_rope(T* X, int BH, int64_t N, int64_t pos0, const RopeTheta& th, cudaStream_t s) {
  constexpr bool F32 = sizeof(T) == 4;
  const auto blocks = [&](int lanes) { return (N + ROPE_THREADS / lanes / (D / 16) - 1) / (ROPE_THREADS / lanes / (D / 16)); };
  int hl = 1;
  while (hl < 8 && blocks(hl) < (2 * hl > BH ? 2 : 2 * (int)sizeof(T)) * 148) hl *= 2;
  const bool pre = F32 && (double)BH * (double)N * D * sizeof(T) > 126e6 && blocks(hl) >= 3 * 148;
  if (F32 && !pre)
    while (hl < 8 && 2 * hl <= BH) hl *= 2;
  const unsigned g = (unsigned)blocks(hl), want = (F32 ? 12 : 3) * 148;
  if (!pre && hl == 8 && BH > 8 && g < want) {
    const unsigned gy = std::min(((unsigned)BH + 7) / 8, (want + g - 1) / g);
    return atf_launch_overlapped(atf_rope_kernel<D, 8, T, true>, dim3(g, gy), ROPE_THREADS, 0, s, X, BH, N, pos0, th);
  }
  void (*kern)(T*, int, int64_t, int64_t, RopeTheta);
  if (hl == 1) kern = pre ? atf_rope_kernel<D, 1, T, false, F32> : atf_rope_kernel<D, 1, T>;
  else if (hl == 2) kern = pre ? atf_rope_kernel<D, 2, T, false, F32> : atf_rope_kernel<D, 2, T>;
  else if (hl == 4) kern = pre ? atf_rope_kernel<D, 4, T, false, F32> : atf_rope_kernel<D, 4, T>;
  else kern = pre ? atf_rope_kernel<D, 8, T, false, F32> : atf_rope_kernel<D, 8, T>;
  return atf_launch_overlapped(kern, dim3(g), ROPE_THREADS, 0, s, X, BH, N, pos0, th);
}

template <typename T>
static atf_status rope(const char* who, T* X, int B, int H, int64_t N, int d, const double* theta, int64_t pos0, void* stream) {
  if (!X || !theta) return atf_fail(ATF_ERR_INVALID_ARG, "%s: null pointer", who);
  if (d != 64 && d != 128) return atf_fail(ATF_ERR_UNSUPPORTED, "%s: d must be 64 or 128 (got %d)", who, d);
  if (B < 1 || H < 1 || N < 1 || pos0 < 0) return atf_fail(ATF_ERR_INVALID_ARG, "%s: bad shape", who);
  if ((uintptr_t)X & 15) return atf_fail(ATF_ERR_INVALID_ARG, "%s: X must be 16-byte aligned", who);
  RopeTheta th;
  for (int r = 0; r < d / 2; ++r) th.t[r] = theta[r];
  for (int r = d / 2; r < ATF_MAX_PAIRS; ++r) th.t[r] = 0.0;
  if ((N * (d / 16) + 255) / 256 > 0x7FFFFFFF) return atf_fail(ATF_ERR_UNSUPPORTED, "%s: N too large", who);
  ATF_CUDA_CHECK(d == 64 ? launch_rope<64>(X, B * H, N, pos0, th, (cudaStream_t)stream)
                         : launch_rope<128>(X, B * H, N, pos0, th, (cudaStream_t)stream));
  return ATF_OK;
}

extern "C" atf_status atf_rope_f32(float* X, int B, int H, int64_t N, int d, const double* theta, int64_t pos0, void* stream) {
  return rope("atf_rope_f32", X, B, H, N, d, theta, pos0, stream);
}

extern "C" atf_status atf_rope(void* X, int B, int H, int64_t N, int d, const double* theta, int64_t pos0, void* stream) {
  return rope("atf_rope", (__nv_bfloat16*)X, B, H, N, d, theta, pos0, stream);
}

// Launch interface of the one-tile-per-CTA prefill pipeline (atf_prefill_pipe.cu); the host code of
// atf_prefill.cu and atf_prefill_split.cu (validation, pre-pass, tensor maps) calls it.
#pragma once

#include "atf_common.cuh"

struct AtfPipeParams {
  uint32_t* sched;            // band schedule, 8 words per tile distance, ceil(N / 128) distances; written per launch
  const __nv_bfloat16* Q;      // the caller's rows, [B*Hq, Nq, D] (not in the split-precision mode)
  const __nv_bfloat16* Qhi;    // split-precision mode: pair-interleaved parts of Q, [B*Hq, Nq, D]
  const __nv_bfloat16* Qlo;
  __nv_bfloat16* O;
  float* LSE;
  unsigned long long* kept;
  unsigned int* status;
  int Hq, Hkv;
  int N;   // number of keys; positions 0..N-1
  int Nq;  // number of query rows: the last Nq positions
};

atf_status atf_launch_prefill_pipe(const CUtensorMap& tk, const CUtensorMap& tv, const AtfPipeParams& P,
                                   const AtfTable& t, int B, int d, int mode, bool count, cudaStream_t s);
// Split-precision mode: Q and K as hi and lo parts, S = Q_hi K_hi^T + Q_hi K_lo^T + Q_lo K_hi^T.
atf_status atf_launch_prefill_pipe_split(const CUtensorMap& tqh, const CUtensorMap& tql, const CUtensorMap& tkh,
                                         const CUtensorMap& tkl, const CUtensorMap& tv, const AtfPipeParams& P,
                                         const AtfTable& t, int B, int d, int mode, bool count, cudaStream_t s);

// The pre-pass of a prefill (layout of K and the band schedule) is one launch of blocks of this many threads: the first
// atf_sched_blocks() write the schedule, the others move rows.
constexpr int ATF_PREP_THREADS = 256;
inline int atf_sched_blocks(int64_t N) { return (int)(((N + 127) / 128 + ATF_PREP_THREADS / 8 - 1) / (ATF_PREP_THREADS / 8)); }

#ifdef __CUDACC__
// A schedule word: an ordinary load that stays behind the wait.  The pre-pass may still be writing when the kernel that
// reads starts, and the read-only path (__ldg) is defined only for what nothing writes while that kernel is resident.
__device__ __forceinline__ uint32_t ld_sched(const uint32_t* p) {
  uint32_t w;
  asm volatile("ld.global.u32 %0, [%1];" : "=r"(w) : "l"(p) : "memory");
  return w;
}

// Schedule words of PREP_THREADS / 8 tile distances, one word a thread (8 (row quarter, key half) blocks for each; see
// PipeWord in atf_prefill_pipe.cu).
__device__ inline void atf_write_schedule(const AtfTable& table, int mode, int H, int ndt, uint32_t* __restrict__ out) {
  constexpr int T = 128;
  __shared__ int w[ATF_MAX_PAIRS];
  if (threadIdx.x < H) w[threadIdx.x] = table.w[threadIdx.x];
  __syncthreads();
  const int dt = blockIdx.x * (ATF_PREP_THREADS / 8) + (threadIdx.x >> 3);
  if (dt >= ndt) return;
  const int wq = (threadIdx.x >> 1) & 3, h = threadIdx.x & 1;
  const int Wmax = w[H - 1];
  auto reaching = [&](int z) {  // pairs (from the low-frequency end) whose window reaches distance z
    int lo = 0, hi = H;         // first r with w[r] >= z, w non-decreasing
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (w[mid] < z) lo = mid + 1; else hi = mid;
    }
    return H - lo;
  };
  const int tile_any = reaching(dt == 0 ? 0 : dt * T - (T - 1));  // live somewhere in the tile
  const int mid0 = reaching(dt == 0 ? 15 : dt * T - 48);           // what the nearest quarter keeps in the MMA
  const int natoms = mode == ATF_MODE_EXACT ? (mid0 + 7) / 8 : (dt == 0 ? H / 8 : (tile_any + 7) / 8);
  const int cols = mode == ATF_MODE_EXACT ? 2 * tile_any : 16 * natoms;  // exact mode also reads the pairs it adds per cell
  const int nkb = max(1, (cols + 63) / 64);
  const int zmax = dt * T + 32 * wq + 31 - 64 * h, zmin = dt * T + 32 * wq - 64 * h - 63;
  const int p_all = reaching(max(0, zmax)), p_any = reaching(max(0, zmin));
  const int p_mid = reaching(dt == 0 ? 16 * wq + 15 : dt * T + 32 * wq - 48);
  bool plain = dt > 0 && natoms > 0;
  if (mode == ATF_MODE_EXACT) plain = plain && zmax <= Wmax && min(p_all, p_mid) >= max(p_any, p_mid);
  out[8 * dt + 2 * wq + h] = (uint32_t)p_all | ((uint32_t)p_any << 7) | ((uint32_t)p_mid << 14) | ((uint32_t)natoms << 21) |
                             ((uint32_t)(nkb - 1) << 25) | ((uint32_t)plain << 27);
}
#endif

// Launch interface of the one-tile-per-CTA prefill pipeline (atf_prefill_pipe.cu); the host code of
// atf_prefill.cu and atf_prefill_split.cu (validation, pre-pass, tensor maps) calls it.
#pragma once

#include <algorithm>

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
  int heads, group;     // all heads (B Hq), heads whose tiles are dealt out together
  int jobs;             // tiles of a group
  int cuts;             // tiles that two blocks share, atf_prefill_cuts()
  unsigned int* flags;  // [cuts], zeroed by the pre-pass
  float* state;         // [cuts][128 (d + 3)]
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
// Cut tiles.  Rows of about the same length in few waves leave the SMs idle at the end (32 tiles of 445 to 477 steps for each of
// 24 heads are 5.2 waves that run as 6).  Then the first ATF_SMS tiles are worked on by two blocks each: blocks 0 .. ATF_SMS - 1
// take the first (j + 1/2) / ATF_SMS of tile j's steps, which lets the SMs fall out of step evenly, and the blocks behind all
// others go on where those stopped, the longest rest first, so that all SMs end together.  O, row sums and reference pass
// through memory in fp32 as they stand: the result is bit for bit that of one block.  The second block of a
// tile comes at a time when the first is long done.  CUDA promises no order in which blocks start, though, so it waits only for a
// first block that has said that it runs (and waits for no other block itself); if that one has not started, the second takes the
// whole tile, and what the first one does later is read by nobody.
// Cut where the idle share is above a fifth: the kernel with the cut is 2 to 4 % slower, rows out of step share fewer K and V
// tiles in L2, and under the power cap idle SMs leave their power to the others (us, whole -> cut: 24 heads of 128, 850 of 9000, 52 %
// idle, exact 189 -> 170, coarse 125 -> 102, 1000 of 12000, 35 %, 225 -> 208, 1000 of 100000, full, 37 %, 1660 -> 1308; 14 heads of 64,
// 1600 of 20000, 49 %, 229 -> 177; 28 heads of 128, 900 of 1000000, full, 17.0 -> 14.6 ms; 24 heads, 900 of 2600, 45 %, 99.7 -> 100.3 us).  Not cut: 2000 of 40000, 9 %, 1020 -> 1078, 1400 of
// 40000, 3 %, 704 -> 783, 4000 of 61003, 15 %, exact 2880 -> 2960, coarse 2750 -> 2660.  The twelve steps an SM beside the fifth stand
// for what a cut costs whatever the length; between 20 and 25 % they refuse calls on both sides: 3000 of 20000, 21 %, 809 -> 817, but
// 1111 of 30000, 23 %, 512 -> 476, and 14 heads of 64, 2000 of 20000, 23 %, 274 -> 250.
constexpr int ATF_SMS = 148;
inline size_t atf_cut_floats(int d) { return (size_t)ATF_SMS * 128 * (d + 3); }
inline int atf_prefill_cuts(int64_t N, int64_t Nq, int64_t heads, int w_max, int d, size_t spare_bytes) {
  const int64_t dlim = ((int64_t)w_max + 127) / 128 + 1, last = (N + 127) / 128, first = (N - Nq) / 128;
  const int64_t jobs = (last - first) * heads, waves = (jobs + ATF_SMS - 1) / ATF_SMS;
  if (jobs <= ATF_SMS || jobs > 0x7FFFFF00 || spare_bytes < (atf_cut_floats(d) + ATF_SMS) * 4) return 0;
  // steps of a block: its key tiles, and three for prologue and epilogue
  const int64_t shortest = std::min(first + 1, dlim) + 3, longest = std::min(last, dlim) + 3;
  const double busy = (double)jobs * (shortest + longest) / 2, idle = (double)(waves * ATF_SMS - jobs) * shortest;
  return idle > 0.2 * busy + 12 * ATF_SMS ? ATF_SMS : 0;
}
inline int atf_sched_blocks(int64_t N) { return (int)(((N + 127) / 128 + ATF_PREP_THREADS / 8 - 1) / (ATF_PREP_THREADS / 8)); }

#ifdef __CUDACC__
// A schedule word: an ordinary load that stays behind the wait.  The pre-pass may still be writing when the kernel that
// reads starts, and the read-only path (__ldg) is defined only for what nothing writes while that kernel is resident.
__device__ __forceinline__ uint32_t ld_sched(const uint32_t* p) {
  uint32_t w;
  asm volatile("ld.global.u32 %0, [%1];" : "=r"(w) : "l"(p) : "memory");
  return w;
}

// The flag between the two blocks of a cut tile, written by the first one.
enum { CUT_RUNS = 1, CUT_STATE_THERE = 2, CUT_OVERFLOW = 4 };
__device__ __forceinline__ void st_release(unsigned int* p, unsigned int v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Schedule words of PREP_THREADS / 8 tile distances, one word a thread (8 (row quarter, key half) blocks for each; see
// PipeWord in atf_prefill_pipe.cu).
__device__ inline void atf_write_schedule(const AtfTable& table, int mode, int H, int ndt, uint32_t* out, int cuts,
                                          unsigned int* flags) {
  if (blockIdx.x == 0 && (int)threadIdx.x < cuts) flags[threadIdx.x] = 0u;
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

// atf_prefill kernel: windowed causal attention for all query rows (Sec. 3.3, Fig. 3) on the sm_100a
// tensor cores, ONE 128-row query tile of one head per CTA.  (Layout of the operands: atf_prefill.cu.)
//
// With a single query tile the 512 tensor-memory columns hold two S buffers, two P buffers and O, so
// the chain "softmax -> O += P V -> next S -> softmax" is cut: S(t + 1) = Q K(t + 1)^T is computed
// while the softmax groups work on S(t), and O += P(t) V runs whenever P(t) is stored.  Warp roles:
//   warp 0      TMA producer: K (live 64-column blocks) and V tiles into rings (stages: PipeSmem) of
//               128-byte-swizzled shared memory;
//   warp 1      issuer of S(t) = Q K(t)^T over the live depth (one thread, tcgen05.mma SS form);
//   warp 2      issuer of O += P(t) V(t), half a tile at a time (one thread, TS form: P is read from
//               tensor memory, V through the MN-major descriptor);
//   warps 4-7   softmax group 0: keys 0..63 of every tile, one query row per thread;
//   warps 8-11  softmax group 1: keys 64..127 of the same rows.
// TURNS (coarse mode; which calls: launch_pipe): behind the diagonal tile the groups take whole tiles in turn instead, so that one
// group's waits and tensor-memory round trips fall into the other's exponentials, and a tile has one of each where it had two.
// The sums of a tile's two key halves then go through shared memory to warp 2, which adds them in the order of the tiles, as the
// two threads of a row do otherwise; at d = 128 the second copy of the exchange area takes the third K stage's place (a second
// copy is worth it: with one, 8192 rows 439 us, with two and three K but two V stages 461, so 410).
// The softmax warps also bring Q in (half a row each, again per pass, see below): they read the caller's rows and
// store them to shared memory in the column order of atf_prefill.cu.  A row of Q is read by one CTA only, so a pre-pass
// that reorders it would move it twice more (8192 rows of 24 heads: 22 us of 700).  The split-precision mode keeps such
// a pre-pass and loads Q by TMA: splitting fp32 rows here took longer (10001 rows: 1.21 against 1.19 ms).  Exact mode
// holds a second, whole copy for the per-cell finish, where a pair fetched from global memory costs an L2 round trip; at
// d = 128 that leaves two K stages instead of three, which pays at every length (24 heads of 8192 rows 596 us against 636,
// of 131072 rows 83.9 ms against 85.8).  Full attention, which finishes nothing, runs the coarse form (atf_prefill.cu).
// The launch overlaps the end of the pre-pass (programmatic dependent launch): everything up to Q needs nothing of it.
// The two threads of a row never meet in the common step: exponentials are taken against the
// row's reference maximum from the diagonal tile (any reference gives the same softmax as long
// as nothing overflows: P is bf16, O and the row sums are fp32), each thread keeps its own
// partial row sum, and the halves are added at the end.  A thread whose sum of a step is not
// below 2^64 raises a flag; the CTA then runs its tile a second time in the safe form (the two
// groups exchange their row maxima through shared memory every step and rescale O at once).
//
// Steps far from the diagonal and from every window boundary ("plain") need neither the mask nor the
// per-cell finish and run in a loop of their own, kept small so that it stays in the instruction
// cache; everything else takes the general step, one step at a time.
//
// Exact mode (the per-term definition).  Whether a pair stays in the MMA is decided per quarter of
// the rows over the whole 128 keys (the pair is live at the distance from the quarter's middle row
// to the tile's middle column); the pairs a quarter does not keep are zeroed in its rows of the
// CTA's copy of Q (pairs only die as the distance grows and the tiles are walked outwards from
// the diagonal, so the zeroing is monotone).  A warp then finishes its 32 x 64 cells with small
// products of its own (mma.sync): pairs in the MMA are taken back out of the cells beyond their window,
// pairs zeroed in Q are added where live.  Coarse mode: depth = pairs live anywhere in the tile rounded up to 8,
// everything on the diagonal tile, no per-cell work.
//
// Appended rows (App. C, "The interval itself"; Sec. 7.3): the tiles stay aligned at position 0 of the
// context, the grid covers only the tiles that hold query rows, Q is addressed at tile * 128 - n0.
// Every wait is bounded and reports through the workspace status words.
#include <cuda.h>

#include <algorithm>

#include "atf_common.cuh"
#include "atf_prefill_pipe.cuh"

namespace {

constexpr int T = 128;
constexpr int BLK_BYTES = T * 128;
constexpr int PP_THREADS = 384;
constexpr float RESCALE_THRESHOLD = 8.f;      // safe form: log2 units the reference may lag behind
constexpr float REF_HEADROOM = 60.f;            // fast pass: log2 units the row's reference sits above the diagonal tile's maximum
constexpr float STALE_REF_GUARD = 1.8446744e19f;  // 2^64: a step's partial row sum must stay below it
static_assert(128 * 56 + 256 * 224 <= PP_THREADS * 168, "setmaxnreg budget exceeds the launch allocation");

// SPLIT (the split-precision mode, atf_prefill_split.cu): Q and K come as bf16 hi and lo parts; the CTA holds both
// Q parts, a K stage is a hi tile followed by a lo tile, and the rings shrink to two K stages and one V stage.
// QCOPY (exact mode, bf16 inputs): a second copy of Q that stays whole, for the per-cell finish; at d = 128 it takes the
// place of the third K stage.
template <int D, bool SPLIT, bool QCOPY, bool TURNS>
struct PipeSmem {
  static constexpr int NB = D / 64;
  static constexpr int TILE = NB * BLK_BYTES;
  static constexpr int QN = SPLIT ? 2 : 1;       // operand parts: hi, lo
  static constexpr int KS = SPLIT || ((QCOPY || TURNS) && D == 128) ? 2 : 3;  // ring depths
  static constexpr int VS = SPLIT ? 1 : 3;
  static constexpr int KSTAGE = QN * TILE;
  static constexpr int Q_OFF = 0;                // hi part, then lo part
  static constexpr int K_OFF = QN * TILE;
  static constexpr int V_OFF = K_OFF + KS * KSTAGE;
  static constexpr int QC_OFF = V_OFF + VS * TILE;
  static constexpr int BAR_OFF = QC_OFF + (QCOPY ? TILE : 0);
  static constexpr int X_OFF = BAR_OFF + 256;  // exchange area of the two softmax groups: [2][128] floats, in turns two of them
  static constexpr int TOTAL = X_OFF + (TURNS ? 2048 : 1024);
  static constexpr int DYN_BYTES = TOTAL + 1024;  // slack for 1024-byte alignment
};
enum { B_QFULL = 0, B_KFULL = 1, B_KEMPTY = 4, B_VFULL = 7, B_VEMPTY = 10, B_SFULL = 13, B_SREAD = 15, B_PFULL = 17,
       B_PVDONE = 21, B_OFULL = 23, B_XCH = 24, B_QZ = 25, B_COUNT = 26 };

__device__ __forceinline__ float2 exp2_poly2(float2 x) {
  x.x = fmaxf(x.x, -126.f);
  x.y = fmaxf(x.y, -126.f);
  const float2 magic = make_float2(12582912.f, 12582912.f);
  const float2 t = __fadd2_rn(x, magic);
  const float2 nf = __fadd2_rn(t, make_float2(-12582912.f, -12582912.f));
  const float2 f = __fadd2_rn(x, make_float2(-nf.x, -nf.y));
  float2 p = __ffma2_rn(make_float2(0.05520550534f, 0.05520550534f), f, make_float2(0.24261397123f, 0.24261397123f));
  p = __ffma2_rn(p, f, make_float2(0.69325476885f, 0.69325476885f));
  p = __ffma2_rn(p, f, make_float2(0.99992769957f, 0.99992769957f));
  float2 r;
  r.x = __int_as_float(__float_as_int(p.x) + (__float_as_int(t.x) << 23));
  r.y = __int_as_float(__float_as_int(p.y) + (__float_as_int(t.y) << 23));
  return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
#ifndef ATF_PIPE_POLY_OF_4
#define ATF_PIPE_POLY_OF_4 1
#endif
// P = 2^(s * scale + neg_m) for 64 columns, packed to bf16 pairs, and their fp32 sum; one packed pair in
// four takes a cubic polynomial on the FMA pipe (relative error < 8e-5, below the bf16 rounding of P), the rest
// MUFU; POLY = 0 (the split-precision mode, whose row sums must be good to 1e-6) is MUFU only.
template <int POLY>
__device__ __forceinline__ float exp_half(float (&s)[64], float scale, float neg_m, uint32_t (&pk)[32]) {
  const float2 sc2 = make_float2(scale, scale), nm2 = make_float2(neg_m, neg_m);
  float2 acc[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
  for (int c = 0; c < 64; c += 2) {
    float2 x = __ffma2_rn(make_float2(s[c], s[c + 1]), sc2, nm2);
    if (((c >> 1) & 3) < POLY) {
      x = exp2_poly2(x);
    } else {
      x.x = ex2_approx(x.x);
      x.y = ex2_approx(x.y);
    }
    acc[(c >> 1) & 3] = __fadd2_rn(acc[(c >> 1) & 3], x);
    pk[c >> 1] = pack_bf16x2(x.x, x.y);
  }
  const float2 a01 = __fadd2_rn(acc[0], acc[1]), a23 = __fadd2_rn(acc[2], acc[3]);
  return (a01.x + a01.y) + (a23.x + a23.y);
}

// C (16 x 8, fp32 fragment) += A (16 x 16) B (16 x 8), bf16.
__device__ __forceinline__ void mma_16816(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Band schedule (Sec. 3.3: the active pairs of a tile are known statically; written by atf_write_schedule, atf_prefill_pipe.cuh).  What a step needs depends only on
// the tile distance dt and on which 32 rows x 64 keys of the tile a softmax warp owns (quarter wq of the rows,
// half h of the keys); it is the same for every CTA of a launch.  A pre-kernel writes one word per (dt, wq, h):
//   p_all  [0:7)   pairs live in every cell of the warp's block,      p_any [7:14)  pairs live in some cell of it,
//   p_mid  [14:21) pairs quarter wq keeps in the MMA (live at the distance from its middle row to the tile's
//                  middle column); the others are zero in its rows of Q,
//   natoms [21:25) 16-column MMA steps of S,   nkb [25:27) 64-column K blocks to load minus one,
//   plain  [27]    the block needs neither mask nor per-cell finish and S is not empty.
// Roles read their word a step ahead, so no schedule arithmetic sits in front of a step.
struct PipeWord {
  int p_all, p_any, p_mid, natoms, nkb;
  bool plain;
  __device__ __forceinline__ explicit PipeWord(uint32_t e)
      : p_all(e & 127), p_any((e >> 7) & 127), p_mid((e >> 14) & 127), natoms((e >> 21) & 15), nkb(((e >> 25) & 3) + 1),
        plain((e >> 27) & 1) {}
};

__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_timer_ns();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 128; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (global_timer_ns() - t0 > ATF_WAIT_LIMIT_NS) {
      *abort_flag = 1;
      return false;
    }
  }
}

template <int D, int MODE, bool COUNT, bool SPLIT, bool TURNS, bool CUT>
__global__ void __launch_bounds__(PP_THREADS, 1)
atf_prefill_pipe_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmQlo,
                        const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmKlo,
                        const __grid_constant__ CUtensorMap tmV, const __grid_constant__ AtfPipeParams P,
                        const __grid_constant__ AtfTable table) {
  constexpr bool QCOPY = MODE == ATF_MODE_EXACT && !SPLIT;
  using SM = PipeSmem<D, SPLIT, QCOPY, TURNS>;
  constexpr int KS = SM::KS, VS = SM::VS;
  constexpr int POLY = SPLIT ? 0 : ATF_PIPE_POLY_OF_4;
  constexpr int H = D / 2;
  constexpr int NB = D / 64;
  constexpr uint32_t TMEM_COLS = 512;  // S0, S1 (128 each) | O (D) at 256 | P0, P1 (64 each) at 384
  constexpr uint32_t IDESC_QK = make_idesc_bf16(128, T, 0, 0);
  constexpr uint32_t IDESC_PV = make_idesc_bf16(128, D, 0, 1);
  const float kScaleLog2 = 1.4426950408889634f / sqrtf((float)D);

  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t sQ = smem_base + SM::Q_OFF, sK = smem_base + SM::K_OFF, sV = smem_base + SM::V_OFF;
  const uint32_t bars = smem_base + SM::BAR_OFF;
  auto bar = [&](int slot) { return bars + 8u * (uint32_t)slot; };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + SM::BAR_OFF + 8 * B_COUNT);
  volatile float* xch = reinterpret_cast<volatile float*>(smem_gen + SM::X_OFF);  // [2][128]
  __shared__ int sW[ATF_MAX_PAIRS];
  __shared__ int s_abort;
  __shared__ int s_redo;
  __shared__ volatile int s_part[CUT ? 2 : 1];  // CUT: first step of the block in the fast pass; whether it ends at the cut

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n0 = P.N - P.Nq;
  // The tiles of a group of heads, longest rows first (blocks start about in the order of their index).  CUT: the first P.cuts
  // tiles are worked on by two blocks (atf_prefill_cuts).
  const int ntq = (P.N + T - 1) / T;
  const bool first = CUT && (int)blockIdx.x < P.cuts, second = CUT && (int)blockIdx.x >= P.jobs;
  const int job = second ? (int)blockIdx.x - P.jobs : (int)blockIdx.x;
  const int head0 = (int)blockIdx.y * P.group, heads = min(P.group, P.heads - head0);
  const int it = ntq - 1 - job / heads;
  if (it < n0 / T) return;  // the last group may have fewer heads
  const int bhq = head0 + job % heads;
  const int b = bhq / P.Hq, hq = bhq - b * P.Hq;
  const int bhk = b * P.Hkv + hq / (P.Hq / P.Hkv);
  const int Wmax = table.w[H - 1];
  const int dlim = (Wmax + T - 1) / T + 1;  // first tile distance no pair reaches
  const int nt = min(it + 1, dlim);         // key tiles it, it - 1, ... walked outwards from the diagonal
  const int cut = first || second ? (int)((long long)nt * (2 * job + 1) / (2 * P.cuts)) : 0;  // steps of the first block
  if (first && cut == 0) return;
  const int t_end = first ? cut : nt;

  if (tid < H) sW[tid] = table.w[tid];
  if (tid == 0) {
    s_abort = 0;
    s_redo = 0;
    if (CUT) {
      s_part[0] = second ? cut : 0;
      s_part[CUT ? 1 : 0] = first;
    }
    mbar_init(bar(B_QFULL), SPLIT ? 1 : 8);
    mbar_init(bar(B_OFULL), 1);
    mbar_init(bar(B_XCH), 8);
    mbar_init(bar(B_QZ), 4);
    for (int i = 0; i < 3; ++i) {
      mbar_init(bar(B_KFULL + i), 1);
      // exact mode: the softmax warps read K for the per-cell finish and release the stage; coarse: the issuer's commit
      mbar_init(bar(B_KEMPTY + i), MODE == ATF_MODE_EXACT ? 8 : 1);
      mbar_init(bar(B_VFULL + i), 1);
      mbar_init(bar(B_VEMPTY + i), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(B_SFULL + i), 1);
      mbar_init(bar(B_SREAD + i), 8);
      mbar_init(bar(B_PFULL + 2 * i), 4);
      mbar_init(bar(B_PFULL + 2 * i + 1), 4);
      mbar_init(bar(B_PVDONE + i), 1);
    }
    mbar_fence_init();
    fence_proxy_async_smem();
    tma_prefetch_desc(&tmK);
    if (SPLIT) {
      tma_prefetch_desc(&tmQ);
      tma_prefetch_desc(&tmQlo);
      tma_prefetch_desc(&tmKlo);
    }
    tma_prefetch_desc(&tmV);
  }
  if (warp == 0) {
    tmem_alloc(smem_u32((const void*)tmem_slot), TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  volatile int* abortp = &s_abort;
  unsigned int fail_site = 0;

  // A cut tile's state: O (fp32, [D / 4][128 rows][4]), the sums of the two key halves, the rows' reference; and a flag (with
  // CUT_OVERFLOW a sum has overflowed: the whole tile takes the safe form).
  auto cut_state = [&]() {
    const int j = (int)blockIdx.x < P.cuts ? (int)blockIdx.x : (int)blockIdx.x - P.jobs;
    return P.state + (int64_t)j * (T * (D + 3));
  };
  if (CUT && second && cut > 0) {
    if (tid == 0) {
      grid_dependency_wait();
      const unsigned int* flag = P.flags + ((int)blockIdx.x - P.jobs);
      if (ld_acquire(flag) == 0u) {
        s_part[0] = 0;  // the first block has not started: the whole tile
      } else {
        const unsigned int f = flag_wait(flag, CUT_STATE_THERE, ATF_WAIT_LIMIT_NS);
        if (!(f & CUT_STATE_THERE)) {
          s_abort = 1;
          fail_site = 38;
        }
        if (f & CUT_OVERFLOW) {
          s_redo = 1;
          s_part[0] = nt;  // no step of the fast pass
        }
      }
    }
    __syncthreads();
  }

  // Every role runs the tile once and, if a softmax thread raised s_redo, once more in the safe form.  The
  // passes end at a CTA-wide barrier (the same barrier from every role's branch); barrier phases of the
  // pipeline run on across the passes (g = steps since the start of the kernel).
  auto another_pass = [&](int pass) {
    asm volatile("bar.sync 0;" ::: "memory");
    return pass == 0 && !(CUT && s_part[CUT ? 1 : 0]) && *reinterpret_cast<volatile int*>(&s_redo) != 0;
  };

  if (warp == 0) {
    // =============================== TMA producer ===============================
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    grid_dependency_wait();
    for (int pass = 0; pass < 2; ++pass) {
      const int tb = CUT && !pass ? s_part[0] : 0, g0 = (pass ? t_end - (CUT ? s_part[0] : 0) : 0) - tb;  // g = g0 + t: steps of this block so far
      if (lane == 0) {
        if (SPLIT) {
          mbar_expect_tx(bar(B_QFULL), SM::QN * SM::TILE);
          for (int kb = 0; kb < NB; ++kb) {
            // rows before n0 do not exist in Q: the (possibly negative) coordinate reads zero fill there
            tma_load_3d(sQ + kb * BLK_BYTES, &tmQ, bar(B_QFULL), kb * 64, it * T - n0, bhq);
            tma_load_3d(sQ + SM::TILE + kb * BLK_BYTES, &tmQlo, bar(B_QFULL), kb * 64, it * T - n0, bhq);
          }
        }
        auto load_k = [&](int t) {
          const int g = g0 + t, ks = g % KS;
          if (!wait_or_abort(bar(B_KEMPTY + ks), ((g / KS) & 1) ^ 1, abortp)) return false;
          const int nkb = PipeWord(ld_sched(P.sched + 8 * t)).nkb;
          mbar_expect_tx(bar(B_KFULL + ks), SM::QN * nkb * BLK_BYTES);
          for (int kb = 0; kb < nkb; ++kb) {
            tma_load_3d(sK + ks * SM::KSTAGE + kb * BLK_BYTES, &tmK, bar(B_KFULL + ks), kb * 64, (it - t) * T, bhk);
            if (SPLIT)
              tma_load_3d(sK + ks * SM::KSTAGE + SM::TILE + kb * BLK_BYTES, &tmKlo, bar(B_KFULL + ks), kb * 64, (it - t) * T, bhk);
          }
          return true;
        };
        auto load_v = [&](int t) {
          const int g = g0 + t, vs = g % VS;
          if (!wait_or_abort(bar(B_VEMPTY + vs), ((g / VS) & 1) ^ 1, abortp)) return false;
          mbar_expect_tx(bar(B_VFULL + vs), SM::TILE);
          for (int kb = 0; kb < NB; ++kb)
            tma_load_3d(sV + vs * SM::TILE + kb * BLK_BYTES, &tmV, bar(B_VFULL + vs), kb * 64, (it - t) * T, bhk);
          return true;
        };
        if (SPLIT || TURNS || D == 128) {
          // S runs ahead of O += P V: K(t + 1) in front of V(t), which may have to wait for a product (24 heads x 8192 rows of 128,
          // coarse: 423 -> 410 us in turns; exact, a layer step: 650 -> 644; 14 heads x 32768 of 64, exact, the other way: 2843
          // against 2822)
          bool pok = tb >= t_end || load_k(tb);
          for (int t = tb; t < t_end && pok; ++t) pok = (t + 1 >= t_end || load_k(t + 1)) && load_v(t);
          if (!pok) fail_site = 10;
        } else {
          for (int t = tb; t < t_end; ++t)
            if (!load_k(t) || !load_v(t)) { fail_site = 10; break; }
        }
      }
      if (!another_pass(pass)) break;
    }
  } else if (warp == 1) {
    // =============================== issuer of S = Q K^T ===============================
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    grid_dependency_wait();
    for (int pass = 0; pass < 2; ++pass) {
      const int tb = CUT && !pass ? s_part[0] : 0, g0 = (pass ? t_end - (CUT ? s_part[0] : 0) : 0) - tb;
      if (lane == 0) {
        const uint64_t dQ = make_smem_desc_sw128(sQ, 16, 1024);
        bool iok = wait_or_abort(bar(B_QFULL), pass & 1, abortp);
        if (!iok) fail_site = 20;
        for (int t = tb; t < t_end && iok; ++t) {
          const int g = g0 + t, sb = g & 1, ks = g % KS;
          const int natoms = PipeWord(ld_sched(P.sched + 8 * t)).natoms;
          iok = wait_or_abort(bar(B_KFULL + ks), (g / KS) & 1, abortp);
          // both softmax groups hold S(g - 2) in registers: its buffer may be written again
          if (iok && g >= 2) iok = wait_or_abort(bar(B_SREAD + sb), ((g >> 1) - 1) & 1, abortp);
          // exact mode: the pairs a quarter does not keep in the MMA of this tile are zero in its rows of Q
          if (iok && MODE == ATF_MODE_EXACT) iok = wait_or_abort(bar(B_QZ), g & 1, abortp);
          if (!iok) { fail_site = 21; break; }
          tc_fence_after();
          const uint64_t dK = make_smem_desc_sw128(sK + ks * SM::KSTAGE, 16, 1024);
          const uint32_t tS = tmem_base + sb * T;
          for (int a = 0; a < natoms; ++a) {
            // K-major operands advance 32 bytes per 16-column step inside a 64-column block, one block per four steps
            const uint64_t off = (uint64_t)((a & 3) * 2 + (a >> 2) * (BLK_BYTES / 16));
            tc_mma_ss(tS, dQ + off, dK + off, IDESC_QK, a > 0 ? 1u : 0u);
            if (SPLIT) {  // + Q_hi K_lo^T + Q_lo K_hi^T (the lo parts sit one tile after the hi parts)
              tc_mma_ss(tS, dQ + off, dK + off + (uint64_t)(SM::TILE / 16), IDESC_QK, 1u);
              tc_mma_ss(tS, dQ + off + (uint64_t)(SM::TILE / 16), dK + off, IDESC_QK, 1u);
            }
          }
          tc_commit(bar(B_SFULL + sb));
          if (MODE != ATF_MODE_EXACT) tc_commit(bar(B_KEMPTY + ks));
        }
      }
      if (!another_pass(pass)) break;
    }
  } else if (warp == 2) {
    // =============================== issuer of O += P V ===============================
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    for (int pass = 0; pass < 2; ++pass) {
      const int tb = CUT && !pass ? s_part[0] : 0, g0 = (pass ? t_end - (CUT ? s_part[0] : 0) : 0) - tb;
      const bool sums = TURNS && pass == 0;  // the whole warp walks the steps, else lane 0 alone
      float sum[2][4] = {};                  // rows 4 lane .. 4 lane + 3, keys 0..63 and 64..127 of the tiles so far
      bool iok = true;
      if (CUT && sums && tb > 0 && tb < t_end) {
        const float* state = cut_state();
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int i = 0; i < 4; ++i) sum[h][i] = __ldcg(state + T * (D + h) + 4 * lane + i);
      }
      for (int t = tb; t < t_end && iok && (sums || lane == 0); ++t) {
        const int g = g0 + t, sb = g & 1, vs = g % VS;
        if (lane == 0) {
          const uint64_t dV = make_smem_desc_sw128(sV + vs * SM::TILE, BLK_BYTES, 1024);
          const uint32_t tO = tmem_base + 2 * T, tP = tmem_base + 3 * T + sb * 64;
          iok = wait_or_abort(bar(B_VFULL + vs), (g / VS) & 1, abortp);
          for (int h = 0; h < 2 && iok; ++h) {
            iok = wait_or_abort(bar(B_PFULL + 2 * sb + h), (g >> 1) & 1, abortp);
            if (!iok) break;
            tc_fence_after();
#pragma unroll
            for (int i = 0; i < 4; ++i)  // V advances 16 key rows (2048 bytes) per step, P 8 columns
              tc_mma_ts(tO, tP + 32 * h + 8 * i, dV + (uint64_t)(512 * h + 128 * i), IDESC_PV,
                        (t > 0 || h > 0 || i > 0) ? 1u : 0u);
          }
          if (!iok) fail_site = 22;
        }
        if (sums) {
          // the tile's sums, added in the order of the tiles
          iok = __shfl_sync(0xffffffffu, (int)iok, 0);
          if (!iok) break;
          __syncwarp();  // lane 0 alone has waited for what the softmax warps wrote, and a shuffle orders no memory
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float v[4];
            lds_f4(smem_base + SM::X_OFF + ((2 * sb + h) * 128 + 4 * lane) * 4, v);
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[h][i] += v[i];
          }
          __syncwarp();
        }
        if (lane == 0 && iok) {
          tc_commit(bar(B_VEMPTY + vs));
          tc_commit(bar(B_PVDONE + sb));
        }
      }
      if (lane == 0 && iok) tc_commit(bar(B_OFULL));
      if (sums) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int i = 0; i < 4; ++i) xch[h * 128 + 4 * lane + i] = sum[h][i];
      }
      if (!another_pass(pass)) break;
    }
  } else if (warp == 3) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    if (first) {
      grid_dependency_wait();  // the pre-pass zeroes the flags
      if (lane == 0) st_release(P.flags + blockIdx.x, CUT_RUNS);
    }
    for (int pass = 0; pass < 2; ++pass)
      if (!another_pass(pass)) break;
  } else {
    // =============================== softmax groups ===============================
    asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    const int h = warp >= 8 ? 1 : 0;  // keys 64h .. 64h + 63 of every tile
    const int wq = warp & 3;
    const int row = (tid - 128) & 127;
    const int n = it * T + row;
    const bool row_ok = n >= n0 && n < P.N;
    const int64_t qrow = (int64_t)bhq * P.Nq + (row_ok ? n - n0 : 0);
    const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
    const uint32_t tO = tmem_base + 2 * T + lane_off;
    // split mode: the hi and lo parts of this row, pairs in column order
    const uint32_t* qsrc = SPLIT ? reinterpret_cast<const uint32_t*>(P.Qhi + qrow * D) : nullptr;
    const uint32_t* qsrc_lo = SPLIT ? reinterpret_cast<const uint32_t*>(P.Qlo + qrow * D) : nullptr;
    float m_used = -INFINITY, l_run = 0.f;
    unsigned long long cnt = 0;
    uint32_t xphase = 0;
    bool ok = true, redone = false;
    // all eight softmax warps meet (bounded): what each wrote to the exchange area before is visible after
    auto softmax_sync = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(B_XCH));
      const bool r = wait_or_abort(bar(B_XCH), xphase & 1, abortp);
      ++xphase;
      return r;
    };
    // This group's half of the pairs of the row, p = h H/2 + i: dims H-1-p and D-1-p, which are QW consecutive elements of
    // each half row in falling order.  Rows that do not exist (before n0, from N on) are zero.  Ordinary loads: a caller may
    // have O written over Q (the rows a CTA writes are those it alone has read).
    constexpr int QW = H / 2;
    auto load_q = [&](uint32_t (&w)[QW]) {
      const __nv_bfloat16* q = P.Q + qrow * D + (H - QW - h * QW);
      uint32_t x[QW / 2], y[QW / 2];
#pragma unroll
      for (int i = 0; i < QW / 2; i += 4) {
        *reinterpret_cast<uint4*>(x + i) = row_ok ? *reinterpret_cast<const uint4*>(q + 2 * i) : make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(y + i) = row_ok ? *reinterpret_cast<const uint4*>(q + H + 2 * i) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int i = 0; i < QW; ++i) w[i] = __byte_perm(x[(QW - 1 - i) >> 1], y[(QW - 1 - i) >> 1], (i & 1) ? 0x5410 : 0x7632);
    };
    for (int pass = 0; pass < 2; ++pass) {
      const int tb = CUT && !pass ? s_part[0] : 0, g0 = (pass ? t_end - (CUT ? s_part[0] : 0) : 0) - tb;
      const bool safe = pass == 1;
      redone = safe;
      uint32_t qw[QW];
      if constexpr (!SPLIT) load_q(qw);
      if (pass == 0) grid_dependency_wait();
      m_used = -INFINITY;
      l_run = 0.f;
      cnt = 0;
      bool overflow = false;
      int zeroed_from = H;  // pairs p >= zeroed_from are zero in this row of the shared copy of Q
      // group 0 owns the rows of Q: zero what the quarter does not keep in the MMA, then tell the issuer
      auto zero_q_down_to = [&](int p_keep) {
        if (h == 0) {
          for (int p = p_keep; p < zeroed_from; ++p) {
            const int col = 2 * p;
            const uint32_t off = (col >> 6) * BLK_BYTES + sw128_offset(row, (col & 63) >> 3) + (col & 7) * 2;
            *reinterpret_cast<uint32_t*>(smem_gen + SM::Q_OFF + off) = 0u;
            if (SPLIT) *reinterpret_cast<uint32_t*>(smem_gen + SM::Q_OFF + SM::TILE + off) = 0u;
          }
          zeroed_from = min(zeroed_from, p_keep);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(B_QZ));
        }
      };
      const uint32_t* sched = P.sched + 2 * wq + h;
      uint32_t e_cur = ld_sched(sched + (CUT ? 8 * min(tb, t_end - 1) : 0));  // schedule word of the step at hand; the next one is fetched a step ahead
      int p_mid = PipeWord(e_cur).p_mid;
      if constexpr (SPLIT) {
        if (MODE == ATF_MODE_EXACT) {
          if (ok && !wait_or_abort(bar(B_QFULL), pass & 1, abortp)) { ok = false; fail_site = 30; }
          if (ok && (!CUT || tb < t_end)) zero_q_down_to(p_mid);
        }
      } else {
        // ---- Q: this group's half of the pairs of the row, p = h H/2 + i.  Exact mode: what the first MMA does not take
        //      is zero, and the copy stays whole. ----
        const int p_keep = MODE == ATF_MODE_EXACT ? p_mid : H;
#pragma unroll
        for (int c = 0; c < QW / 4; ++c) {
          const int p = h * QW + 4 * c;
          const uint32_t off = (p >> 5) * BLK_BYTES + sw128_offset(row, (p & 31) >> 2);
          *reinterpret_cast<uint4*>(smem_gen + SM::Q_OFF + off) =
              make_uint4(p < p_keep ? qw[4 * c] : 0u, p + 1 < p_keep ? qw[4 * c + 1] : 0u,
                         p + 2 < p_keep ? qw[4 * c + 2] : 0u, p + 3 < p_keep ? qw[4 * c + 3] : 0u);
          if (QCOPY) *reinterpret_cast<uint4*>(smem_gen + SM::QC_OFF + off) = make_uint4(qw[4 * c], qw[4 * c + 1], qw[4 * c + 2], qw[4 * c + 3]);
        }
        zeroed_from = p_keep;
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(bar(B_QFULL));
          if (MODE == ATF_MODE_EXACT && h == 0 && (!CUT || tb < t_end)) mbar_arrive(bar(B_QZ));
        }
      }
      if (CUT && tb > 0 && tb < t_end) {  // the second block of a cut tile goes on from what the first left
        const float* state = cut_state();
        l_run = __ldcg(state + T * (D + h) + row);
        m_used = __ldcg(state + T * (D + 2) + row);
        if (h == 0) {  // O: the first product waits for this group's P
          const float4* src = reinterpret_cast<const float4*>(state) + row;
#pragma unroll 1
          for (int c0 = 0; c0 < D; c0 += 32) {
            uint32_t o[32];
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
              const float4 v = __ldcg(src + (c0 + e) / 4 * T);
              o[e] = __float_as_uint(v.x);
              o[e + 1] = __float_as_uint(v.y);
              o[e + 2] = __float_as_uint(v.z);
              o[e + 3] = __float_as_uint(v.w);
            }
            tc_st32(tO + c0, o);
          }
          tc_wait_st();
          tc_fence_before();
        }
      }
      int t = tb;
      while (t < t_end && ok) {
        if constexpr (TURNS) {
          // ---- In turns: behind the diagonal tile group h takes the steps g with g % 2 == h, all 128 keys of its rows. ----
          if (t > 0 && !safe) {
            const float neg_m = -m_used * kScaleLog2;
            const uint32_t tS = tmem_base + h * T + lane_off, tP = tmem_base + 3 * T + h * 64 + lane_off;
            for (t += (g0 + t + h) & 1; t < t_end; t += 2) {
              const int g = g0 + t;
              if (!wait_or_abort(bar(B_SFULL + h), (g >> 1) & 1, abortp)) { ok = false; fail_site = 31; break; }
              tc_fence_after();
              float sa[64], sb[64];
              tc_ld32(tS, reinterpret_cast<uint32_t*>(sa));
              tc_ld32(tS + 32, reinterpret_cast<uint32_t*>(sa) + 32);
              tc_wait_ld();
              tc_ld32(tS + 64, reinterpret_cast<uint32_t*>(sb));  // on its way behind the first half's exponentials
              tc_ld32(tS + 96, reinterpret_cast<uint32_t*>(sb) + 32);
              uint32_t pk[32];
              const float la = exp_half<POLY>(sa, kScaleLog2, neg_m, pk);
              // the product that read the previous contents of this P buffer must be complete
              if (g >= 2 && !wait_or_abort(bar(B_PVDONE + h), ((g - 2) >> 1) & 1, abortp)) { ok = false; fail_site = 35; break; }
              tc_fence_after();
              tc_st32(tP, pk);
              tc_wait_ld_pin64(sb);
              tc_wait_st();
              tc_fence_before();
              __syncwarp();
              if (lane == 0) {
                mbar_arrive_n(bar(B_SREAD + h), 2);  // for the other group's warp too
                mbar_arrive(bar(B_PFULL + 2 * h));
              }
              const float lb = exp_half<POLY>(sb, kScaleLog2, neg_m, pk);
              tc_st32(tP + 32, pk);
              overflow |= !(la < STALE_REF_GUARD) || !(lb < STALE_REF_GUARD);
              xch[h * 256 + row] = la;  // PVDONE above: warp 2 has taken what was there
              xch[h * 256 + 128 + row] = lb;
              tc_wait_st();
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(bar(B_PFULL + 2 * h + 1));
            }
            break;
          }
        }
        // ---- plain steps: no mask, no per-cell finish, reference from the diagonal tile.  A loop of its own,
        //      kept small so that it stays in the instruction cache; everything else takes the general step. ----
        for (; !TURNS && t < t_end && !safe && t > 0; ++t) {
          const int g = g0 + t, sb = g & 1, ks = g % KS;
          const PipeWord E(e_cur);
          if (!E.plain) break;
          const uint32_t e_next = t + 1 < t_end ? ld_sched(sched + 8 * (t + 1)) : 0u;
          const int p_all = E.p_all, natoms = E.natoms;
          const int p_mid_next = PipeWord(e_next).p_mid;
          if (!wait_or_abort(bar(B_SFULL + sb), (g >> 1) & 1, abortp)) { ok = false; fail_site = 31; break; }
          tc_fence_after();
          if (MODE == ATF_MODE_EXACT && t + 1 < t_end) zero_q_down_to(p_mid_next);
          float s[64];
          tc_ld32(tmem_base + sb * T + 64 * h + lane_off, reinterpret_cast<uint32_t*>(s));
          tc_ld32(tmem_base + sb * T + 64 * h + lane_off + 32, reinterpret_cast<uint32_t*>(s) + 32);
          tc_wait_ld();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(bar(B_SREAD + sb));
            if (MODE == ATF_MODE_EXACT) mbar_arrive(bar(B_KEMPTY + ks));
          }
          if (COUNT && row_ok)
            cnt += (unsigned long long)(MODE == ATF_MODE_EXACT ? p_all : min(H, 8 * natoms)) * 64ull;
          uint32_t pk[32];
          const float lsum = exp_half<POLY>(s, kScaleLog2, -m_used * kScaleLog2, pk);
          overflow |= !(lsum < STALE_REF_GUARD);
          if (g >= 2 && !wait_or_abort(bar(B_PVDONE + sb), ((g - 2) >> 1) & 1, abortp)) { ok = false; fail_site = 35; break; }
          tc_st32(tmem_base + 3 * T + sb * 64 + 32 * h + lane_off, pk);
          l_run += lsum;
          tc_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(B_PFULL + 2 * sb + h));
          p_mid = p_mid_next;
          e_cur = e_next;
        }
        if (t >= t_end || !ok) break;
        // ---- one general step ----
        const int g = g0 + t, sb = g & 1, ks = g % KS;
        const int dt = t;
        const int zrow = dt * T + row;             // distance from this row to column 0 of the key tile
        const int zmax_w = dt * T + 32 * wq + 31 - 64 * h;  // over the warp's 32 x 64 cells
        const PipeWord E(e_cur);
        const uint32_t e_next = t + 1 < t_end ? ld_sched(sched + 8 * (t + 1)) : 0u;
        const int p_all = E.p_all, p_any = E.p_any, natoms = E.natoms;
        const int p_mid_next = PipeWord(e_next).p_mid;
        const uint32_t tS = tmem_base + sb * T + 64 * h + lane_off;
        const uint32_t tP = tmem_base + 3 * T + sb * 64 + 32 * h + lane_off;
        if (!wait_or_abort(bar(B_SFULL + sb), (g >> 1) & 1, abortp)) { ok = false; fail_site = 31; break; }
        tc_fence_after();
        // S(t) is complete, so Q is not being read: zero what the quarter does not keep in the next tile's MMA
        if (MODE == ATF_MODE_EXACT && t + 1 < t_end) zero_q_down_to(p_mid_next);
        bool s_valid = natoms > 0;  // else no pair is kept in the MMA of this tile and S was not written
        if (MODE == ATF_MODE_EXACT) {
          // ---- per-cell finish.  Pairs [p_all, p_mid) went through the MMA and are not live in every cell of
          //      the warp's block: take their term back out of the cells beyond the window.  Pairs [p_mid, p_any)
          //      are zero in Q and live somewhere in the block: add their term inside the window.
          //      One pair's masked term of 16 rows x 8 keys is ONE m16n8k16 product: the contraction runs over
          //      eight slots of two elements, slot j = key j; B holds the pair of key j in slot j only, A the
          //      pair of each row in the slots of the keys it takes.  The terms are summed from zero and added to S
          //      once, rounded to nearest: mma.sync cuts a sum off, and onto S itself that cost up to a unit in the
          //      last place of the score for every pair (LSE of the outlier inputs 5 % further from 64 bits).  S is
          //      brought in 16 rows at a time for that (24 heads x 8192 rows of 128: 596 us, both halves at once 623,
          //      before the pairs 659; summing onto S 586; seven CUDA-core instructions a cell, the first form, 704).
          //      A step here still takes about twice a plain one: mma.sync waits beside tcgen05, ~270 clocks an
          //      instruction when that pipe is full, K words wait for the S product's reads of shared memory, and this
          //      code is seldom in the instruction cache. ----
          const int p_lo = min(p_all, p_mid), p_hi = max(p_any, p_mid);
          if (p_lo < p_hi && zmax_w >= 0) {
            uint32_t q_next = 0u, ql_next = 0u;
            const uint32_t qrow0 = smem_base + SM::QC_OFF + (32 * wq + (lane >> 2)) * 128;
            uint32_t qr_next[4];  // QCOPY: the pair of rows lane / 4 + 8 j, fetched a pair ahead
            auto fetch_q = [&](int p) {
              if (QCOPY) {
                const uint32_t a = qrow0 + (p >> 5) * BLK_BYTES + ((((p & 31) >> 2) ^ (lane >> 2)) << 4) + (p & 3) * 4;
#pragma unroll
                for (int j = 0; j < 4; ++j) asm volatile("ld.shared.b32 %0, [%1];" : "=r"(qr_next[j]) : "r"(a + j * 1024));
              } else {
                q_next = qsrc[p];
                ql_next = qsrc_lo[p];
              }
            };
            fetch_q(p_lo);
            if (!wait_or_abort(bar(B_KFULL + ks), (g / KS) & 1, abortp)) { ok = false; fail_site = 32; break; }
            float f[2][32];  // rows 16 hf + {lane / 4, lane / 4 + 8}, keys 64h + 8 cb + 2 (lane % 4) + {0, 1}
#pragma unroll
            for (int e = 0; e < 32; ++e) f[0][e] = f[1][e] = 0.f;
            const int g8 = lane >> 2, t4 = lane & 3;
            const uint32_t slot0 = g8 == t4 ? 0xFFFFFFFFu : 0u, slot4 = g8 == t4 + 4 ? 0xFFFFFFFFu : 0u;
            const int zw_lo = dt * T + wq * 32, zw_hi = zw_lo + 31;  // zrow over the warp's rows
            const uint32_t krow = sK + ks * SM::KSTAGE + (64 * h + g8) * 128;
#pragma unroll 1
            for (int p = p_lo; p < p_hi; ++p) {
              const bool subtract = p < p_mid;
              const uint32_t flip = subtract ? 0x80008000u : 0u;
              uint32_t qr[4], qrl[SPLIT ? 4 : 1];  // the pair of rows g8 + 8 j
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                qr[j] = QCOPY ? qr_next[j] ^ flip : __shfl_sync(0xffffffffu, q_next, g8 + 8 * j) ^ flip;
                if (SPLIT) qrl[j] = __shfl_sync(0xffffffffu, ql_next, g8 + 8 * j) ^ flip;
              }
              if (p + 1 < p_hi) fetch_q(p + 1);
              const int wp = sW[H - 1 - p];
              // row g8 + 8 j takes the key of slot t4 (t4 + 4) of block cb inside the window iff 8 (cb - j) >= u (u - 4)
              const int u = zw_lo + g8 - t4 - 64 * h - wp;
              const uint32_t kp = krow + ((2 * p) >> 6) * BLK_BYTES + (((((2 * p) & 63) >> 3) ^ g8) << 4) + ((2 * p) & 7) * 2;
              uint32_t kk[8], kl[SPLIT ? 8 : 1];
#pragma unroll
              for (int cb = 0; cb < 8; ++cb) {
                asm volatile("ld.shared.b32 %0, [%1];" : "=r"(kk[cb]) : "r"(kp + cb * 1024));
                if (SPLIT) asm volatile("ld.shared.b32 %0, [%1];" : "=r"(kl[cb]) : "r"(kp + SM::TILE + cb * 1024));
              }
              // Two halves of 32 keys, each taken whole if any cell of it changes (warp-uniform).  Branches cost more here
              // than the products they save (measured with S itself as the sum): 24 heads x 8192 rows of 128 took 650 us a
              // layer step so, 667 with no branch, 680 with one for every 16 keys, 785 for 16 keys x 16 rows, 910 for
              // 8 keys x 16 rows.
#pragma unroll
              for (int c4 = 0; c4 < 2; ++c4) {
                const int zhi = zw_hi - 64 * h - 32 * c4;  // the half's distances: [zhi - 62, zhi]
                if (subtract ? zhi <= wp : (zhi - 62 > wp || zhi < 0)) continue;
#pragma unroll
                for (int cb = 4 * c4; cb < 4 * c4 + 4; ++cb) {
#pragma unroll
                  for (int hf = 0; hf < 2; ++hf) {
                    const int i0 = 8 * (cb - 2 * hf), i1 = i0 - 8;  // rows g8 and g8 + 8 of the half
                    const bool m0 = (i0 >= u) != subtract, m1 = (i1 >= u) != subtract;
                    const bool m2 = (i0 + 4 >= u) != subtract, m3 = (i1 + 4 >= u) != subtract;
                    const uint32_t a0 = m0 ? qr[2 * hf] : 0u, a1 = m1 ? qr[2 * hf + 1] : 0u;
                    const uint32_t a2 = m2 ? qr[2 * hf] : 0u, a3 = m3 ? qr[2 * hf + 1] : 0u;
                    mma_16816(f[hf] + 4 * cb, a0, a1, a2, a3, kk[cb] & slot0, kk[cb] & slot4);
                    if (SPLIT) {  // the other two products of the split scores
                      mma_16816(f[hf] + 4 * cb, a0, a1, a2, a3, kl[cb] & slot0, kl[cb] & slot4);
                      mma_16816(f[hf] + 4 * cb, m0 ? qrl[2 * hf] : 0u, m1 ? qrl[2 * hf + 1] : 0u, m2 ? qrl[2 * hf] : 0u,
                                m3 ? qrl[2 * hf + 1] : 0u, kk[cb] & slot0, kk[cb] & slot4);
                    }
                  }
                }
              }
            }
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              if (s_valid) {
                float sf[32];
                tc_ld_frag64(tS + ((uint32_t)(16 * hf) << 16), sf);
                tc_wait_ld();
#pragma unroll
                for (int e = 0; e < 32; e += 2) {
                  const float2 v = __fadd2_rn(make_float2(f[hf][e], f[hf][e + 1]), make_float2(sf[e], sf[e + 1]));
                  f[hf][e] = v.x;
                  f[hf][e + 1] = v.y;
                }
              }
              tc_st_frag64(tS + ((uint32_t)(16 * hf) << 16), f[hf]);
            }
            s_valid = true;
            tc_wait_st();
          }
        }
        float s[64];
        if (s_valid) {
          tc_ld32(tS, reinterpret_cast<uint32_t*>(s));
          tc_ld32(tS + 32, reinterpret_cast<uint32_t*>(s) + 32);
          tc_wait_ld();
        } else {
#pragma unroll
          for (int c = 0; c < 64; ++c) s[c] = 0.f;
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(B_SREAD + sb));
        // ---- causal mask on the diagonal tile, dropped keys (exact mode: no pair reaches the cell) ----
        if (dt == 0 || (MODE == ATF_MODE_EXACT && zmax_w > Wmax)) {
          const int zdrop = MODE == ATF_MODE_EXACT ? Wmax : 0x7FFFFFFF;
#pragma unroll
          for (int c = 0; c < 64; ++c) {
            const int z = zrow - 64 * h - c;
            s[c] = (z >= 0 && z <= zdrop) ? s[c] : -INFINITY;
          }
        }
        if (COUNT && row_ok) {
          const int c_lo = 64 * h, c_hi = min(64 * h + 63, zrow);  // causal cells of this thread's half
          if (c_hi >= c_lo) {
            if (MODE == ATF_MODE_EXACT) {
              cnt += (unsigned long long)p_all * (unsigned long long)(c_hi - c_lo + 1);
              for (int p = p_all; p < p_any; ++p) {
                const int lo = max(c_lo, zrow - sW[H - 1 - p]);
                cnt += (unsigned long long)max(0, c_hi - lo + 1);
              }
            } else {
              cnt += (unsigned long long)min(H, 8 * natoms) * (unsigned long long)(c_hi - c_lo + 1);
            }
          }
        }
        if (MODE == ATF_MODE_EXACT) {  // done with K of this tile
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(B_KEMPTY + ks));
        }

        // ---- reference maximum ----
        float scale_o = 1.f;
        if (t == 0 || safe) {
          float mx = -INFINITY;
#pragma unroll
          for (int c = 0; c < 64; ++c) mx = fmaxf(mx, s[c]);
          xch[h * 128 + row] = mx;
          if (!softmax_sync()) { ok = false; fail_site = 33; break; }
          mx = fmaxf(mx, xch[(h ^ 1) * 128 + row]);
          if (!softmax_sync()) { ok = false; fail_site = 33; break; }  // both have read: the area may be written again
          bool moved = false;
          if (mx > m_used && (m_used == -INFINITY || (mx - m_used) * kScaleLog2 > RESCALE_THRESHOLD)) {
            scale_o = m_used == -INFINITY ? 0.f : ex2_approx((m_used - mx) * kScaleLog2);
            m_used = mx;
            // Fast pass: the reference stays for the whole row, so it is put REF_HEADROOM above the diagonal tile's
            // maximum: sums overflow only ~120 log2 units above that maximum instead of ~60, and what the shift can
            // flush to zero lies 2^-66 below the diagonal's own largest term.
            if (!safe) m_used += REF_HEADROOM / kScaleLog2;
            moved = t > 0;  // nothing has been accumulated before the first tile
          }
          if (__any_sync(0xffffffffu, moved)) {
            // every product into O issued so far must be complete; the two threads of a row take half of O each
            if (!wait_or_abort(bar(B_PVDONE + ((g - 1) & 1)), ((g - 1) >> 1) & 1, abortp)) { ok = false; fail_site = 34; break; }
            tc_fence_after();
#pragma unroll
            for (int q4 = 0; q4 < D / 64; ++q4) {
              uint32_t o[32];
              tc_ld32(tO + (D / 2) * h + q4 * 32, o);
              tc_wait_ld();
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * scale_o);
              tc_st32(tO + (D / 2) * h + q4 * 32, o);
            }
            tc_wait_st();
          }
        }
        uint32_t pk[32];
        const float lsum = exp_half<POLY>(s, kScaleLog2, m_used == -INFINITY ? 0.f : -m_used * kScaleLog2, pk);
        overflow |= !(lsum < STALE_REF_GUARD);
        // the product that read the previous contents of this P buffer must be complete
        if (g >= 2 && !wait_or_abort(bar(B_PVDONE + sb), ((g - 2) >> 1) & 1, abortp)) { ok = false; fail_site = 35; break; }
        tc_st32(tP, pk);
        l_run = l_run * scale_o + lsum;
        if (TURNS && !safe) xch[h * 128 + row] = lsum;  // the diagonal tile's
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(B_PFULL + 2 * sb + h));
        p_mid = p_mid_next;
        e_cur = e_next;
        ++t;
      }
      if (ok && nt > 0 && !wait_or_abort(bar(B_OFULL), pass & 1, abortp)) { ok = false; fail_site = 36; }
      if (!safe && overflow && row_ok) s_redo = 1;
      if (!another_pass(pass)) break;
    }
    // ---- both halves of the row sum (after a fast pass in turns warp 2 has left them there), then the output ----
    if (!TURNS || redone) {
      xch[h * 128 + row] = l_run;
      if (ok && !softmax_sync()) { ok = false; fail_site = 37; }
    }
    const float l_tot = xch[h * 128 + row] + xch[(h ^ 1) * 128 + row];
    if (CUT && s_part[CUT ? 1 : 0]) {
      if (ok) {
        tc_fence_after();
        float* state = cut_state();
        float4* dst = reinterpret_cast<float4*>(state) + row;
#pragma unroll 1
        for (int q4 = 0; q4 < D / 64; ++q4) {
          const int c0 = (D / 2) * h + q4 * 32;
          float o[32];
          tc_ld32(tO + c0, reinterpret_cast<uint32_t*>(o));
          tc_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; e += 4) __stcg(dst + (c0 + e) / 4 * T, make_float4(o[e], o[e + 1], o[e + 2], o[e + 3]));
        }
        state[T * (D + h) + row] = xch[h * 128 + row];
        if (h == 0) state[T * (D + 2) + row] = m_used;
      }
      __threadfence();
    } else if (ok) {
      tc_fence_after();
      const float inv = 1.f / l_tot;
      __nv_bfloat16* orow = P.O + qrow * D;
#pragma unroll
      for (int q4 = 0; q4 < D / 64; ++q4) {
        const int cbase = (D / 2) * h + q4 * 32;  // group h writes its half of the row
        uint32_t o[32];
        tc_ld32(tO + cbase, o);
        tc_wait_ld();
        if (row_ok) {
#pragma unroll
          for (int e = 0; e < 32; e += 8) {
            uint4 v4;
            v4.x = pack_bf16x2(__uint_as_float(o[e]) * inv, __uint_as_float(o[e + 1]) * inv);
            v4.y = pack_bf16x2(__uint_as_float(o[e + 2]) * inv, __uint_as_float(o[e + 3]) * inv);
            v4.z = pack_bf16x2(__uint_as_float(o[e + 4]) * inv, __uint_as_float(o[e + 5]) * inv);
            v4.w = pack_bf16x2(__uint_as_float(o[e + 6]) * inv, __uint_as_float(o[e + 7]) * inv);
            *reinterpret_cast<uint4*>(orow + cbase + e) = v4;
          }
        }
      }
      if (P.LSE && row_ok && h == 0) P.LSE[qrow] = (m_used * kScaleLog2 + log2f(l_tot)) * 0.6931471805599453f;
      if (COUNT) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, off);
        if (lane == 0 && cnt) atomicAdd(P.kept + bhq, cnt);
      }
    }
  }

  if (fail_site) {
    atomicExch(P.status, 1u);
    atomicExch(P.status + 1, fail_site);
  }
  tc_fence_before();
  __syncthreads();
  if (CUT && tid == 0 && s_part[CUT ? 1 : 0] && !s_abort) st_release(P.flags + blockIdx.x, CUT_RUNS | CUT_STATE_THERE | (s_redo ? CUT_OVERFLOW : 0));
  if (warp == 0) tmem_dealloc(tmem_base, TMEM_COLS);
}

template <int D, bool SPLIT>
atf_status launch_pipe(const CUtensorMap& tq, const CUtensorMap& tql, const CUtensorMap& tk, const CUtensorMap& tkl,
                       const CUtensorMap& tv, AtfPipeParams P, const AtfTable& t, int B, int mode, bool count,
                       cudaStream_t s) {
  const int tiles = (P.N + T - 1) / T - (P.N - P.Nq) / T;  // from the first one with a query row
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  // Order of the tiles.  Rows of different lengths: longest first over all heads, so that no head's longest row starts when the
  // others are done (us, head by head -> so: 24 heads x 8192 rows 596 -> 581, 3000 rows 174 -> 141, 3500 of 5000 277 -> 250, 14
  // heads x 5000 of 8000, d = 64, 224 -> 200).  Rows of about the same length: head by head (2048 rows of 16384 403, over all
  // heads 418; B = 2, 4096 of 8192 778, 795; 2 x 2 heads, 16000 of 60000 1226, 1264; but 14 heads, 6000 of 20000, 599, 589).  Head by
  // head, too, where a head has tiles for half the SMs, so that it alone comes near a sorted wave, and longest first would leave the
  // last wave, of the shortest rows, idle for more than a quarter of a mean tile (2 x 2 heads: 14700 of 25000, last wave 0.14 full, 430
  // against 451, 16384 of 31955, 0.49, 580, 612; 13100 of 22277, 0.81, 354 against 340: longest first; 14 heads: 8000 of 13607, 64
  // tiles, 0.05, 490, 501, 16384 of 31955, 0.20, 1969, 2015; 14700 of 25000, 0.97, 1378, 1349: longest first; fewer tiles: 1664 of 2605,
  // 24 heads, 0.27, 129, 109, 3200 of 5935, B = 2, 0.43, 541, 524: longest first).
  // Groups of heads whose K and V take up to 64 MB together, because what all SMs read at a time is to stay in L2: 24 heads x 131072 rows
  // 85.0 ms, in groups of 128 MB 85.5, over all heads 88.8.  32 to 48 MB are within 1.5 % of 64 (7000 to 131072 rows, 39 shapes).
  // Where one KV head's alone take more, head by head (28/4 heads of 128, full attention: 262144 rows 417, grouped 417 ms, 524288 1667,
  // 1730, 1048576 6757, 8820, coarse 5675, 5840, exact 5935, 5915; in the slow one the power cap holds the clock at 945 MHz instead of
  // 1410, presumably for K and V that come from DRAM again).
  const int64_t dlim = ((int64_t)t.w[D / 2 - 1] + T - 1) / T + 1, per_kv = P.Hq / P.Hkv;
  const int64_t longest = std::min<int64_t>((P.N + T - 1) / T, dlim), shortest = std::min<int64_t>((P.N - P.Nq) / T + 1, dlim);
  P.heads = P.Hq * B;
  const int64_t rest = ATF_SMS - 1 - ((int64_t)tiles * P.heads - 1) % ATF_SMS;  // blocks that the last wave lacks
  int64_t group = 1;
  if (P.cuts) {
    group = P.heads;
  } else if (2 * shortest <= longest && (tiles < 64 || 8 * rest * shortest <= ATF_SMS * (longest + shortest))) {
    const int64_t fit = (64ll << 20) / ((int64_t)P.N * D * 2 * (SPLIT ? 3 : 2)) * per_kv;
    if (fit > 0) {
      const int64_t groups = (P.heads + fit - 1) / fit;
      group = std::min<int64_t>(((P.heads + groups - 1) / groups + per_kv - 1) / per_kv * per_kv, P.heads);
    }
  }
  P.group = (int)std::max<int64_t>(group, (P.heads + 65534) / 65535);  // gridDim.y
  P.jobs = tiles * P.group;
  if ((int64_t)tiles * P.group > 0x7FFFFF00) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill: problem too large for the grid");
  cfg.gridDim = dim3((unsigned)(P.jobs + P.cuts), (P.heads + P.group - 1) / P.group);
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cfg.blockDim = dim3(PP_THREADS);
#define ATF_PP_LAUNCH(MODE_, COUNT_, TURNS_)                                                          \
  do {                                                                                                 \
    auto kern = P.cuts && !COUNT_ ? atf_prefill_pipe_kernel<D, MODE_, COUNT_, SPLIT, TURNS_, !COUNT_>  \
                                  : atf_prefill_pipe_kernel<D, MODE_, COUNT_, SPLIT, TURNS_, false>;   \
    const int smem = PipeSmem<D, SPLIT, MODE_ == ATF_MODE_EXACT && !SPLIT, TURNS_>::DYN_BYTES;                 \
    ATF_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));     \
    cfg.dynamicSmemBytes = smem;                                                                       \
    ATF_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kern, tq, tql, tk, tkl, tv, P, t));                        \
  } while (0)
  // In turns or in step: the results are the same, bit for bit.  In turns pays where the softmax holds the pace and no warp has
  // cells to finish (us, in step -> in turns: coarse, 24 heads of 128, 8192 rows 415 -> 397, 32768 5595 -> 5105, 131072 81.3 -> 78.0 ms,
  // 4000 of 61003 2596 -> 2413; 14 heads of 64, 4096 rows, coarse 59.2 -> 57.4, 32768 rows 2539 -> 2381, full 2718 -> 2518).  Full
  // attention at d = 128 is bound by the tensor pipe: the same either way up to 4096 rows, above that 1 to 2 % less in turns, inside the
  // spread of one side's runs (8192 rows 433, 426; 32768 5760, 5700); so is the split-precision form, whose operands leave no room for a
  // second exchange area.  Exact mode's finish is slower by one warp for all 128 keys (8192 rows 596 -> 690), and a kernel with both forms of it slower in either; calls that count terms stay in step.
  if (mode == ATF_MODE_EXACT) {
    if (count) ATF_PP_LAUNCH(ATF_MODE_EXACT, true, false); else ATF_PP_LAUNCH(ATF_MODE_EXACT, false, false);
  } else if (count) {
    ATF_PP_LAUNCH(ATF_MODE_COARSE, true, false);
  } else if (!SPLIT && (D == 64 || t.w[0] < P.N - 1)) {
    ATF_PP_LAUNCH(ATF_MODE_COARSE, false, !SPLIT);
  } else {
    ATF_PP_LAUNCH(ATF_MODE_COARSE, false, false);
  }
#undef ATF_PP_LAUNCH
  return ATF_OK;
}

}  // namespace

atf_status atf_launch_prefill_pipe(const CUtensorMap& tk, const CUtensorMap& tv, const AtfPipeParams& P,
                                   const AtfTable& t, int B, int d, int mode, bool count, cudaStream_t s) {
  return d == 64 ? launch_pipe<64, false>(tk, tk, tk, tk, tv, P, t, B, mode, count, s)
                 : launch_pipe<128, false>(tk, tk, tk, tk, tv, P, t, B, mode, count, s);
}

atf_status atf_launch_prefill_pipe_split(const CUtensorMap& tqh, const CUtensorMap& tql, const CUtensorMap& tkh,
                                         const CUtensorMap& tkl, const CUtensorMap& tv, const AtfPipeParams& P,
                                         const AtfTable& t, int B, int d, int mode, bool count, cudaStream_t s) {
  return d == 64 ? launch_pipe<64, true>(tqh, tql, tkh, tkl, tv, P, t, B, mode, count, s)
                 : launch_pipe<128, true>(tqh, tql, tkh, tkl, tv, P, t, B, mode, count, s);
}

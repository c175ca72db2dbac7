// atf_prefill_split: the windowed causal prefill with scores of more than bf16 input precision
// (App. D, "Precision as the other side of the compute-accuracy trade": a low-precision product is
// split to recover accuracy, paid for with part of what the window saves; Sec. 6.2 had to score
// five tasks with fp32 attention scores because bf16 rounding flipped low-margin retrievals).
//
// Q and K arrive as fp32, already rotated and never rounded to bf16.  A pre-pass writes each as
// two bf16 tensors, hi = bf16(x) and lo = bf16(x - hi) (hi + lo holds x to 2^-17 of its size), in
// the pair-interleaved lowest-frequency-first column order of atf_prefill, so the live pairs of
// a tile are again a column prefix.  The scores are
//     S = Q_hi K_hi^T + Q_hi K_lo^T + Q_lo K_hi^T
// accumulated in fp32 in tensor memory: three tcgen05.mma per 16-column step of the LIVE depth
// only (the lo x lo product, 2^-16 of the result, is left out).  The kernel is the prefill kernel
// of atf_prefill_pipe.cu in its SPLIT form: both Q parts resident, a K stage = a hi tile and a lo
// tile, the per-cell finish of the exact mode with the same three products, every exponential
// MUFU ex2 (no polynomial), the row sums from the unrounded fp32 values.  V, P and O are bf16
// operands with fp32 accumulation as in atf_prefill; term counts are those of atf_prefill.
#include <cuda.h>

#include "atf_common.cuh"
#include "atf_prefill_pipe.cuh"

namespace {

constexpr int T = 128;

// The pre-pass, one launch: band schedule, then hi = bf16(x), lo = bf16(x - hi) of Q and of K in the pair-interleaved
// column order.  One thread moves eight pairs of a row; memory bounds it (10001 rows of 24 + 8 heads of 128: 49 us, 327 MB).
// Q and K may be what a rotation that still runs is writing: no pointer is __restrict__, the loads stay behind the wait.
__global__ void __launch_bounds__(ATF_PREP_THREADS)
atf_split_prep_kernel(const __grid_constant__ AtfTable table, int mode, int ndt, int sched_blocks, uint32_t* sched,
                      int cuts, unsigned int* flags,
                      const float* Q, const float* K, __nv_bfloat16* Qhi,
                      __nv_bfloat16* Qlo, __nv_bfloat16* Khi, __nv_bfloat16* Klo,
                      int64_t rows_q, int64_t rows_k, int D) {
  grid_dependency_wait();
  grid_dependency_launch();
  const int H = D / 2, per_row = D / 16;
  if ((int)blockIdx.x < sched_blocks) return atf_write_schedule(table, mode, H, ndt, sched, cuts, flags);
  const int64_t gid = (int64_t)(blockIdx.x - sched_blocks) * ATF_PREP_THREADS + threadIdx.x;
  int64_t row = gid / per_row;
  const int c = (int)(gid % per_row);           // dims 8c .. 8c + 7 of each half, pairs 8j .. 8j + 7 in falling order
  if (row >= rows_q + rows_k) return;
  const bool is_k = row >= rows_q;
  if (is_k) row -= rows_q;
  const float* src = (is_k ? K : Q) + row * D + 8 * c;
  float x[8], y[8];
  *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(src);
  *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(src + 4);
  *reinterpret_cast<float4*>(y) = *reinterpret_cast<const float4*>(src + H);
  *reinterpret_cast<float4*>(y + 4) = *reinterpret_cast<const float4*>(src + H + 4);
  uint32_t hi[8], lo[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float a = x[7 - i], b = y[7 - i];
    hi[i] = pack_bf16x2(a, b);
    lo[i] = pack_bf16x2(a - bf16lo_to_f32(hi[i]), b - bf16hi_to_f32(hi[i]));
  }
  const int64_t off = row * D + 16 * (per_row - 1 - c);
  uint4* dh = reinterpret_cast<uint4*>((is_k ? Khi : Qhi) + off);
  uint4* dl = reinterpret_cast<uint4*>((is_k ? Klo : Qlo) + off);
  dh[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
  dh[1] = make_uint4(hi[4], hi[5], hi[6], hi[7]);
  dl[0] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  dl[1] = make_uint4(lo[4], lo[5], lo[6], lo[7]);
}

size_t part_bytes(int B, int H, int64_t N, int d) {
  size_t b = (size_t)B * H * N * d * 2;
  return (b + 255) & ~(size_t)255;
}

}  // namespace

atf_status atf_validate_table(const char* who, const int64_t* table, int d, int64_t N, AtfTable* out);

// band schedule of the kernel: eight words per tile distance
static size_t split_sched_bytes(int64_t N) { return ((size_t)((N + T - 1) / T + 1) * 32 + 255) & ~(size_t)255; }

size_t atf_prefill_split_workspace_bytes(int B, int Hq, int Hkv, int64_t N, int d) {
  return ATF_WS_HEADER + split_sched_bytes(N) + 2 * part_bytes(B, Hq, N, d) + 2 * part_bytes(B, Hkv, N, d);
}

extern "C" atf_status atf_prefill_split_chunk(const float* Q, const float* K, const void* V, void* O, float* LSE, int B,
                                              int Hq, int Hkv, int64_t Nq, int64_t N, int d, const int64_t* table,
                                              int causal, const atf_opts* opts, void* stream) {
  if (!Q || !K || !V || !O) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill_split: null pointer");
  if (d != 64 && d != 128) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill_split: d must be 64 or 128 (got %d)", d);
  if (B < 1 || Hq < 1 || Hkv < 1 || N < 1) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill_split: bad shape");
  if (Nq < 1 || Nq > N) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill_split: need 1 <= Nq <= N (got Nq = %lld, N = %lld)", (long long)Nq, (long long)N);
  if (Hq % Hkv) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill_split: Hq must be a multiple of Hkv");
  if (!causal) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill_split: only causal attention is defined (distance z = n - m >= 0)");
  if (N >= (1ll << 31) - 4 * T) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill_split: N too large");
  if (Hq > 65535 || B > 65535) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill_split: B and Hq must be <= 65535");
  if (((uintptr_t)Q | (uintptr_t)K | (uintptr_t)V | (uintptr_t)O) & 15)
    return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill_split: pointers must be 16-byte aligned");
  const int mode = opts ? opts->mode : ATF_MODE_EXACT;
  if (mode != ATF_MODE_EXACT && mode != ATF_MODE_COARSE) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill_split: unknown mode %d", mode);
  if (opts && (opts->kcache_groups || opts->rope_tables))
    return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill_split: kcache_groups and rope_tables are not taken by this call");
  AtfTable t;
  atf_status st = atf_validate_table("atf_prefill_split", table, d, N, &t);
  if (st != ATF_OK) return st;

  AtfWorkspace ws = atf_bound_workspace();
  if (opts && opts->workspace) ws = AtfWorkspace{opts->workspace, opts->workspace_bytes};
  const size_t need = atf_prefill_split_workspace_bytes(B, Hq, Hkv, N, d);
  if (!ws.ptr) return atf_fail(ATF_ERR_WORKSPACE, "atf_prefill_split: no workspace bound");
  if (ws.bytes < need) return atf_fail(ATF_ERR_WORKSPACE, "atf_prefill_split: workspace has %zu bytes, needs %zu", ws.bytes, need);
  if ((uintptr_t)ws.ptr & 255) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill_split: workspace must be 256-byte aligned");

  char* base = (char*)ws.ptr;
  const size_t qb = part_bytes(B, Hq, Nq, d), kb = part_bytes(B, Hkv, N, d);
  char* parts = base + ATF_WS_HEADER + split_sched_bytes(N);
  __nv_bfloat16* Qhi = (__nv_bfloat16*)parts;
  __nv_bfloat16* Qlo = (__nv_bfloat16*)(parts + qb);
  __nv_bfloat16* Khi = (__nv_bfloat16*)(parts + 2 * qb);
  __nv_bfloat16* Klo = (__nv_bfloat16*)(parts + 2 * qb + kb);
  cudaStream_t s = (cudaStream_t)stream;
  const size_t used = ATF_WS_HEADER + split_sched_bytes(N) + 2 * (qb + kb);  // `need` is that of N query rows
  const int cuts = opts && opts->kept_terms ? 0 : atf_prefill_cuts(N, Nq, (int64_t)B * Hq, t.w[d / 2 - 1], d, ws.bytes - used);
  float* state = (float*)(base + used);
  unsigned int* flags = (unsigned int*)(state + atf_cut_floats(d));
  {
    const int64_t rows_q = (int64_t)B * Hq * Nq, rows_k = (int64_t)B * Hkv * N;
    if ((rows_q * (d / 8) + 255) / 256 > 0x7FFFFFFF) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill_split: problem too large for the repack grid");
    const int sb = atf_sched_blocks(N);
    const int64_t blocks = sb + ((rows_q + rows_k) * (d / 16) + ATF_PREP_THREADS - 1) / ATF_PREP_THREADS;
    if (blocks > 0x7FFFFFFF) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill_split: problem too large for the repack grid");
    ATF_CUDA_CHECK(atf_launch_overlapped(atf_split_prep_kernel, dim3((unsigned)blocks), ATF_PREP_THREADS, 0, s, t, mode, (int)((N + T - 1) / T), sb,
                                                                        (uint32_t*)(base + ATF_WS_HEADER), cuts, flags, Q, K, Qhi, Qlo, Khi,
                                                                        Klo, rows_q, rows_k, d));
  }
  CUtensorMap tqh, tql, tkh, tkl, tv;
  if ((st = atf_make_tile_map(&tqh, Qhi, (int64_t)B * Hq, Nq, d, Nq, T)) != ATF_OK) return st;
  if ((st = atf_make_tile_map(&tql, Qlo, (int64_t)B * Hq, Nq, d, Nq, T)) != ATF_OK) return st;
  if ((st = atf_make_tile_map(&tkh, Khi, (int64_t)B * Hkv, N, d, N, T)) != ATF_OK) return st;
  if ((st = atf_make_tile_map(&tkl, Klo, (int64_t)B * Hkv, N, d, N, T)) != ATF_OK) return st;
  if ((st = atf_make_tile_map(&tv, V, (int64_t)B * Hkv, N, d, N, T)) != ATF_OK) return st;

  AtfPipeParams P;
  P.sched = (uint32_t*)(base + ATF_WS_HEADER);
  P.Q = nullptr;
  P.Qhi = Qhi;
  P.Qlo = Qlo;
  P.O = (__nv_bfloat16*)O;
  P.LSE = LSE;
  P.cuts = cuts;
  P.flags = flags;
  P.state = state;
  P.kept = opts ? (unsigned long long*)opts->kept_terms : nullptr;
  P.status = (unsigned int*)base;
  P.Hq = Hq;
  P.Hkv = Hkv;
  P.N = (int)N;
  P.Nq = (int)Nq;
  return atf_launch_prefill_pipe_split(tqh, tql, tkh, tkl, tv, P, t, B, d, mode, P.kept != nullptr, s);
}

extern "C" atf_status atf_prefill_split(const float* Q, const float* K, const void* V, void* O, float* LSE, int B, int Hq,
                                        int Hkv, int64_t N, int d, const int64_t* table, int causal,
                                        const atf_opts* opts, void* stream) {
  return atf_prefill_split_chunk(Q, K, V, O, LSE, B, Hq, Hkv, N, N, d, table, causal, opts, stream);
}

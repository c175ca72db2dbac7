// atf_prefill: windowed causal attention for all query rows (Sec. 3.3, Fig. 3) on the sm_100a
// tensor cores.  This file holds the host side (validation, workspace, tensor maps, entry points)
// and the layout pre-pass; the kernel is in atf_prefill_pipe.cu.
//
// Data layout.  A pre-pass copies K into a pair-interleaved column order, lowest frequency first:
// column 2p holds dim (h-1-p), column 2p+1 holds dim (d-1-p), h = d/2; the kernel puts its rows of
// Q into the same order as it reads them (a row of Q is read by one CTA, one of K by many).  A
// query-key dot product does not change under a common column permutation, and in this order
// the pairs that are live at a distance (a contiguous low-frequency slice, Sec. 3.3) are a
// PREFIX of the columns, so "advance the start of the pair loop" becomes "contract over the
// first few 16-column MMA steps", and the K columns beyond the prefix are not loaded.  The K
// pass can also write the tiled group-major K cache that decode reads (Sec. 7.2: the cache the
// prefill wrote is the cache the decode reads).
#include <cuda.h>

#include "atf_common.cuh"
#include "atf_prefill_pipe.cuh"

namespace {

constexpr int T = 128;  // query rows per tile and key columns per tile

// The pre-pass, one launch: band schedule, and K in the column order above.  One thread moves eight pairs of a row: 16
// bytes of each half row become 32 bytes of output, so that the pass is bound by memory (8 heads x 8192 rows of 128 into
// the copy and the cache: 11.7 us from cold caches, 50 MB).  The source holds src_head_rows rows per head of which the
// first n_per_head are copied, the result is dense.
// With Kg the same eight pairs, a group of the tiled group-major K cache (kg_tiles tiles per head), also go there for the
// rows from kg_first_row on.
// X may be what a rotation that still runs is writing (launch: atf_launch_overlapped), so no pointer is __restrict__: the loads
// are ordinary ones and stay behind the wait.
__global__ void __launch_bounds__(ATF_PREP_THREADS)
atf_prefill_prep_kernel(const __grid_constant__ AtfTable table, int mode, int ndt, int sched_blocks, uint32_t* sched,
                        int cuts, unsigned int* flags,
                        const __nv_bfloat16* X, __nv_bfloat16* Y, int64_t rows, int D,
                        int64_t n_per_head, int64_t src_head_rows, __nv_bfloat16* Kg, int64_t kg_tiles,
                        int64_t kg_first_row) {
  grid_dependency_wait();  // before the prefill kernel may start: it reads Q ahead of its own wait
  grid_dependency_launch();
  const int H = D / 2, per_row = D / 16;
  if ((int)blockIdx.x < sched_blocks) return atf_write_schedule(table, mode, H, ndt, sched, cuts, flags);
  const int64_t gid = (int64_t)(blockIdx.x - sched_blocks) * ATF_PREP_THREADS + threadIdx.x;
  if (gid >= rows * per_row) return;
  const int64_t row = gid / per_row;
  const int c = (int)(gid % per_row);           // dims 8c .. 8c + 7 of each half, pairs 8j .. 8j + 7 in falling order
  const int j = per_row - 1 - c;
  const int64_t head = row / n_per_head;
  const int64_t m = row - head * n_per_head;  // position of the row in its head
  const __nv_bfloat16* src = X + (head * src_head_rows + m) * D + 8 * c;
  const uint4 lo = *reinterpret_cast<const uint4*>(src), hi = *reinterpret_cast<const uint4*>(src + H);
  uint4 a, b;
  a.x = __byte_perm(lo.w, hi.w, 0x7632);
  a.y = __byte_perm(lo.w, hi.w, 0x5410);
  a.z = __byte_perm(lo.z, hi.z, 0x7632);
  a.w = __byte_perm(lo.z, hi.z, 0x5410);
  b.x = __byte_perm(lo.y, hi.y, 0x7632);
  b.y = __byte_perm(lo.y, hi.y, 0x5410);
  b.z = __byte_perm(lo.x, hi.x, 0x7632);
  b.w = __byte_perm(lo.x, hi.x, 0x5410);
  uint4* dst = reinterpret_cast<uint4*>(Y + row * D + 16 * j);
  dst[0] = a;
  dst[1] = b;
  if (Kg && m >= kg_first_row) {
    const int64_t KT = 8192 / D;  // keys per 16 KiB tile
    const int64_t tile = m / KT, kin = m % KT;
    const int swap = (int)((kin >> 2) & 1);  // keys with bit 2 set store their two 16-byte halves swapped
    uint4* g = reinterpret_cast<uint4*>(Kg + (((head * kg_tiles + tile) * (D / 16) + j) * KT + kin) * 16);
    g[swap] = a;
    g[swap ^ 1] = b;
  }
}

size_t repack_bytes(int B, int H, int64_t N, int d) {
  size_t b = (size_t)B * H * N * d * 2;
  return (b + 255) & ~(size_t)255;
}

}  // namespace

atf_status atf_validate_table(const char* who, const int64_t* table, int d, int64_t N, AtfTable* out);

// band schedule: one 32-byte record (eight words) per tile distance a launch over N keys can meet
static int sched_entries(int64_t N) { return (int)((N + T - 1) / T) + 1; }
static size_t sched_bytes(int64_t N) { return ((size_t)sched_entries(N) * 32 + 255) & ~(size_t)255; }

// Counts room for a reordered Q, which an earlier form of the pre-pass wrote: callers' sizes stay what they were.  What a workspace
// has behind schedule and K, this room or more, holds the state of cut tiles: with less than that state takes a call is not cut
// (atf_prefill_cuts; from B Hq N = 40000 on the size asked for here is enough).
size_t atf_prefill_workspace_bytes(int B, int Hq, int Hkv, int64_t N, int d) {
  return ATF_WS_HEADER + sched_bytes(N) + repack_bytes(B, Hq, N, d) + repack_bytes(B, Hkv, N, d);
}
static size_t prefill_chunk_workspace_bytes(int B, int Hq, int Hkv, int64_t Nq, int64_t N, int d) {
  return ATF_WS_HEADER + sched_bytes(N) + repack_bytes(B, Hq, Nq, d) + repack_bytes(B, Hkv, N, d);
}

// kv_head_rows: rows between two heads of K and of V in memory (>= N; N for dense tensors).  A caller that
// fills a full-length cache chunk by chunk passes the cache's length here and the rows present as N.
atf_status atf_prefill_impl(const void* Q, const void* K, const void* V, void* O, float* LSE, int B, int Hq, int Hkv,
                            int64_t Nq, int64_t N, int d, const int64_t* table, int causal, const atf_opts* opts,
                            void* stream, int64_t kv_head_rows) {
  if (!Q || !K || !V || !O) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill: null pointer");
  if (kv_head_rows < N) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill: K/V head stride smaller than N");
  if (Nq < 1 || Nq > N) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill: need 1 <= Nq <= N (got Nq = %lld, N = %lld)", (long long)Nq, (long long)N);
  if (d != 64 && d != 128) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill: d must be 64 or 128 (got %d)", d);
  if (B < 1 || Hq < 1 || Hkv < 1 || N < 1) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill: bad shape");
  if (Hq % Hkv) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill: Hq must be a multiple of Hkv");
  if (!causal) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill: only causal attention is defined (distance z = n - m >= 0)");
  if (N >= (1ll << 31) - 4 * T) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill: N too large");
  if (Hq > 65535 || B > 65535) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill: B and Hq must be <= 65535");
  if (((uintptr_t)Q | (uintptr_t)K | (uintptr_t)V | (uintptr_t)O) & 15)
    return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill: pointers must be 16-byte aligned");
  int mode = opts ? opts->mode : ATF_MODE_EXACT;
  if (mode != ATF_MODE_EXACT && mode != ATF_MODE_COARSE) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill: unknown mode %d", mode);
  if (opts && opts->kcache_groups) {
    if (opts->kcache_capacity < N) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill: kcache_capacity (%lld) is smaller than N", (long long)opts->kcache_capacity);
    if ((uintptr_t)opts->kcache_groups & 15) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill: kcache_groups must be 16-byte aligned");
  }
  AtfTable t;
  atf_status st = atf_validate_table("atf_prefill", table, d, N, &t);
  if (st != ATF_OK) return st;

  // Every pair reaches every key (full attention): there is nothing to finish per cell, and the two modes are one computation,
  // bit for bit.  The coarse form of the kernel has a third K stage where the exact one keeps its copy of Q, and the softmax
  // warps need not release K (24 heads of 128: 1000 rows 42.8 -> 24.6 us, 32768 6.00 -> 5.82 ms, 131072 92.3 -> 90.4 ms;
  // two K stages alone had cost the long ones 1 %).
  if (t.w[0] >= N - 1) mode = ATF_MODE_COARSE;

  AtfWorkspace ws = atf_bound_workspace();
  if (opts && opts->workspace) ws = AtfWorkspace{opts->workspace, opts->workspace_bytes};
  const size_t need = prefill_chunk_workspace_bytes(B, Hq, Hkv, Nq, N, d);
  if (!ws.ptr) return atf_fail(ATF_ERR_WORKSPACE, "atf_prefill: no workspace bound");
  if (ws.bytes < need) return atf_fail(ATF_ERR_WORKSPACE, "atf_prefill: workspace has %zu bytes, needs %zu", ws.bytes, need);
  if ((uintptr_t)ws.ptr & 255) return atf_fail(ATF_ERR_INVALID_ARG, "atf_prefill: workspace must be 256-byte aligned");

  char* base = (char*)ws.ptr;
  uint32_t* sched = (uint32_t*)(base + ATF_WS_HEADER);
  __nv_bfloat16* Kp = (__nv_bfloat16*)(base + ATF_WS_HEADER + sched_bytes(N));
  cudaStream_t s = (cudaStream_t)stream;
  // The state of cut tiles lies where the reordered Q that `need` counts once was; a call that counts terms does not cut.
  const size_t used = ATF_WS_HEADER + sched_bytes(N) + repack_bytes(B, Hkv, N, d);
  const int cuts = opts && opts->kept_terms ? 0 : atf_prefill_cuts(N, Nq, (int64_t)B * Hq, t.w[d / 2 - 1], d, ws.bytes - used);
  float* state = (float*)(base + used);
  unsigned int* flags = (unsigned int*)(state + atf_cut_floats(d));

  {
    const int64_t rows_q = (int64_t)B * Hq * Nq, rows_k = (int64_t)B * Hkv * N;
    if ((rows_q * (d / 8) + 255) / 256 > 0x7FFFFFFF) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill: problem too large for the repack grid");
    const int sb = atf_sched_blocks(N);
    const int64_t blocks = sb + (rows_k * (d / 16) + ATF_PREP_THREADS - 1) / ATF_PREP_THREADS;
    if (blocks > 0x7FFFFFFF) return atf_fail(ATF_ERR_UNSUPPORTED, "atf_prefill: problem too large for the repack grid");
    __nv_bfloat16* Kg = opts ? (__nv_bfloat16*)opts->kcache_groups : nullptr;
    const int64_t kt = 8192 / d;
    const int64_t kg_tiles = Kg ? (opts->kcache_capacity + kt - 1) / kt : 0;
    ATF_CUDA_CHECK(atf_launch_overlapped(
        atf_prefill_prep_kernel, dim3((unsigned)blocks), ATF_PREP_THREADS, 0, s, t, mode, (int)((N + T - 1) / T), sb, sched, cuts, flags, (const __nv_bfloat16*)K,
        Kp, rows_k, d, N, kv_head_rows, Kg, kg_tiles, N - Nq));
  }

  CUtensorMap tk, tv;
  if ((st = atf_make_tile_map(&tk, Kp, (int64_t)B * Hkv, N, d, N, T)) != ATF_OK) return st;
  if ((st = atf_make_tile_map(&tv, V, (int64_t)B * Hkv, N, d, kv_head_rows, T)) != ATF_OK) return st;

  AtfPipeParams P;
  P.sched = sched;
  P.Q = (const __nv_bfloat16*)Q;
  P.Qhi = P.Qlo = nullptr;
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
  return atf_launch_prefill_pipe(tk, tv, P, t, B, d, mode, P.kept != nullptr, s);
}

extern "C" atf_status atf_prefill_chunk_ex(const void* Q, const void* K, const void* V, void* O, float* LSE, int B,
                                           int Hq, int Hkv, int64_t Nq, int64_t N, int d, const int64_t* table,
                                           int causal, const atf_opts* opts, void* stream) {
  return atf_prefill_impl(Q, K, V, O, LSE, B, Hq, Hkv, Nq, N, d, table, causal, opts, stream, N);
}

extern "C" atf_status atf_prefill_ex(const void* Q, const void* K, const void* V, void* O, float* LSE, int B, int Hq,
                                     int Hkv, int64_t N, int d, const int64_t* table, int causal,
                                     const atf_opts* opts, void* stream) {
  return atf_prefill_chunk_ex(Q, K, V, O, LSE, B, Hq, Hkv, N, N, d, table, causal, opts, stream);
}

extern "C" atf_status atf_prefill_chunk(const void* Q, const void* K, const void* V, void* O, float* LSE, int B, int Hq,
                                        int Hkv, int64_t Nq, int64_t N, int d, const int64_t* table, int causal,
                                        void* stream) {
  return atf_prefill_chunk_ex(Q, K, V, O, LSE, B, Hq, Hkv, Nq, N, d, table, causal, nullptr, stream);
}

extern "C" atf_status atf_prefill(const void* Q, const void* K, const void* V, void* O, float* LSE, int B, int Hq,
                                  int Hkv, int64_t N, int d, const int64_t* table, int causal, void* stream) {
  return atf_prefill_ex(Q, K, V, O, LSE, B, Hq, Hkv, N, d, table, causal, nullptr, stream);
}

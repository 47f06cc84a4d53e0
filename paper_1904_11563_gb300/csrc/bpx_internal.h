// Internal declarations shared by the host code and the CUDA translation
// units of libbpx.  Not part of the ABI.
#pragma once

#include <cstddef>
#include <cstdint>
#include <string>
#include <vector>

#include "bpx.h"

// Host-side code graph (Section III): cells of each column, sources of each
// cell, and the transposed source -> cells adjacency the scheduler walks.
struct bpx_code {
  int variant = 0, n = 0, k = 0, e = 0, b = 0, q_e = 0;
  int S = 0, num_cells = 0, num_edges = 0, sigma = 0;
  double eps = 0.0;
  std::vector<int32_t> col_ptr, cell_ptr, cell_src, col_of_cell, heights, proj_p, proj_q;
  std::vector<int32_t> src_ptr, src_cell;  // source -> cells (ascending cell id)
  // Two-dimensional scheme (source s = z k + l is the block product A_z B_l):
  // every cell as a list of products of summed operands, term i of cell c at
  // [t2_ptr[c], t2_ptr[c+1]) = (A operand t2_a[i], B operand t2_b[i]); A
  // operand e sums the row blocks a2_blk[a2_ptr[e] ..], B operand f the
  // column blocks b2_blk[b2_ptr[f] ..]; t2_order lists the cells by
  // decreasing term count (ties by id); gray2 counts cells with > 1 term.
  std::vector<int32_t> t2_ptr, t2_a, t2_b, a2_ptr, a2_blk, b2_ptr, b2_blk, t2_order;
  int gray2 = 0;
  // Schedule: every cell's initial word (count and id sum, sched_count_bits;
  // empty when 32 bits do not hold them), and for a projection grid -- each
  // source (z, l) in one cell of every column j, cell = affine[j] + affine[n
  // + j] z + affine[2 n + j] l -- that table (else empty).
  std::vector<uint32_t> word0;
  std::vector<int32_t> affine;
  int32_t live_cells[8] = {};  // cells that masks of e erased columns leave: eight quantiles over the masks
};

namespace bpx {

// Thread-local error text; returns `code` for `return fail(...)`.
int fail(int code, const char* fmt, ...);
void clear_error();

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Byte offsets of every array in the device workspace.  The graph section is
// filled once by bpx_workspace_init; the plan section by bpx_schedule; the
// product and staging sections by bpx_coded_products.
struct WsLayout {
  // graph (int32)
  size_t g_hdr, g_col_of_cell, g_cell_ptr, g_cell_src, g_src_ptr, g_src_cell;
  size_t g_t2_ptr, g_t2_a, g_t2_b, g_a2_ptr, g_a2_blk, g_b2_ptr, g_b2_blk, g_t2_order;
  // plan (int32)
  size_t p_info, p_ctr, p_cnt, p_surv, p_direct, p_front0, p_pos, p_word;
  size_t p_depth, p_resolver, p_order, p_wave_ptr, p_cursor;  // p_word, p_cursor: also uploaded (word0, affine)
  size_t p_pl_res, p_pl_ptr, p_pl_list;  // peel list: resolver and subtrahends per order entry
  size_t plan_end;
  // products (float, num_cells * h * N)
  size_t products;
  // staging for the tensor-core paths (bf16 / fp8 operands; exact-slice
  // digit planes in a_hi / b_hi)
  size_t a_hi, a_lo, b_hi, b_lo, a_scale, b_scale;
  size_t a_3, b_3;  // FP32 on the tensor cores: the third bf16 parts
  // exact-slice: max |A| per row position (h words) then max |B| per column
  // (N words), as float bits; decoded sources as exact int64 (S h N)
  size_t ex_amax, ex_c64;
  // exact-slice, digits narrower than 8 bits: every source row's digit planes
  // as int8, computed once (0 = no such region)
  size_t ex_src;
  size_t total;
};

// Exact-slice representation of a code (see bpx_exact_params): digit width
// w, digit planes S (also the number of kept diagonals), fixed-point bits,
// K elements per exact FP32 accumulation segment, K padded to 64.
struct ExactParams {
  int w = 0, S = 0, bits = 0, seg = 0, Kp = 0;
  int step = 1, np = 0;  // diagonals computed: S - 1, S - 1 - step, ...: np of them (see exact_pair_digits)
};

// Fills *P for the code's sigma and K; BPX_ERR_UNSUPPORTED (with a message)
// when the digits or the exact integer sums would not fit.
int exact_params(const bpx_code* c, int K, ExactParams* P);

// The whole path's form for narrow digits (w <= 4: codes of sigma > 16, S 6
// or 8): B plane l holds two of B's digits, E_{l-1} 2^w + E_l (plane 0: E_0),
// still exact in bf16 (at most 136), so that the diagonals S - 1, S - 3, ...
// of A digits and these planes, A_i x plane d - i, hold the same kept digit
// pairs as all S diagonals: 12 products instead of 21 (S = 6), 20 instead of
// 36 (S = 8), and half the product planes.  Sets step 2, np = S / 2 and the
// segment for the larger products, where the int32 diagonal sums still fit.
void exact_pair_digits(const bpx_code* c, ExactParams* P);

// Coded rows that masks of e erased columns leave (launch heuristics; the
// mask itself is on the device): the mean, and eight quantiles over the masks.
struct RowsRange {
  long long mean, rows[8];
};
RowsRange rows_range(const bpx_code* c, int h);

// Whether BPX_FP32 products of this shape run on the tensor cores (three bf16
// parts per operand, six products) rather than on the CUDA cores.
bool f32_on_tensor_cores(const bpx_code* c, int N, int K, int h);

// The tile that a product takes when its caller names none (gemm_tc.cu).
enum TileKind { kTileBf16 = 0, kTileBf16x3, kTileF32, kTileF16x3 };
int auto_bn(TileKind kind, const RowsRange& range, int N, int K);

// twod: the two-dimensional scheme (products are h x (N / k) blocks, operand
// staging holds the summed A and B operands of the code's factored cells).
WsLayout ws_layout(const bpx_code* code, int M, int N, int K, int h, int precision, bool twod = false);

// Completes a code from its cells (supports ascending) and the column of
// each cell (grouped by ascending column): CSR views, source -> cells,
// sigma, the worst-case overhead, the two-dimensional factoring.  c->n, k,
// b, S and e must be set; col_ptr / heights / projections are derived when
// empty.
void finish_code(bpx_code* c, const std::vector<std::vector<int32_t>>& cells,
                 const std::vector<int32_t>& col_of_cell);

// The schedule's per-cell word holds the cell's unknown-source count in its
// low sched_count_bits (the top one of them marks an erased cell) and the sum
// of its unknown sources' ids + 1 (values 1 .. S) above, modulo the word: when
// one source is left, the sum is its id + 1.  sched_id_bits: the bits of S; a
// 32-bit word (kept in shared memory) fits when both fields do, else the plan
// keeps 64-bit words in global memory.
constexpr int sched_id_bits(int S) {
  int b = 0;
  while (b < 31 && (S >> b) != 0) ++b;
  return b;
}
constexpr bool sched_packable32(int S, int sigma) {
  const int b = sched_id_bits(S);
  return b <= 30 && sigma < (1 << (31 - b));
}

constexpr int sched_count_bits(int sigma) { return sched_id_bits(sigma) + 1; }

// Fills the code's schedule tables (word0, affine).
void build_schedule_tables(bpx_code* c);

// Fills live_cells.
void count_live_cells(bpx_code* c);

// Factors every cell for the two-dimensional scheme (fills the t2_* / a2_* /
// b2_* arrays of the code).
void build_terms_2d(bpx_code* c);

constexpr int32_t kWsMagic = 0x42505831;  // "BPX1"

// Graph header layout (int32 words at g_hdr)
enum { HDR_MAGIC = 0, HDR_N, HDR_S, HDR_CELLS, HDR_EDGES, HDR_SIGMA, HDR_LEN = 16 };

// Plan counters at p_ctr (int32 words)
enum {
  CTR_NSURV = 0,  // surviving cells
  CTR_NWAVES,     // rounds
  CTR_NREC,       // recovered sources
  CTR_PLAN,       // kPlanReady once a whole plan is in place (zeroed by bpx_workspace_init)
  // FP32 on the tensor cores (cleared by every call's products): an operand
  // holds an element that the parts cannot; the float bits of the largest
  // magnitude of the coded rows and of B (kF32Plain and below: not noted)
  CTR_F32_SIMT,
  CTR_F32_AMAX,
  CTR_F32_BMAX,
  CTR_LEN = 16
};
constexpr int32_t kPlanReady = 0x504C414E;  // "PLAN"
constexpr int kF32Words = CTR_F32_BMAX - CTR_F32_SIMT + 1;
constexpr float kF32Plain = 4294967296.f;  // 2^32

}  // namespace bpx

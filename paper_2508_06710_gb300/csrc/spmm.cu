// SpMM over k interleaved right-hand sides (Sec. 2, Eq. (1), Algorithm 1), for CSR and
// sliced-ELL operators, plus the extruded-plane form (Sec. 2, repeated geometries):
//
//   Y[i, j] = c[j] * sum_p val[p] * X[idx[p], j]
//   extruded: Y[i, z] = c[z] * ( dz * sum_p val[p] X[idx[p], z] + w_i (X[i, z-1] - 2 X[i, z] + X[i, z+1]) )
//
// Each matrix coefficient and column index is read from HBM once and used for all k
// columns.  Threads are laid out as (row, chunk of VEC columns, lane within row): the KP
// chunks of a row sit in adjacent lanes, so the X rows they gather (k * sizeof(T) bytes)
// are read with coalesced 16-byte loads, and Y is written the same way.  The block's
// contiguous range of nonzeros (column indices and values) is staged in shared memory with
// coalesced loads before use, and broadcast from there to the KP chunk lanes of each row.
// With LPR > 1 several lanes split one row's nonzeros and are reduced with warp shuffles.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "spmm_impl.cuh"

namespace rb {

rb_status spmm_launch_f64(const rb_op* op, const SpmmSched& sc, const void* X, int64_t ldx, void* Y, int64_t ldy,
                          int k, const double* cs, cudaStream_t s);
rb_status spmm_launch_f32(const rb_op* op, const SpmmSched& sc, const void* X, int64_t ldx, void* Y, int64_t ldy,
                          int k, const double* cs, cudaStream_t s);
rb_status stencil_spmm_launch(const rb_op* op, const SpmmSched& sc, const void* X, int64_t ldx, void* Y, int64_t ldy,
                              int k, const double* cs, cudaStream_t s);
rb_status spmm_launch_df(const rb_op* op, const SpmmSched& sc, const void* X, int64_t ldx, void* Y, int64_t ldy,
                         int k, const double* cs, cudaStream_t s);

namespace {

bool sched_valid(const rb_op* op, const SpmmSched& sc, int k, int64_t ldx, int64_t ldy, const void* X,
                 const void* Y) {
  const int eb = op->dtype == RB_F32 ? 4 : 8;
  if (sc.vec < 1 || sc.vec > 4 || !vec_ok(eb, sc.vec, k, ldx, ldy, X, Y)) return false;
  if (sc.kp != next_pow2(k / sc.vec) || sc.kp > 32) return false;
  if (sc.kp * sc.lpr > 32) return false;
  if ((op->format == RB_SELL || op->format == RB_STENCIL) && (sc.lpr != 1 || sc.stage)) return false;
  if (sc.stage == 2 && sc.lpr != 1) return false;
  if (op->dtype == RB_DF64 && sc.stage) return false;  // double-float: the direct kernel only
  if (op->ext_nz > 0 && sc.vec == 3) return false;  // the spanwise epilogue takes widths dividing Nz only
  if (op->ext_nz > 0 && (op->ext_nz % sc.vec)) return false;
  return true;
}

// Widths worth trying for k columns, best first: one thread per row for k <= 4 (3-wide
// scalar loads for k = 3), else the widest aligned vector.
std::vector<int> vec_candidates(int eb, int k) {
  std::vector<int> v;
  if (k == 3 || (k % 3 == 0 && k <= 96)) v.push_back(3);
  for (int w = 4; w >= 1; w >>= 1)
    if (k % w == 0 && !(eb == 8 && w == 4 && k > 4)) v.push_back(w);
  return v;
}

}  // namespace

// The schedule of a call that nobody tuned.  Width: 16-byte vectors with one thread per row, then
// three columns, then the widest aligned vector.  The other choices by measurement (us; channel
// 192 x 128 x 96 Laplacian L, gradient G and divergence, 150^3 13- and 27-point operators 13p and 27p,
// the extruded mesh):
//   long rows (12 entries on).  A row's sum has up to eight parts, fewer with more columns: eight lanes
//     split the row while each still has a few chunks.  Where the rows are of like length, 12 to 40
//     entries and enough of them (even_long_rows, rows_by_chains), the parts are chains of one lane: the
//     same sums without the shuffles (eight lanes took 13p FP64 k = 1, 3 375 and 935, 27p 482 and 1236).
//     Rows of uneven length keep the lanes, and so do few rows (24^3: too few for one lane each to hide
//     its gathers, 27p FP32 k = 3 3.4 and in the ring 5.2).
//   the chains in the TMA ring.  FP32, whose loads matter most, always, but for rows below 20 entries with
//     more columns than a row has parts (27p k = 1, 3, 4, 8 136, 146, 150, 185 and direct 195, 221, 222, 287;
//     13p k = 1, 3, 8, 12 78, 83, 117, 199 and direct 88, 107, 139, 214).  FP64 is bound by its pipe: the
//     ring for one column and 27p k = 2 in halves (13p k = 1 113 and direct 135; 27p 248 and 269, k = 2 408
//     and 437), direct otherwise (13p k = 2, 3 195, 281 and in the ring 199, 305; 27p k = 3, 4 619, 680 and
//     640, 831), but for 27p k = 3 below 100,000 rows (34^3 13.0 in the ring, direct 17.5).
//   grid, direct kernels.  FP64 with two columns or more: one block per row block, not a resident
//     wave (L k = 3 91 and 97, k = 8 226 and 248, extruded k = 64 150 and 157; 27p k = 4 680 and 738); one
//     column, the gradient's rows of two and eight chains: the wave (G k = 3 86 and 93; 27p k = 3 619 and
//     641).  FP32 and rows split over lanes: the wave.
//   width.  FP64 k = 4, 8, 16, 32 on short rows: four doubles a thread (G k = 4 107 and 115, the
//     divergence k = 8 191 and 224 with the grid), on rows of two up to 16 (G k = 32 879 and 851).
//   the TMA ring on short rows.  FP32, a matrix that does not stay in L2, and little work per entry
//     loaded (rows of two: G k = 3 49 and 58) or many columns, up to 32, that use three quarters of the
//     chunks laid out (L k = 12, 16, 24, 32 82, 87, 170, 160 and 92, 99, 176, 180; but k = 20, 48 178, 395 and
//     170, 327).
// The ring is taken only where every tile fits its stages (no row far above the average).
// (`pipelined` false: a caller with kernels of its own, whose rows are read directly.)
SpmmSched default_sched(const rb_op* op, int k, int64_t ldx, int64_t ldy, const void* X, const void* Y,
                        bool pipelined = true) {
  const int eb = op->dtype == RB_F32 ? 4 : 8;
  const bool f64 = op->dtype == RB_F64, f32 = op->dtype == RB_F32;
  const bool csr = op->format == RB_CSR && op->ext_nz == 0;
  const double len = op->avg_row_len;
  const bool even = op->max_row_len <= 1.25 * len + 1.0;  // every tile within the ring's capacity
  const bool mid = even_long_rows(op);
  const bool many = csr && f32 && k >= 12 && k <= 32 && k % 4 == 0 && 3 * next_pow2(k / 4) <= k && len < 12.0;
  SpmmSched sc;
  sc.lpr = 1;
  sc.stage = 0;
  sc.grid_cap = -1;
  std::vector<int> order;
  if (mid && pipelined && f64 && k == 2 && len >= 20.0) order.push_back(1);
  // (up to 32 columns: beyond, unaligned rows are refused, and four doubles need no alignment)
  if (csr && f64 && k % 4 == 0 && (k & (k - 1)) == 0 && k <= (len < 4.0 ? 16 : 32) && len < 12.0) order.push_back(4);
  if (many) order.push_back(4);
  if (k * eb == 16 || k * eb == 8) order.push_back(k);
  if (k % 3 == 0 && k <= 12) order.push_back(3);
  for (int w = 16 / eb; w >= 1; w >>= 1) order.push_back(w);
  if (eb == 8 && k == 4 && order[0] != 4) order.insert(order.begin(), 2);
  for (int w : order) {
    SpmmSched t = sc;
    t.vec = w;
    if (k % w) continue;
    t.kp = next_pow2(k / w);
    if (!sched_valid(op, t, k, ldx, ldy, X, Y)) continue;
    if (op->format != RB_SELL && len >= 12.0) {
      t.lpr = std::max(1, std::min(8, 32 / t.kp / 4));
      if (mid && len < kEightSums) t.lpr = std::min(t.lpr, 4);
      if (!sched_valid(op, t, k, ldx, ldy, X, Y)) t.lpr = 1;
    }
    if (op->format == RB_CSR && f64 && k >= 2 && len >= 4.0 && (rows_by_chains(op, t.kp) ? t.lpr < 8 : t.lpr == 1)) t.grid_cap = 0;
    const double matrix = (double)op->nnz * (4 + eb) + 4.0 * op->n_rows;
    const bool ring = mid ? (f32 ? t.lpr > 1 || k <= 8 || len >= 20.0 : k == 1 || (len >= 20.0 && (k == 2 || (k == 3 && !rows_by_chains(op, t.kp)))))
                          : csr && f32 && matrix > 100e6 && (len < 4.0 || (many && w == 4)) && op->n_rblk <= 1;
    if (ring && even && pipelined) {
      SpmmSched r = t;
      r.stage = 2;
      r.lpr = 1;
      r.grid_cap = 0;
      if (sched_valid(op, r, k, ldx, ldy, X, Y)) t = r;
    }
    return t;
  }
  sc.vec = 1;
  sc.kp = next_pow2(k);
  return sc;
}

rb_status spmm_launch(const rb_op* op, const SpmmSched& sc, const void* X, int64_t ldx, void* Y, int64_t ldy, int k,
                      const double* cs, cudaStream_t s) {
  if (op->format == RB_STENCIL) return stencil_spmm_launch(op, sc, X, ldx, Y, ldy, k, cs, s);
  if (op->dtype == RB_F64) return spmm_launch_f64(op, sc, X, ldx, Y, ldy, k, cs, s);
  if (op->dtype == RB_DF64) return spmm_launch_df(op, sc, X, ldx, Y, ldy, k, cs, s);
  return spmm_launch_f32(op, sc, X, ldx, Y, ldy, k, cs, s);
}

rb_status spmm_validate(const rb_op* op, const void* X, int64_t ldx, const void* Y, int64_t ldy, int k) {
  RB_REQUIRE(op != nullptr, "spmm: null operator");
  RB_REQUIRE(k >= 1 && k <= RB_MAX_K, "spmm: k = %d outside [1, %d]", k, RB_MAX_K);
  RB_REQUIRE(ldx >= k && ldy >= k, "spmm: leading dimensions (%lld, %lld) smaller than k = %d", (long long)ldx,
             (long long)ldy, k);
  RB_REQUIRE((op->n_cols == 0 || X) && (op->n_rows == 0 || Y), "spmm: null X or Y");
  RB_REQUIRE(op->ext_nz == 0 || k == op->ext_nz, "spmm: extruded operator needs k == extruded_nz (%d), got %d",
             op->ext_nz, k);
  const int eb = op->dtype == RB_F32 ? 4 : 8;
  RB_REQUIRE((uintptr_t)X % eb == 0 && (uintptr_t)Y % eb == 0, "spmm: X or Y not aligned to the element size");
  const SpmmSched sc = default_sched(op, k, ldx, ldy, X, Y);
  if (!sched_valid(op, sc, k, ldx, ldy, X, Y)) {
    set_error("spmm: no schedule for k = %d with these leading dimensions and alignments (k > 32 needs "
              "8- or 16-byte aligned rows)", k);
    return RB_EUNSUPPORTED;
  }
  // X and Y must not overlap (the bytes each spans: its last row ends after k columns)
  const uintptr_t xb = (uintptr_t)X, xe = xb + (uintptr_t)(((int64_t)(op->n_cols - 1) * ldx + k) * eb);
  const uintptr_t yb = (uintptr_t)Y, ye = yb + (uintptr_t)(((int64_t)(op->n_rows - 1) * ldy + k) * eb);
  RB_REQUIRE(op->n_rows == 0 || op->n_cols == 0 || xe <= yb || ye <= xb, "spmm: X and Y overlap");
  return RB_OK;
}

SpmmSched pick_sched(const rb_op* op, int k, int64_t ldx, int64_t ldy, const void* X, const void* Y) {
  auto it = op->tuned.find(k);
  if (it != op->tuned.end() && sched_valid(op, it->second, k, ldx, ldy, X, Y)) return it->second;
  return default_sched(op, k, ldx, ldy, X, Y);
}

// The schedule whose lanes per row the solvers' own products take (they read rows directly).
SpmmSched solver_sched(const rb_op* op, int k, int64_t ldx, int64_t ldy, const void* X, const void* Y) {
  auto it = op->tuned.find(k);
  if (it != op->tuned.end() && sched_valid(op, it->second, k, ldx, ldy, X, Y)) return it->second;
  return default_sched(op, k, ldx, ldy, X, Y, false);
}

std::vector<SpmmSched> tune_candidates(const rb_op* op, int k, int64_t ldx, int64_t ldy, const void* X,
                                       const void* Y) {
  std::vector<SpmmSched> cands;
  const int eb = op->dtype == RB_F32 ? 4 : 8;
  for (int vec : vec_candidates(eb, k)) {
    for (int lpr = 1; lpr <= 8; lpr <<= 1) {
      if (lpr > 1 && op->avg_row_len < 2.0 * lpr) continue;  // lanes would idle on short rows
      for (int stage = 0; stage <= 2; ++stage) {
        for (int gc : {-1, 0}) {
          if (stage && gc != 0) continue;
          SpmmSched sc;
          sc.vec = vec;
          sc.kp = next_pow2(k / vec);
          sc.lpr = lpr;
          sc.stage = stage;
          sc.grid_cap = gc;
          if (!sched_valid(op, sc, k, ldx, ldy, X, Y)) continue;
          if (op->format == RB_SELL && gc != -1) continue;
          cands.push_back(sc);
        }
      }
    }
  }
  return cands;
}

}  // namespace rb

using namespace rb;

extern "C" rb_status rb_spmm(rb_op_t A, const void* X, int64_t ldx, void* Y, int64_t ldy, int32_t k, const double* c,
                             rb_stream_t stream) {
  clear_error();
  RB_TRY(spmm_validate(A, X, ldx, Y, ldy, k));
  if (A->n_rows == 0) return RB_OK;
  const SpmmSched sc = pick_sched(A, k, ldx, ldy, X, Y);
  return spmm_launch(A, sc, X, ldx, Y, ldy, k, c, S(stream));
}

extern "C" rb_status rb_tune_spmm(rb_op_t A, const void* X, int64_t ldx, void* Y, int64_t ldy, int32_t k,
                                  rb_stream_t stream) {
  clear_error();
  RB_TRY(spmm_validate(A, X, ldx, Y, ldy, k));
  if (A->n_rows == 0) return RB_OK;
  cudaStream_t s = S(stream);
  const std::vector<SpmmSched> cands = tune_candidates(A, k, ldx, ldy, X, Y);
  if (cands.empty()) {
    set_error("rb_tune_spmm: no valid schedule for k = %d", k);
    return RB_EUNSUPPORTED;
  }
  cudaEvent_t e0, e1;
  RB_CUDA(cudaEventCreate(&e0));
  RB_CUDA(cudaEventCreate(&e1));
  float best = 1e30f;
  SpmmSched best_sc = cands[0];
  for (const SpmmSched& sc : cands) {
    rb_status st = RB_OK;
    for (int w = 0; w < 2 && st == RB_OK; ++w) st = spmm_launch(A, sc, X, ldx, Y, ldy, k, nullptr, s);
    if (st != RB_OK) continue;
    float times[5];
    for (int r = 0; r < 5; ++r) {
      cudaEventRecord(e0, s);
      spmm_launch(A, sc, X, ldx, Y, ldy, k, nullptr, s);
      cudaEventRecord(e1, s);
      cudaEventSynchronize(e1);
      cudaEventElapsedTime(&times[r], e0, e1);
    }
    std::sort(times, times + 5);
    if (times[2] < best) {
      best = times[2];
      best_sc = sc;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  RB_CUDA(cudaGetLastError());
  A->tuned[k] = best_sc;
  return RB_OK;
}

extern "C" rb_status rb_set_spmm_schedule(rb_op_t A, int32_t k, const rb_spmm_schedule* sched) {
  clear_error();
  RB_REQUIRE(A && sched, "rb_set_spmm_schedule: null argument");
  RB_REQUIRE(k >= 1 && k <= RB_MAX_K, "rb_set_spmm_schedule: k = %d outside [1, %d]", k, RB_MAX_K);
  SpmmSched sc;
  sc.vec = sched->vec;
  sc.lpr = sched->lpr;
  sc.stage = sched->stage;
  sc.grid_cap = sched->grid_cap;
  RB_REQUIRE(sc.vec >= 1 && sc.vec <= 4 && k % sc.vec == 0, "rb_set_spmm_schedule: vec %d does not divide k", sc.vec);
  sc.kp = next_pow2(k / sc.vec);
  RB_REQUIRE(sc.lpr == 1 || sc.lpr == 2 || sc.lpr == 4 || sc.lpr == 8, "rb_set_spmm_schedule: lpr must be 1, 2, 4 or 8");
  RB_REQUIRE(sc.stage >= 0 && sc.stage <= 2, "rb_set_spmm_schedule: stage must be 0, 1 or 2");
  RB_REQUIRE(sc.kp * sc.lpr <= 32, "rb_set_spmm_schedule: (k / vec) * lpr exceeds a warp");
  RB_REQUIRE(!(A->format == RB_SELL && (sc.lpr != 1 || sc.stage)), "rb_set_spmm_schedule: sliced ELL takes lpr 1, stage 0");
  RB_REQUIRE(!(A->format == RB_STENCIL && (sc.lpr != 1 || sc.stage)),
             "rb_set_spmm_schedule: a stencil operator takes lpr 1, stage 0");
  RB_REQUIRE(!(sc.stage == 2 && sc.lpr != 1), "rb_set_spmm_schedule: the TMA pipeline takes lpr 1");
  RB_REQUIRE(!(A->dtype == RB_DF64 && sc.stage), "rb_set_spmm_schedule: a double-float operator takes stage 0");
  RB_REQUIRE(!(A->ext_nz > 0 && (sc.vec == 3 || A->ext_nz % sc.vec)), "rb_set_spmm_schedule: vec must divide Nz");
  A->tuned[k] = sc;
  return RB_OK;
}

extern "C" rb_status rb_get_spmm_schedule(rb_op_t A, int32_t k, int64_t ldx, int64_t ldy, const void* X,
                                          const void* Y, rb_spmm_schedule* sched) {
  clear_error();
  RB_REQUIRE(A && sched, "rb_get_spmm_schedule: null argument");
  RB_REQUIRE(k >= 1 && k <= RB_MAX_K, "rb_get_spmm_schedule: k = %d outside [1, %d]", k, RB_MAX_K);
  const SpmmSched sc = pick_sched(A, k, ldx, ldy, X, Y);
  sched->vec = sc.vec;
  sched->lpr = sc.lpr;
  sched->stage = sc.stage;
  sched->grid_cap = sc.grid_cap;
  return RB_OK;
}

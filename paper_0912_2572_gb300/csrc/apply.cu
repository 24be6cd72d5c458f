// Application of the TSQR orthogonal factor (sm_103a): B <- Q^T B, B <- Q B, and the
// thin Q = Q [I_n; 0] (paper §4, Table 2: Q costs what R costs; Property 1).
//
// The factor set is a list of launches of jobs; each job walks its tiles and each tile
// holds n reflectors v = [1 at pivot row j; scale_j * tail_j] (tsqr_internal.h). Q^T
// applies jobs launch by launch, tiles and reflectors in factorization order; Q applies
// everything in reverse.
//
// B with at most 8 columns runs here, and the thin Q of up to 8 columns in passes of 4, and 9
// to 32 columns against few reflectors (k_apply_tile); other widths go to the tensor-core
// kernel (apply_mma.cu). k_apply_warp: one warp per job; each
// reflector is a dot product over the tile rows, one warp-level transpose-reduce, and an
// update; no block barrier is needed. With 4 columns a job stages 16.6 KB of a 512-row tile,
// so three CTAs of four jobs fit per SM, and the independent jobs of a sub-partition's three
// warps hide one another's reduction and shared-memory latency. k_apply_vec: one column,
// tile pairs per warp.
#include "tsqr_internal.h"
#include "warp_reduce.cuh"

namespace tsqr {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// Runs BODY(r) for r = ra-1 down to 0 (ra <= 32, warp-uniform) through a fall-through
// switch: only the row slots the reflector needs are issued (a predicated-off FP64
// instruction still occupies the FP64 pipe), while r stays a compile-time register index.
#define TSQR_ROW_SLOTS(ra, RM, BODY)                                                        \
  switch ((ra) > (RM) ? (RM) : (ra)) {                                                      \
    case 32: if (RM >= 32) BODY(31)                                                         \
    case 31: if (RM >= 31) BODY(30)                                                         \
    case 30: if (RM >= 30) BODY(29)                                                         \
    case 29: if (RM >= 29) BODY(28)                                                         \
    case 28: if (RM >= 28) BODY(27)                                                         \
    case 27: if (RM >= 27) BODY(26)                                                         \
    case 26: if (RM >= 26) BODY(25)                                                         \
    case 25: if (RM >= 25) BODY(24)                                                         \
    case 24: if (RM >= 24) BODY(23)                                                         \
    case 23: if (RM >= 23) BODY(22)                                                         \
    case 22: if (RM >= 22) BODY(21)                                                         \
    case 21: if (RM >= 21) BODY(20)                                                         \
    case 20: if (RM >= 20) BODY(19)                                                         \
    case 19: if (RM >= 19) BODY(18)                                                         \
    case 18: if (RM >= 18) BODY(17)                                                         \
    case 17: if (RM >= 17) BODY(16)                                                         \
    case 16: if (RM >= 16) BODY(15)                                                         \
    case 15: if (RM >= 15) BODY(14)                                                         \
    case 14: if (RM >= 14) BODY(13)                                                         \
    case 13: if (RM >= 13) BODY(12)                                                         \
    case 12: if (RM >= 12) BODY(11)                                                         \
    case 11: if (RM >= 11) BODY(10)                                                         \
    case 10: if (RM >= 10) BODY(9)                                                          \
    case 9: if (RM >= 9) BODY(8)                                                            \
    case 8: if (RM >= 8) BODY(7)                                                            \
    case 7: if (RM >= 7) BODY(6)                                                            \
    case 6: if (RM >= 6) BODY(5)                                                            \
    case 5: if (RM >= 5) BODY(4)                                                            \
    case 4: if (RM >= 4) BODY(3)                                                            \
    case 3: if (RM >= 3) BODY(2)                                                            \
    case 2: if (RM >= 2) BODY(1)                                                            \
    case 1: BODY(0)                                                                         \
    default: break;                                                                         \
  }

// ------------------------------------------------------------- one warp per job
// One reflector (pivot row j, tail xv over rows [lo, hi), tau, scale) applied to the NA
// columns c0 .. c0 + NA - 1 of the warp's staged tile: dot products, one transpose-
// reduce, the pivot-row update, then the tail update. NA is exact, so no column that the
// reflector leaves unchanged issues an FMA (forming Q: reflector j touches columns >= j).
template <int NA, int RW, typename R>
__device__ __forceinline__ void warp_reflector(R *Bt, R *PR, int ldt, int n, int c0, bool ge, int j, int lo,
                                               int hi, int lane, const R (&xv)[RW], R tau, R sc) {
  constexpr int KP = pow2ceil(NA);
  R part[KP];
#pragma unroll
  for (int a = 0; a < KP; ++a) part[a] = R(0);
  R *Bc = Bt + (size_t)c0 * ldt;
  const int ra = (hi - lo + 31) >> 5;
#define TSQR_WDOT(r)                                                                        \
  {                                                                                         \
    const int i = lo + lane + 32 * (r);                                                     \
    if (i < hi) {                                                                           \
      _Pragma("unroll") for (int a = 0; a < NA; ++a) part[a] = fma(xv[r], Bc[a * ldt + i], part[a]); \
    }                                                                                       \
  }
  TSQR_ROW_SLOTS(ra, RW, TSQR_WDOT)
#undef TSQR_WDOT
  int idx;
  const R tot = treduce32<KP, R>(part, lane, idx);
  R cfv = R(0);
  if ((lane & (32 / KP - 1)) == 0 && idx < NA) {
    const int c = c0 + idx;
    R *pp = ge ? &Bt[c * ldt + j] : &PR[c * n + j];
    const R piv = *pp;
    const R w = fma(sc, tot, piv);
    *pp = fma(-tau, w, piv);
    cfv = tau * sc * w;
  }
  R cf[NA];
#pragma unroll
  for (int a = 0; a < NA; ++a) cf[a] = __shfl_sync(kFull, cfv, treduce32_lane<KP>(a));
  __syncwarp();
#define TSQR_WUPD(r)                                                                        \
  {                                                                                         \
    const int i = lo + lane + 32 * (r);                                                     \
    if (i < hi) {                                                                           \
      _Pragma("unroll") for (int a = 0; a < NA; ++a) Bc[a * ldt + i] = fma(-cf[a], xv[r], Bc[a * ldt + i]); \
    }                                                                                       \
  }
  TSQR_ROW_SLOTS(ra, RW, TSQR_WUPD)
#undef TSQR_WUPD
  __syncwarp();
}

// Lane l handles rows lo + l + 32 r of each reflector's tail (RW slots at most, entered
// through TSQR_ROW_SLOTS so only the needed slots issue); the K columns of B are exact.
template <int K, int RW, typename R>
__global__ void __launch_bounds__(128, 2) k_apply_warp(const ApplyParamsT<R> p, int njobs) {
  extern __shared__ __align__(16) unsigned char smraw[];
  R *sm = reinterpret_cast<R *>(smraw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int jid = blockIdx.x * 4 + warp;
  if (jid >= njobs) return;  // warp-uniform; this kernel uses no block barrier
  const int n = p.n, ldt = p.ldt;
  R *Bt = sm + (size_t)warp * ((size_t)ldt + n) * K;  // tile rows, column-major
  R *PR = Bt + (size_t)ldt * K;                        // pivot rows, PR[c*n + j]
  TSQR_CHECK_OR_SKIP(p.njobs == 0 || p.job0 + jid < p.njobs, p.err)
  const JobDesc job = p.jobs[p.job0 + jid];
  const int64_t pr = job.piv_row;
  auto bcol = [&](int c) -> R * { return p.B + (int64_t)(p.col0 + c) * p.ldb; };
  TSQR_CHECK_OR_SKIP(pr >= 0 && (p.rows == 0 || pr + n <= p.rows) &&
                         (p.ntiles == 0 || job.tile_begin + job.tile_count <= p.ntiles),
                     p.err)

#pragma unroll
  for (int c = 0; c < K; ++c)
    for (int j = lane; j < n; j += 32) PR[c * n + j] = bcol(c)[pr + j];
  __syncwarp();

  const int nt = job.tile_count;
  for (int q = 0; q < nt; ++q) {
    const int tt = p.trans ? q : nt - 1 - q;
    const TileDesc td = p.tiles[job.tile_begin + tt];
    const int ht = td.nrows, kind = td.kind;
    const bool ge = (kind == GEQRT);
    const int64_t r0 = td.row0;
    TSQR_CHECK_OR_SKIP(r0 >= 0 && ht >= 1 && ht <= ldt && (p.rows == 0 || r0 + ht <= p.rows) && td.refl >= 0 &&
                           (p.nrefl == 0 || td.refl + n <= p.nrefl),
                       p.err)
#pragma unroll
    for (int c = 0; c < K; ++c) {
      const R *src = bcol(c) + r0;
      for (int i = lane; i < ht; i += 32)
        Bt[c * ldt + i] = (ge && i < n) ? PR[c * n + i] : (p.formq ? R(0) : src[i]);
    }
    __syncwarp();

    const R *Vt = p.V + r0;
    // the next D reflectors' tails (and tau, scale) are in flight while one is applied:
    // each step is a short dependent chain, so one reflector ahead leaves HBM latency
    // exposed
    constexpr int D = RW <= 8 ? 4 : 2;
    R xb[D][RW], tb[D], sb[D];
    auto load_refl = [&](R(&dst)[RW], R &tau_d, R &scl_d, int s) {
      const int j = p.trans ? s : n - 1 - s;
      int lo, hi;
      refl_rows(kind, j, ht, lo, hi, td.off);
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const int i = lo + lane + 32 * r;
        dst[r] = (i < hi) ? __ldg(Vt + i + (int64_t)j * p.ldv) : R(0);
      }
      tau_d = __ldg(p.tau + td.refl + j);
      scl_d = __ldg(p.scl + td.refl + j);
    };
    // forming Q (reverse order), the reflectors j >= col0 + K change none of the pass's
    // columns: the pass starts after them
    const int s_beg = (p.formq && !p.trans) ? max(0, n - (p.col0 + K)) : 0;
#pragma unroll
    for (int d = 0; d < D; ++d)
      if (s_beg + d < n) load_refl(xb[d], tb[d], sb[d], s_beg + d);
    for (int s0 = s_beg; s0 < n; s0 += D) {
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const int s = s0 + d;
        if (s >= n) break;
        const int j = p.trans ? s : n - 1 - s;
        int lo, hi;
        refl_rows(kind, j, ht, lo, hi, td.off);
        const R(&xv)[RW] = xb[d];
        const R tau = tb[d], sc = sb[d];
        // forming Q, reflector j leaves the pass's columns below j unchanged
        const int c0 = p.formq ? max(0, j - p.col0) : 0;
        switch (K - c0) {
          case 8: if (K >= 8) warp_reflector<(K >= 8 ? 8 : 1), RW, R>(Bt, PR, ldt, n, c0, ge, j, lo, hi, lane, xv, tau, sc); break;
          case 7: if (K >= 7) warp_reflector<(K >= 7 ? 7 : 1), RW, R>(Bt, PR, ldt, n, c0, ge, j, lo, hi, lane, xv, tau, sc); break;
          case 6: if (K >= 6) warp_reflector<(K >= 6 ? 6 : 1), RW, R>(Bt, PR, ldt, n, c0, ge, j, lo, hi, lane, xv, tau, sc); break;
          case 5: if (K >= 5) warp_reflector<(K >= 5 ? 5 : 1), RW, R>(Bt, PR, ldt, n, c0, ge, j, lo, hi, lane, xv, tau, sc); break;
          case 4: if (K >= 4) warp_reflector<(K >= 4 ? 4 : 1), RW, R>(Bt, PR, ldt, n, c0, ge, j, lo, hi, lane, xv, tau, sc); break;
          case 3: if (K >= 3) warp_reflector<(K >= 3 ? 3 : 1), RW, R>(Bt, PR, ldt, n, c0, ge, j, lo, hi, lane, xv, tau, sc); break;
          case 2: if (K >= 2) warp_reflector<(K >= 2 ? 2 : 1), RW, R>(Bt, PR, ldt, n, c0, ge, j, lo, hi, lane, xv, tau, sc); break;
          case 1: warp_reflector<1, RW, R>(Bt, PR, ldt, n, c0, ge, j, lo, hi, lane, xv, tau, sc); break;
          default: break;
        }
        if (s + D < n) load_refl(xb[d], tb[d], sb[d], s + D);
      }
    }
#pragma unroll
    for (int c = 0; c < K; ++c) {
      R *dst = bcol(c) + r0;
      for (int i = lane; i < ht; i += 32) {
        if (ge && i < n)
          PR[c * n + i] = Bt[c * ldt + i];
        else
          dst[i] = Bt[c * ldt + i];
      }
    }
    __syncwarp();
  }
#pragma unroll
  for (int c = 0; c < K; ++c)
    for (int j = lane; j < n; j += 32) bcol(c)[pr + j] = PR[c * n + j];
}

// ------------------------------------------- one column: tile pairs per warp
// Q^T b or Q b for a single column is, per reflector, a dot product over the tile rows, a
// reduction and an update of one vector. With a whole warp on one tile (k_apply_warp) a
// lane holds about five rows of a 144-row tile, and the FP64 pipe spends as much on the
// 32-lane reduction and the scalar step as on the dot product and the update. Here a job's
// tiles are dealt alternately to the two half-warps: half 1 runs the next tile in the
// processing order one reflector step behind half 0. Reflector j of a tile needs only the
// pivot entry PR[j] as the previous tile's reflector j left it (and reflectors j' > j do
// not touch it), so the lag of one step is enough. Each warp instruction then carries two
// reflector applications, each lane holds about ten rows, and a reduction spans 16 lanes.
//
// Half h runs local steps u = 0, 1, ...: tile position q = 2 (u / n) + h, reflector step
// u mod n, at warp step t = u + h. The pivot entries live in two buffers: tile q reads
// buffer q mod 2 and writes the other, so no entry is rewritten in the step that reads it,
// and the final pivot rows are in buffer nt mod 2. A leaf tile (GEQRT) holds the pivot
// rows themselves: applying Q^T (the leaf first) it starts from the input buffer and
// publishes row j after reflector j (later reflectors touch rows > j only); applying Q
// (the leaf last) it takes row j from the input buffer at reflector j (reflectors j' > j,
// which run before, touch rows >= j' only) and writes its rows < n out at the end.

template <int RV>
__global__ void __launch_bounds__(128, 3) k_apply_vec(const ApplyParamsT<double> p, int njobs) {
  // reflector tails loaded ahead per half (fewer for tall tiles, to stay in registers)
  constexpr int kVecD = RV <= 16 ? 3 : 1;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = lane >> 4, hl = lane & 15;
  const int jid = blockIdx.x * 4 + warp;
  if (jid >= njobs) return;  // warp-uniform; this kernel uses no block barrier
  const int n = p.n, ldt = p.ldt;
  double *PR = reinterpret_cast<double *>(smraw) + (size_t)warp * (2 * (size_t)ldt + 2 * n);  // 2 x n
  double *Bt = PR + 2 * n + (size_t)h * ldt;  // this half's tile
  double *B = p.B + (int64_t)p.col0 * p.ldb;
  TSQR_CHECK_OR_SKIP(p.njobs == 0 || p.job0 + jid < p.njobs, p.err)
  const JobDesc job = p.jobs[p.job0 + jid];
  const int64_t pr = job.piv_row;
  const int nt = job.tile_count;
  TSQR_CHECK_OR_SKIP(pr >= 0 && (p.rows == 0 || pr + n <= p.rows) &&
                         (p.ntiles == 0 || job.tile_begin + nt <= p.ntiles),
                     p.err)
#ifdef TSQR_CHECK
  // every tile is checked before the pipeline starts: a check inside it would let one half
  // leave while the other waits for it in a shuffle
  for (int q = 0; q < nt; ++q) {
    const TileDesc tq = p.tiles[job.tile_begin + q];
    TSQR_CHECK_OR_SKIP(tq.row0 >= 0 && tq.nrows >= 1 && tq.nrows <= ldt &&
                           (p.rows == 0 || tq.row0 + tq.nrows <= p.rows) && tq.refl >= 0 &&
                           (p.nrefl == 0 || tq.refl + n <= p.nrefl),
                       p.err)
  }
#endif
  for (int j = lane; j < n; j += 32) PR[j] = B[pr + j];

  const int usteps = ((nt - h + 1) >> 1) * n;                 // this half's local steps
  const int T = max(((nt + 1) >> 1) * n, (nt >> 1) * n + 1);  // warp steps
  auto tile_of = [&](int u) -> TileDesc {
    const int q = 2 * (u / n) + h;
    return p.tiles[job.tile_begin + (p.trans ? q : nt - 1 - q)];
  };
  auto refl_of = [&](int u) -> int { return p.trans ? u % n : n - 1 - u % n; };
  // this lane's rows of the tail of local step u's reflector, its tau, scale, tau * scale
  double xb[kVecD][RV], tb[kVecD], sb[kVecD], cb[kVecD];
  auto load = [&](int d, int u) {
#pragma unroll
    for (int r = 0; r < RV; ++r) xb[d][r] = 0.0;
    tb[d] = sb[d] = cb[d] = 0.0;
    if (u < 0 || u >= usteps) return;
    const TileDesc tq = tile_of(u);
    const int j = refl_of(u);
    int lo, hi;
    refl_rows(tq.kind, j, tq.nrows, lo, hi, tq.off);
    const double *v = p.V + tq.row0 + (int64_t)j * p.ldv;
#pragma unroll
    for (int r = 0; r < RV; ++r) {
      const int i = lo + hl + 16 * r;
      if (i < hi) xb[d][r] = __ldg(v + i);
    }
    tb[d] = __ldg(p.tau + tq.refl + j);
    sb[d] = __ldg(p.scl + tq.refl + j);
    cb[d] = tb[d] * sb[d];
  };
#pragma unroll
  for (int d = 0; d < kVecD; ++d) load(d, d - h);

  TileDesc td{};  // the half's current tile
  double *Pin = PR, *Pout = PR + n;  // its pivot buffers (tile q: in = q mod 2)
  // A tile leaves shared memory at the warp step after its last reflector (the rows of
  // that update belong to other lanes); the leaf's pivot rows go back to PR (applying Q)
  // or were published row by row (applying Q^T).
  auto store_prev = [&](int u) {
    const int up = u - 1;
    if (up < 0 || up >= usteps || up % n != n - 1) return;
    const bool ge = (td.kind == GEQRT);
    for (int i = hl; i < td.nrows; i += 16) {
      if (ge && i < n) {
        if (!p.trans) Pout[i] = Bt[i];
      } else {
        B[td.row0 + i] = Bt[i];
      }
    }
  };
  for (int t0 = 0; t0 < T; t0 += kVecD) {
#pragma unroll
    for (int d = 0; d < kVecD; ++d) {
      const int t = t0 + d;
      if (t >= T) break;  // warp-uniform
      const int u = t - h;
      const bool act = (u >= 0 && u < usteps);
      __syncwarp();  // the previous step's updates and head entries are visible
      store_prev(u);
      if (act && u % n == 0) {  // stage the next tile
        td = tile_of(u);
        const int q = 2 * (u / n) + h;
        Pin = PR + (q & 1) * n;
        Pout = PR + ((q + 1) & 1) * n;
        const bool ge = (td.kind == GEQRT);
        for (int i = hl; i < td.nrows; i += 16) {
          if (ge && i < n) {
            if (p.trans) Bt[i] = Pin[i];
          } else {
            Bt[i] = B[td.row0 + i];
          }
        }
      }
      __syncwarp();
      const int j = refl_of(act ? u : 0);
      int lo = 0, hi = 0;
      if (act) refl_rows(td.kind, j, td.nrows, lo, hi, td.off);
      const int rh = (hi - lo + 15) >> 4;
      const int ra = max(rh, __shfl_xor_sync(kFull, rh, 16));
      const double(&xv)[RV] = xb[d];
      double acc = 0.0;
#define TSQR_VDOT(r)                                                                         \
  {                                                                                          \
    const int i = lo + hl + 16 * (r);                                                        \
    if (i < hi) acc = fma(xv[r], Bt[i], acc);                                                \
  }
      TSQR_ROW_SLOTS(ra, RV, TSQR_VDOT)
#undef TSQR_VDOT
#pragma unroll
      for (int m = 8; m >= 1; m >>= 1) acc += __shfl_xor_sync(kFull, acc, m);
      if (act) {
        // v = [1; scale * tail]: w = v^T b, the head entry becomes piv - tau w and the tail
        // rows take b_i - (tau scale w) x_i
        const bool ge = (td.kind == GEQRT);
        const double piv = (ge && p.trans) ? Bt[j] : Pin[j];
        const double w = fma(sb[d], acc, piv);
        const double cf = cb[d] * w;
#define TSQR_VUPD(r)                                                                         \
  {                                                                                          \
    const int i = lo + hl + 16 * (r);                                                        \
    if (i < hi) Bt[i] = fma(-cf, xv[r], Bt[i]);                                              \
  }
        TSQR_ROW_SLOTS(ra, RV, TSQR_VUPD)
#undef TSQR_VUPD
        if (hl == 0) {
          const double np = fma(-tb[d], w, piv);
          if (ge && !p.trans)
            Bt[j] = np;  // later reflectors j' < j update row j as a tail row
          else
            Pout[j] = np;
        }
      }
      load(d, u + kVecD);
    }
  }
  __syncwarp();
  store_prev(T - h);
  __syncwarp();
  const double *Pf = PR + (nt & 1) * n;
  for (int j = lane; j < n; j += 32) B[pr + j] = Pf[j];
}

// ------------------------------------------- 9..32 columns, few reflectors: a CTA per job
// With few reflectors per tile the tensor-core kernel is bound by what it does once per tile
// and panel (digits of V and of the tile, eight of its warps on two column groups); here the
// tile of up to 32 columns is in shared memory, a half-warp per column of 16, and the next
// reflector's tail and pivot row are loaded one step ahead. The columns rotate over the
// warps with the reflector, so that no SM sub-partition's FP64 pipe takes the extra half-warp
// of an odd count at every step. Q^T B, n rows cleared and Q B of 1,000,000 x 8 with 9 / 16
// columns 1.35 / 1.78 ms (1.99 / 2.02 on the tensor cores, 2 x 1.88 in passes of 8 columns),
// x 12 with 16 2.52 (2.79), x 16 with 9 2.41 (2.75).
constexpr int kTileThreads = 256, kTileCols = 32;

template <int RM, int MINB>
__global__ void __launch_bounds__(kTileThreads, MINB) k_apply_tile(const ApplyParamsT<double> p) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int n = p.n, ldt = p.ldt, kc = p.k;
  double *Bt = reinterpret_cast<double *>(smraw);  // kc columns of ldt rows
  double *PC = Bt + (size_t)kc * ldt;              // dot products, then update coefficients
  double *PV = PC + kTileCols;                     // the pivot row (TSQRT / TTQRT)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, hl = tid & 15;
  TSQR_CHECK_OR_SKIP(p.njobs == 0 || p.job0 + (int)blockIdx.x < p.njobs, p.err)
  const JobDesc job = p.jobs[p.job0 + blockIdx.x];
  const int64_t pr = job.piv_row;
  auto bp = [&](int64_t row, int c) -> double * { return p.B + row + (int64_t)(p.col0 + c) * p.ldb; };
  TSQR_CHECK_OR_SKIP(kc <= kTileCols && pr >= 0 && (p.rows == 0 || pr + n <= p.rows) &&
                         (p.ntiles == 0 || job.tile_begin + job.tile_count <= p.ntiles),
                     p.err)
  const int nt = job.tile_count;
  for (int q = 0; q < nt; ++q) {
    const TileDesc td = p.tiles[job.tile_begin + (p.trans ? q : nt - 1 - q)];
    const int ht = td.nrows, kind = td.kind;
    const bool ge = (kind == GEQRT);
    const int64_t r0 = td.row0;
    TSQR_CHECK_OR_SKIP(r0 >= 0 && ht >= 1 && ht <= ldt && (p.rows == 0 || r0 + ht <= p.rows) && td.refl >= 0 &&
                           (p.nrefl == 0 || td.refl + n <= p.nrefl),
                       p.err)
    const double *Vt = p.V + r0;
    for (int c = warp; c < kc; c += kTileThreads / 32)
      for (int i = lane; i < ht; i += 32) Bt[(size_t)c * ldt + i] = *bp(r0 + i, c);
    const int j0 = p.trans ? 0 : n - 1;
    if (!ge && tid < kc) PV[tid] = __ldcg(bp(pr + j0, tid));
    double xv[RM], xn[RM];
    double tau = 0.0, sc = 0.0, tau_n = 0.0, sc_n = 0.0;  // warp 0's
    if (warp == 0) {
      tau = __ldg(p.tau + td.refl + j0);
      sc = __ldg(p.scl + td.refl + j0);
    }
    auto load = [&](double(&x)[RM], int j) {
      int lo, hi;
      refl_rows(kind, j, ht, lo, hi, td.off);
#pragma unroll
      for (int r = 0; r < RM; ++r) {
        const int i = lo + hl + 16 * r;
        x[r] = (i < hi) ? __ldg(Vt + i + (int64_t)j * p.ldv) : 0.0;
      }
    };
    load(xv, j0);
    __syncthreads();
    for (int s = 0; s < n; ++s) {
      const int j = p.trans ? s : n - 1 - s, jn = p.trans ? j + 1 : j - 1;
      const bool more = s + 1 < n;
      int lo, hi;
      refl_rows(kind, j, ht, lo, hi, td.off);
      double pf = 0.0;
      const bool do_pf = !ge && warp == 1 && more && lane < kc;
      if (more) {
        if (warp == 0) {
          tau_n = __ldg(p.tau + td.refl + jn);
          sc_n = __ldg(p.scl + td.refl + jn);
        }
        load(xn, jn);
        if (do_pf) pf = __ldcg(bp(pr + jn, lane));
      }
      const int rw = (warp + s) & 7;        // this reflector's pair of columns of every 16
      const int ra = (hi - lo + 15) >> 4;
      for (int g = 2 * rw; g < kc; g += 16) {  // warp-uniform
        const int c = g + ((tid >> 4) & 1);
        const double *b = Bt + (size_t)c * ldt;
        double acc = 0.0;
#define TSQR_TDOT(r)                                                                        \
  {                                                                                         \
    const int i = lo + hl + 16 * (r);                                                       \
    if (i < hi && c < kc) acc = fma(xv[r], b[i], acc);                                      \
  }
        TSQR_ROW_SLOTS(ra, RM, TSQR_TDOT)
#undef TSQR_TDOT
#pragma unroll
        for (int m = 8; m >= 1; m >>= 1) acc += __shfl_xor_sync(kFull, acc, m);
        if (hl == 0 && c < kc) PC[c] = acc;
      }
      __syncthreads();
      if (warp == 0 && lane < kc) {
        const double piv = ge ? Bt[(size_t)lane * ldt + j] : PV[lane];
        const double w = fma(sc, PC[lane], piv);
        const double np = fma(-tau, w, piv);
        PC[lane] = tau * sc * w;
        if (ge) Bt[(size_t)lane * ldt + j] = np;
        else *bp(pr + j, lane) = np;
      }
      __syncthreads();
      for (int g = 2 * rw; g < kc; g += 16) {
        const int c = g + ((tid >> 4) & 1);
        double *b = Bt + (size_t)c * ldt;
        const double cf = c < kc ? PC[c] : 0.0;
#define TSQR_TUPD(r)                                                                        \
  {                                                                                         \
    const int i = lo + hl + 16 * (r);                                                       \
    if (i < hi && c < kc) b[i] = fma(-cf, xv[r], b[i]);                                     \
  }
        TSQR_ROW_SLOTS(ra, RM, TSQR_TUPD)
#undef TSQR_TUPD
      }
      if (do_pf) PV[lane] = pf;
#pragma unroll
      for (int r = 0; r < RM; ++r) xv[r] = xn[r];
      tau = tau_n;
      sc = sc_n;
      __syncthreads();
    }
    for (int c = warp; c < kc; c += kTileThreads / 32)
      for (int i = lane; i < ht; i += 32) *bp(r0 + i, c) = Bt[(size_t)c * ldt + i];
    __syncthreads();
  }
}

template <int RM, int MINB>
cudaError_t launch_tile_t(const ApplyParamsT<double> &p, int njobs, cudaStream_t s) {
  const size_t bytes = sizeof(double) * ((size_t)p.k * p.ldt + 2 * kTileCols);
  cudaError_t e = cudaFuncSetAttribute(k_apply_tile<RM, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  k_apply_tile<RM, MINB><<<njobs, kTileThreads, bytes, s>>>(p);
  return cudaGetLastError();
}

template <int K, int RW, typename R>
cudaError_t launch_warp_t(const ApplyParamsT<R> &p, int njobs, cudaStream_t s) {
  const size_t bytes = sizeof(R) * 4 * ((size_t)p.ldt + p.n) * K;
  cudaError_t e = cudaFuncSetAttribute(k_apply_warp<K, RW, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)bytes);
  if (e != cudaSuccess) return e;
  k_apply_warp<K, RW, R><<<(njobs + 3) / 4, 128, bytes, s>>>(p, njobs);
  return cudaGetLastError();
}

template <int K, typename R>
cudaError_t launch_warp_k(const ApplyParamsT<R> &p, int njobs, cudaStream_t s) {
  if (p.ldt <= 256) return launch_warp_t<K, 8, R>(p, njobs, s);
  return launch_warp_t<K, 16, R>(p, njobs, s);
}

template <int RV>
cudaError_t launch_vec_t(const ApplyParamsT<double> &p, int njobs, cudaStream_t s) {
  const size_t bytes = sizeof(double) * 4 * (2 * (size_t)p.ldt + 2 * (size_t)p.n);
  cudaError_t e = cudaFuncSetAttribute(k_apply_vec<RV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  k_apply_vec<RV><<<(njobs + 3) / 4, 128, bytes, s>>>(p, njobs);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_apply_any(const ApplyParamsT<R> &p, int njobs, cudaStream_t s) {
  if (njobs <= 0 || p.k <= 0) return cudaSuccess;
  if (p.ldt > 512) return cudaErrorInvalidValue;
  if (p.k <= 8) {
    switch (p.k) {
      case 1: return launch_warp_k<1, R>(p, njobs, s);
      case 2: return launch_warp_k<2, R>(p, njobs, s);
      case 3: return launch_warp_k<3, R>(p, njobs, s);
      case 4: return launch_warp_k<4, R>(p, njobs, s);
      case 5: return launch_warp_k<5, R>(p, njobs, s);
      case 6: return launch_warp_k<6, R>(p, njobs, s);
      case 7: return launch_warp_k<7, R>(p, njobs, s);
      default: return launch_warp_k<8, R>(p, njobs, s);
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_apply(const ApplyParamsT<double> &p, int njobs, cudaStream_t s, bool tile_pairs) {
  // one column of B over jobs of several tiles: the tile-pair kernel (its one-step lag
  // needs n >= 2; forming Q keeps the warp kernel)
  if (tile_pairs && p.k == 1 && !p.formq && p.n >= 2 && njobs > 0) {
    const int rows_per_lane = (p.ldt + 15) / 16;
    if (rows_per_lane <= 8) return launch_vec_t<8>(p, njobs, s);
    if (rows_per_lane <= 9) return launch_vec_t<9>(p, njobs, s);
    if (rows_per_lane <= 16) return launch_vec_t<16>(p, njobs, s);
    if (rows_per_lane <= 32) return launch_vec_t<32>(p, njobs, s);
    return cudaErrorInvalidValue;
  }
  return launch_apply_any(p, njobs, s);
}

cudaError_t launch_apply_tile(const ApplyParamsT<double> &p, int njobs, cudaStream_t s) {
  if (njobs <= 0 || p.k <= 0) return cudaSuccess;
  if (p.k > kTileCols || p.formq || p.ldt > 512) return cudaErrorInvalidValue;
  if (p.ldt <= 128) return launch_tile_t<8, 2>(p, njobs, s);
  if (p.ldt <= 256) return launch_tile_t<16, 2>(p, njobs, s);
  return launch_tile_t<32, 1>(p, njobs, s);
}

}  // namespace tsqr

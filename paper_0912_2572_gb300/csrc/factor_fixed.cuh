// Device code of the FP64 factorization job in 64-bit fixed point (register tiles).
//
// What bounds the FP64 job of factor_job.cuh is the FP64 pipe: one warp instruction per 64
// cycles and SM sub-partition, the same for one lane as for 32. The integer pipe takes a
// 32 x 32 + 64 multiply-add (IMAD.WIDE) every 2 cycles (measured 2.1-2.6), so a product of
// two 60-bit numbers kept to about 60 bits, three IMAD.WIDE, costs a tenth of one DFMA and
// keeps more bits (with operands that change every time it takes about 4 cycles: 17 for the
// three products and two limb extractions of a dot product entry, 20 for an update). This job
// therefore runs the column steps on integers and uses the FP64
// pipe only to convert the tile (one conversion per entry in, one out).
//
// Numbers. Column c of [R; tile] is held as C = x 2^(60 - E_c) with E_c chosen so that the
// 2-norm of the whole column stays below 2^60 (a reflection preserves it, so no entry can
// overflow later; along a chain E_c only grows, when the tile's norm makes it). An entry is
// exact to 2^-61 of its column's norm, where FP64 rounds to 2^-54 of the entry at every
// update; the normwise error is the smaller one (Householder QR's bounds are normwise, per
// column). The reflector's tail x and its pivot alpha are shifted left together until
// 0.49 < ||[alpha; x]|| / 2^60 < 0.995 (exact: the shift is the only change), so a column
// that cancelled down to few bits still gives a reflector orthogonal to 2^-58. Every few
// columns what is left of a column is shifted up again (rescale below).
//
// Limbs. In the row loops a = ah 2^29 + al (C: al its low 29 bits; x and the coefficient q:
// al signed), elsewhere 2^30; high limbs stay within 32 bits by the norm bounds. A product
// keeps ah bh and ah bl + al bh; the dropped al bl is below 2^-59 of ||x|| ||C||.
//
// Work split. A warp owns a group of GC consecutive columns of the whole tile height: lane
// (lc, lr) holds CPL columns and the row pairs 2 lr + 2 LR r'. A dot product is summed over
// the LR lanes of a column (three to five shuffle stages), every lane of a column computes
// its coefficient, and nothing is broadcast; groups left of the step's column are done and
// only keep the barrier. Wider splits (all columns on every warp, a few rows per lane) spent
// two thirds of their instructions on reductions and needed an unrolled copy of the step
// per count of active columns, more than the instruction cache holds. One block barrier per
// step: the owner of column j+1 updates its group, publishes reflector j+1 (tail limbs and
// scalars, double-buffered by step parity), and the barrier makes it visible. Group g sits
// on warp g or 11 - g, so each SM sub-partition holds an early and a late group.
//
// Measured on GB300 (chain launches, against the FP64 job): 4,194,304 x 64 in 144-row tiles
// 37.0 -> 22.1 ms (18.9 without the rescaling and the unbiased scalars, with a 4 to 50 times
// larger error of least-squares solutions at condition number 1e4), 16M x 16 9.6 -> 6.7; a
// tree level of one 64-column node 162 -> 100 us. A step of a 144 x 64 tile takes 5,250 cycles
// on one CTA and 6,850 on two: the owner's dot products 1,800, coefficients 570, update 1,700,
// next reflector 2,000.
#pragma once
#include <cstdint>

#include "factor_job.cuh"
#include "fixed_point.cuh"

namespace tsqr {
namespace {

#ifdef TSQR_CHECK
#define TSQR_CHECK_OR_SKIP_FX(cond, err, ret) \
  if (!(cond)) {                              \
    if ((err) != nullptr) atomicOr((err), 2); \
    return (ret);                             \
  }
#else
#define TSQR_CHECK_OR_SKIP_FX(cond, err, ret)
#endif

// The scalars of reflector [alpha; x] from the raw column integers: alpha and T = alpha^2 +
// ||x||^2 > 0. sh: the final shift of alpha and x;
//   P = ||[alpha; x]|| 2^sh, D = |alpha| 2^sh + P, y = 2^119 / P, rD = 2^119 / D,
//   tq = 2^59 (1 + |alpha| / P)
// The reciprocal square root and the reciprocal start from the FP32 functions (2^-20 or
// better) and take one step of the third-order iterations
//   y (1 + e/2 + 3/8 e^2), e = 1 - s y^2      and      r (1 + e + e^2), e = 1 - d r
// (the binomial and geometric series cut after e^2: Householder's iterations of order three),
// which leaves e^3 < 2^-60. On the FP64 pipe the same chain is a dozen dependent instructions
// of 64 cycles. A product cut to its upper half is taken at the middle of what it can be
// (2 hi + 1): over a million rows the roundings of the entries average out, and errors of the
// scalars with one sign (2^-59, from products cut down) were what remained of the error.
struct FxRefl {
  long long P, y, rD, tq;
  int sh;
};
__device__ __forceinline__ FxRefl fx_reflector(long long alpha, unsigned __int128 T) {
  FxRefl f;
  const unsigned long long th = (unsigned long long)(T >> 64), tl = (unsigned long long)T;
  const int L = th ? 128 - __clzll((long long)th) : 64 - __clzll((long long)tl);
  int k = L - 62;
  k += k & 1;
  const unsigned long long S = (unsigned long long)(k >= 0 ? T >> k : T << -k);  // [2^60, 2^62)
  // s = S / 2^62 in [1/4, 1]; P = 2^60 sqrt(s), or half of it where sqrt(s) is within 1% of 1
  // (the high limb of a tail entry as large as P must stay below 2^31)
  const int ext = S >= 4519760000000000000ull ? 1 : 0;
  const float sf = __int2float_rn((int)(S >> 32)) * 0x1p-30f;
  const int y0 = __float2int_rn(rsqrtf(sf) * 0x1p29f);
  const unsigned long long y2 = (unsigned long long)fx_mad(y0, y0, 0) << 2;   // 2^60 y0^2
  const long long e = (1ll << 59) - 1 - 2 * (long long)__umul64hi(S, y2);     // 2^59 (1 - s y0^2)
  const int ee = (int)(e >> 13);
  const long long u2e = e + ((3 * (fx_mad(ee, ee, 0) >> 33) + 2) >> 2);       // 2^59 (e + 3/4 e^2)
  const long long Y0 = (long long)y0 << 32;
  const long long y = Y0 + ((__mul64hi(Y0, u2e * (1ll << 22)) + (1ll << 17)) >> 18);  // 2^61 / sqrt(s)
  f.P = 2 * (long long)__umul64hi(S, (unsigned long long)y) + 1;
  if (ext) f.P >>= 1;
  f.sh = 29 - (k >> 1) - ext;
  const long long af = fx_shift(alpha, f.sh);
  const long long aa = af < 0 ? -af : af;
  const long long D = aa + f.P;  // in (2^58.9, 2^61)
  const float df = __int2float_rn((int)(D >> 31)) * 0x1p-30f;
  const int r0 = __float2int_rn(__fdividef(1.0f, df) * 0x1p28f);
  const unsigned long long R0 = (unsigned long long)r0 << 32;
  const long long e2 = (1ll << 59) - 1 - 2 * (long long)__umul64hi((unsigned long long)D << 1, R0);  // 2^59 (1 - d r0)
  const int ee2 = (int)(e2 >> 13);
  const long long u2 = e2 + ((fx_mad(ee2, ee2, 0) + (1ll << 32)) >> 33);
  const long long r = (long long)R0 + ((__mul64hi((long long)R0, u2 * (1ll << 22)) + (1ll << 16)) >> 17);  // 2^121 / D
  f.rD = (r + 2) >> 2;
  f.y = ((y << ext) + 2) >> 2;
  f.tq = (1ll << 59) + (long long)((__umul64hi((unsigned long long)aa << 3, (unsigned long long)f.y << 2) + 1) >> 1);
  return f;
}

// Shared memory of the job: tails of two reflectors, the next pivot column, scalars (two
// steps' limbs; every reflector's for the tile's end), column exponents and norms, R and the
// scales of its row blocks.
__host__ __device__ constexpr int fx_block(int n, int lr) {
  const int rb = n <= 8 ? 1 : n <= 16 ? 2 : n <= 32 ? 4 : 8;
  return rb < lr ? rb : lr;
}
__host__ __device__ constexpr size_t fx_smem_bytes(int n, int nc, int lc, int rpl) {
  const int rb = fx_block(n, 32 / lc), nb = (n + rb - 1) / rb, rows = (32 / lc * rpl + 31) / 32 * 32;
  return (size_t)3 * rows * 8 + 64 + (size_t)n * 24 + (size_t)((nc + 1) & ~1) * 12 +
         ((size_t)n * nc - (size_t)n * (n - 1) / 2) * 8 + (size_t)nb * ((nc + 1) & ~1) * 2 + 16;
}

// One job. Geometry: CPL columns per lane, LC lane columns, RPL (even) rows per lane; the
// warp's group has GC = CPL LC columns, a tile at most LR RPL rows with LR = 32 / LC, and
// nc <= NW GC. Returns the number of tiles done: all of them, or fewer when a tile holds an
// entry the fixed-point form cannot take (not finite, or outside 2^+-900) or is light (above);
// the chain's state is then in global memory, where the FP64 job goes on from.
//
// KEEP = false (the batched kernels, which apply nothing later): only R and the right-hand
// sides' pivot rows are written, to storage of their own (V and B; the tiles come from A and
// Bin). A leaf tile is then a triangle-on-tile step from R = 0, so a tile may be shorter than
// n, and only light tiles end the job early: an entry that is not finite makes the R it would
// have reached NaN.
template <int CPL, int LC, int RPL, int NW, bool KEEP = true, bool COH = false>
__device__ __forceinline__ int run_job_fx(const FactorParamsT<double> &p, const JobDesc job, unsigned char *smraw) {
  constexpr int GC = CPL * LC, LR = 32 / LC, kRpw = (LR * RPL + 31) / 32, kRows = 32 * kRpw;
  static_assert(RPL % 2 == 0 && CPL >= 1 && CPL <= 3 && LR >= 4, "row pairs; one to three columns");
  const int n = p.n, nc = p.nc;
  auto ro = [nc](int i) { return i * nc - i * (i + 1) / 2; };  // R(i, c), c >= i, at Rs[ro(i) + c]
  int2 *xb = reinterpret_cast<int2 *>(smraw);                       // tail limbs, buffer j mod 2
  long long *xw = reinterpret_cast<long long *>(xb + 2 * kRows);    // the next pivot column, raw
  int2 *sb = reinterpret_cast<int2 *>(xw + kRows);                  // limbs of rD, y, tq, buffer j mod 2
  long long *sr = reinterpret_cast<long long *>(sb + 8);            // rD and tq of every reflector
  long long *st = sr + n;
  int *ssh = reinterpret_cast<int *>(st + n);                       // and its shift (n, padded to 2n)
  int *Es = ssh + 2 * n;
  float *nbs = reinterpret_cast<float *>(Es + ((nc + 1) & ~1));
  long long *Rs = reinterpret_cast<long long *>(nbs + ((nc + 1) & ~1));
  const int rb = fx_block(n, LR), rbl = 31 - __clz(rb), nbk = (n + rb - 1) >> rbl, lds = (nc + 1) & ~1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lr = lane % LR, lc = lane / LR;
  // SM sub-partition w mod 4 gets groups from both ends
  const int grp = (warp & 4) ? (warp & ~7) + 11 - (warp & 7) : warp;
  const int cb = GC * grp;          // the group's first column
  int *cbad = reinterpret_cast<int *>(Rs + (size_t)n * nc - (size_t)n * (n - 1) / 2);  // KEEP = false: a
                                      // column's first spoilt row (n: none)
  short *Sc = reinterpret_cast<short *>(cbad + lds);  // R's rows of block b are x 2^(60 - E_c + Sc[b lds + c])
  const int64_t pr = job.piv_row;
  long long v[CPL][RPL];            // column cb + lc + LC t, rows 2 lr + 2 LR (r / 2) + r % 2
  int cur[CPL];                     // and its scale: x 2^(60 - E_c + cur)
  TSQR_CHECK_OR_SKIP_FX(pr >= 0 && (p.rows == 0 || pr + n <= p.rows) && job.tile_begin >= 0 &&
                            (p.ntiles == 0 || job.tile_begin + job.tile_count <= p.ntiles) && nc <= NW * GC,
                        p.err, job.tile_count)
  auto gptr = [&](int64_t row, int c) -> double * {
    return (c < n) ? p.V + row + (int64_t)c * p.ldv : p.B + row + (int64_t)(c - n) * p.ldb;
  };
  auto exp_of = [](int E) { return E == kFxNone ? 0 : E; };  // nothing but zeros so far: any exponent
  // the chain's R to its pivot rows in global memory
  auto write_r = [&]() {
    int first = n;  // the first spoilt column of A
    if constexpr (!KEEP)
      for (int c = n - 1; c >= 0; --c)
        if (cbad[c] < n) first = c;
    for (int c = warp; c < nc; c += NW) {
      double *dst = gptr(pr, c);
      const int lim = c < n ? c + 1 : n;
      const int sh = exp_of(Es[c]) - 60;
      for (int i = lane; i < lim; i += 32) {
        const long long x = Rs[ro(i) + c];
        const int s2 = sh - Sc[(i >> rbl) * lds + c];
        double d;
        if (KEEP || (s2 > -960 && s2 < 900)) d = fx_to_double(x, s2);
        else d = scalbn(__ll2double_rn(x), s2);
        if constexpr (!KEEP)
          if (i >= cbad[c] || (c >= first && i >= first)) d = __longlong_as_double(0x7ff8000000000000ll);
        dst[i] = d;
      }
    }
  };
  auto row_of = [&](int r) { return 2 * lr + 2 * LR * (r >> 1) + (r & 1); };

  for (int tt = 0; tt < job.tile_count; ++tt) {
    const TileDesc td = load_tile<COH>(p.tiles + job.tile_begin + tt);
    const int ht = td.nrows, kind = td.kind, off = td.off;
    const int64_t r0 = td.row0;
    TSQR_CHECK_OR_SKIP_FX(r0 >= 0 && ht >= 1 && ht <= LR * RPL && (p.rows == 0 || r0 + ht <= p.rows) &&
                              kind >= GEQRT && kind <= TTQRT && off >= 0 && off < n && td.refl >= 0 &&
                              (p.nrefl == 0 || td.refl + n <= p.nrefl),
                          p.err, job.tile_count)
    const bool ge = KEEP && kind == GEQRT, tri = (kind == TTQRT);
    const bool zero = tt == 0 && kind == GEQRT;  // nothing in R yet
    const int j0 = tri ? (off >> rbl) << rbl : 0;  // reflectors before a piece's first row are H = I
    // the tile's bits; a child's triangle is zero below its diagonal
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
      const int c = cb + lc + LC * t;
      const bool in = (c < n || !KEEP) && !tri;  // from the inputs (first touch)
      const double *src = !in ? gptr(r0, c) : c < n ? p.A + r0 + (int64_t)c * p.lda : p.Bin + r0 + (int64_t)(c - n) * p.ldbin;
      const int lim = c >= nc ? 0 : (tri && c < n ? min(ht, c + 1 - off) : ht);
      const bool al = (reinterpret_cast<uintptr_t>(src) & 15) == 0;  // row pairs are 16-byte aligned then
#pragma unroll
      for (int r = 0; r < RPL; r += 2) {
        const int i = row_of(r);
        double2 d = make_double2(0.0, 0.0);
        if (al && i + 1 < lim) {
          const double2 *q = reinterpret_cast<const double2 *>(src + i);
          d = in ? ld_input<COH>(q) : __ldcg(q);
        } else {
          if (i < lim) d.x = in ? ld_input<COH>(src + i) : __ldcg(src + i);
          if (i + 1 < lim) d.y = in ? ld_input<COH>(src + i + 1) : __ldcg(src + i + 1);
        }
        v[t][r] = __double_as_longlong(d.x);
        v[t][r + 1] = __double_as_longlong(d.y);
      }
    }
    // exponents and norm bounds of the lane's columns
    // rbad: the first of R's rows that an entry which is not finite spoils in the column
    bool bad = false;
    int En[CPL], rbad[CPL];
    float nbn[CPL];
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
      const int c = cb + lc + LC * t;
      int E = (tt == 0 || c >= nc) ? kFxNone : Es[c];
      float nb = (tt == 0 || c >= nc) ? 0.f : nbs[c];
      rbad[t] = n;
      float sl = 0.f;  // of the last set: the sum of squares in 4^tl
      int tl = 0;
      // one set of entries: their largest exponent field, then their squares relative to it
      auto grow = [&](unsigned mx, auto squares) {
#pragma unroll
        for (int m = LR / 2; m >= 1; m >>= 1) mx = max(mx, __shfl_xor_sync(kFull, mx, m));
        const unsigned e = mx >> 20;
        const bool ok = KEEP ? e >= 1023u - kFxMaxExp && e <= 1023u + kFxMaxExp : e != 0;
        if (KEEP && mx != 0 && !ok) bad = true;
        float s = ok ? squares(e) : 0.f;
#pragma unroll
        for (int m = LR / 2; m >= 1; m >>= 1) s += __shfl_xor_sync(kFull, s, m);
        sl = s;
        tl = (int)e - 1022;
        if (ok) fx_grow(E, nb, tl, s);
      };
      auto habs = [](long long x) { return (unsigned)(x >> 32) & 0x7fffffffu; };
      if (tt == 0 && !zero && !ge) {  // a tree node starts from the first child's triangle
        const double *src = gptr(pr, c);
        const int rl = c >= nc ? 0 : (c < n ? c + 1 : n);
        auto entry = [&](int i) {
          const unsigned h = habs(__double_as_longlong(__ldcg(src + i)));
          return !KEEP && h >= 0x7ff00000u ? 0u : h;
        };
        unsigned mx = 0;
#pragma unroll 4
        for (int i = lr; i < rl; i += LR) {
          const unsigned h = habs(__double_as_longlong(__ldcg(src + i)));
          if (!KEEP && h >= 0x7ff00000u) rbad[t] = min(rbad[t], i);
          else mx = max(mx, h);
        }
        grow(mx, [&](unsigned e) {
          float s = 0.f;
#pragma unroll 4
          for (int i = lr; i < rl; i += LR) s += fx_square_rel(entry(i), e);
          return s;
        });
      }
      unsigned mx = 0;
#pragma unroll
      for (int r = 0; r < RPL; ++r) {
        const unsigned h = habs(v[t][r]);
        if (!KEEP && h >= 0x7ff00000u) {
          rbad[t] = tri ? min(rbad[t], off + row_of(r)) : 0;
          v[t][r] = 0;
        } else {
          mx = max(mx, h);
        }
      }
      grow(mx, [&](unsigned e) {
        float s = 0.f;
#pragma unroll
        for (int r = 0; r < RPL; ++r) s += fx_square_rel(habs(v[t][r]), e);
        return s;
      });
      if constexpr (!KEEP) {
#pragma unroll
        for (int m = LR / 2; m >= 1; m >>= 1) rbad[t] = min(rbad[t], __shfl_xor_sync(kFull, rbad[t], m));
      }
      if (off == 0) {
        const int lim = (E + 1023 - kFxLightBits) * (1 << 20);
        unsigned cnt = 0;  // entries, and light ones
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
          const unsigned h = habs(v[t][r]);
          if (h != 0) cnt += (int)h < lim ? 0x10001u : 1u;
        }
#pragma unroll
        for (int m = LR / 2; m >= 1; m >>= 1) cnt += __shfl_xor_sync(kFull, cnt, m);
        if (E > kFxNone && fx_light(cnt & 0xffff, cnt >> 16, sl, tl - E, tri)) bad = true;
      }
      En[t] = E;
      nbn[t] = nb;
    }
    if (__syncthreads_or(bad)) {
      if (tt > 0) write_r();
      __threadfence();
      __syncthreads();
      return tt;
    }
    if constexpr (!KEEP) {
#pragma unroll
      for (int t = 0; t < CPL; ++t) {
        const int c = cb + lc + LC * t;
        if (lr == 0 && c < nc) cbad[c] = tt > 0 ? min(cbad[c], rbad[t]) : rbad[t];
      }
      __syncthreads();
    }
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
      const int c = cb + lc + LC * t;
      const int E = exp_of(En[t]);
      const int rl = c >= nc ? 0 : (c < n ? c + 1 : n);
      if (tt == 0) {
        // each block of R's rows at its own scale, its largest entry below 2^56
        const double *src = gptr(pr, c);
#pragma unroll 4
        for (int k = 0; k < nbk; ++k) {
          const int i = (k << rbl) + lr;
          const bool in = !ge && lr < rb && i < rl;
          long long x = in && !zero ? __double_as_longlong(__ldcg(src + i)) : 0;
          int e = (int)((x >> 52) & 0x7ff);
          if (!KEEP && e == 2047) x = e = 0;
#pragma unroll
          for (int m = LR / 2; m >= 1; m >>= 1) e = max(e, __shfl_xor_sync(kFull, e, m));
          const int sc = e == 0 ? 0 : min(max(E - (e - 1022) - 4, 0), 400);
          if (in) Rs[ro(i) + c] = fx_of_double(x, 60 - E + sc);
          if (lr == 0 && c < nc) Sc[k * lds + c] = (short)sc;
        }
      } else if (c < nc) {
        const int d = En[t] - Es[c];  // the scales are relative to the exponent
        if (d != 0 && Es[c] != kFxNone)
          for (int k = lr; k < nbk; k += LR) Sc[k * lds + c] = (short)(Sc[k * lds + c] + d);
      }
      __syncwarp();  // the old exponent has been read
      if (c < nc && lr == 0) {
        Es[c] = En[t];
        nbs[c] = nbn[t];
      }
#pragma unroll
      for (int r = 0; r < RPL; ++r) v[t][r] = fx_of_double(v[t][r], 60 - E);
      cur[t] = 0;
    }
    // what is left of the squared norm of a lane's column in the coefficient phase, in 4^E_c:
    // R's finished rows are taken off (an upper bound up to rounding)
    constexpr int kH = LR / 2, kQ = LR / 4;
    // the column of the coefficient phase: one per half of a column's lanes, or per quarter of
    // them (three columns, the last quarter idle)
    const int sel = CPL == 1 ? 0 : CPL == 2 ? (lr & kH) / kH : lr / kQ;
    const bool up = (lr & kH) != 0;
    auto pick = [sel](const auto (&a)[CPL]) {
      if constexpr (CPL == 1) return a[0];
      else if constexpr (CPL == 2) return sel ? a[1] : a[0];
      else return sel == 0 ? a[0] : sel == 1 ? a[1] : a[2];
    };
    const int cs = sel < CPL ? cb + lc + LC * sel : nc;
    float qrem = pick(nbn);
    __syncthreads();

    // Before reflector jn, every rb columns: a column that has become short of its 60 bits by
    // two or more ([R's rows from jn on; tile]) is shifted up to fill them again. Columns
    // lose most of their norm to the leading ones when they are nearly dependent; FP64 entries
    // keep their bits then, and so do these. R's rows of the block take the column's scale.
    // The estimate costs three instructions a step; the rescaling itself is rare on
    // well-conditioned blocks (done at every block it took 15% of the chain's time).
    auto rescale = [&](int jn) {
      const int k = jn >> rbl;
      // qrem 4^cur < 0.05
      const bool mine = qrem < 0.05f * __int_as_float((127 - 2 * pick(cur)) << 23);
      bool stay = !mine || cs < jn || cs >= nc;
#pragma unroll
      for (int t = 0; t < CPL; ++t) {
        const int c = cb + lc + LC * t;
        stay = stay && (c < jn || c >= nc || Sc[k * lds + c] == cur[t]);
      }
      if (__all_sync(kFull, stay)) return;
#pragma unroll
      for (int t = 0; t < CPL; ++t) {
        const int c = cb + lc + LC * t;
        const bool on = c >= jn && c < nc;
        const int rl = c < n ? c + 1 : n;
        if (__any_sync(kFull, on && mine && sel == t)) {
          float q = 0.f;
#pragma unroll
          for (int r = 0; r < RPL; ++r) {
            const float f = (!ge || row_of(r) >= jn) ? fabsf(__int2float_rn((int)(v[t][r] >> 32))) + 1.f : 0.f;
            q = fmaf(f, f, q);
          }
          q *= exp2f((float)(-56 - 2 * cur[t]));
          if (on && !ge)
            for (int i = jn + lr; i < rl; i += LR) {
              const float f = (fabsf(__int2float_rn((int)(Rs[ro(i) + c] >> 32))) + 1.f) *
                              exp2f((float)(-28 - min(Sc[(i >> rbl) * lds + c], 90)));
              q = fmaf(f, f, q);
            }
#pragma unroll
          for (int m = LR / 2; m >= 1; m >>= 1) q += __shfl_xor_sync(kFull, q, m);
          // the largest s with q 4^s < 0.9, at least the present one
          int s2 = cur[t];
          if (on) s2 = max(s2, min((126 - ((__float_as_int(q * 1.1112f) >> 23) & 0xff)) >> 1, 30));
          const int d = s2 - cur[t];
          if (on) {
#pragma unroll
            for (int r = 0; r < RPL; ++r) v[t][r] = (long long)((unsigned long long)v[t][r] << d);
            cur[t] = s2;
            if (sel == t) qrem = q;
          }
        }
        if (on) {
          const int d = cur[t] - Sc[k * lds + c];
          if (!ge && d != 0 && lr < rb && jn + lr < rl) {
            long long *x = Rs + ro(jn + lr) + c;
            *x = fx_shift(*x, d);
          }
        }
        __syncwarp();
        if (on && lr == 0) Sc[k * lds + c] = (short)cur[t];
      }
      __syncwarp();
    };
    // reflector jn, published by the warp whose group holds column jn
    auto publish = [&](int jn) {
      const int b = jn & 1;
#pragma unroll
      for (int t = 0; t < CPL; ++t)
        if (cb + lc + LC * t == jn)
#pragma unroll
          for (int r = 0; r < RPL; r += 2)
            *reinterpret_cast<longlong2 *>(xw + row_of(r)) = make_longlong2(v[t][r], v[t][r + 1]);
      __syncwarp();
      const long long alpha = ge ? xw[jn] : Rs[ro(jn) + jn];
      long long x[kRpw];
      long long hh = 0, hl = 0, ll = 0;
      unsigned any = 0;
#pragma unroll
      for (int r = 0; r < kRpw; ++r) {
        const int i = lane + 32 * r;
        x[r] = ((ge && i <= jn) || i >= LR * RPL) ? 0 : xw[i];
        any |= (unsigned)x[r] | (unsigned)(x[r] >> 32);
        int h, l;
        fx_limbs(x[r], h, l);
        hh = fx_mad(h, h, hh);
        hl = fx_mad(h, l, hl);
        ll = fx_mad(l, l, ll);
      }
      any = __ballot_sync(kFull, any != 0);
      __syncwarp();  // every lane has read alpha before lane 0 replaces it
      if (any == 0) {  // an empty tail: H = I
#pragma unroll
        for (int r = 0; r < kRpw; ++r) xb[b * kRows + lane + 32 * r] = make_int2(0, 0);
        if (lane < 3) sb[4 * b + lane] = make_int2(0, 0);
        if (lane == 0) {
          Rs[ro(jn) + jn] = alpha;
          sr[jn] = 0;
          st[jn] = 0;
          ssh[jn] = 0;
        }
        return;
      }
      if (lane == 0) {
        int h, l;
        fx_limbs(alpha, h, l);
        hh = fx_mad(h, h, hh);
        hl = fx_mad(h, l, hl);
        ll = fx_mad(l, l, ll);
      }
      // the sum of squares over the warp, exact: five integer reductions of 26 bits
      const unsigned __int128 q =
          ((unsigned __int128)(unsigned long long)hh << 60) + (unsigned __int128)((__int128)hl << 31) + (unsigned long long)ll;
      constexpr unsigned kM = (1u << 26) - 1;
      const unsigned s0 = __reduce_add_sync(kFull, (unsigned)q & kM);
      const unsigned s1 = __reduce_add_sync(kFull, (unsigned)(q >> 26) & kM);
      const unsigned s2 = __reduce_add_sync(kFull, (unsigned)(q >> 52) & kM);
      const unsigned s3 = __reduce_add_sync(kFull, (unsigned)(q >> 78) & kM);
      const unsigned s4 = __reduce_add_sync(kFull, (unsigned)(q >> 104));
      const unsigned long long lo = s0 + ((unsigned long long)s1 << 26), hi = s3 + ((unsigned long long)s4 << 26);
      const FxRefl f = fx_reflector(alpha, ((unsigned __int128)hi << 78) + ((unsigned __int128)s2 << 52) + lo);
      if (f.sh >= 0) {
#pragma unroll
        for (int r = 0; r < kRpw; ++r) x[r] = (long long)((unsigned long long)x[r] << f.sh);
      } else {
#pragma unroll
        for (int r = 0; r < kRpw; ++r) x[r] = fx_shift(x[r], f.sh);
      }
#pragma unroll
      for (int r = 0; r < kRpw; ++r) {
        const int h = (int)((x[r] + (1ll << 28)) >> 29);
        const int l = (int)((unsigned)x[r] - ((unsigned)h << 29));
        xb[b * kRows + lane + 32 * r] = make_int2(h, l);
      }
      const bool neg = alpha < 0;
      if (lane == 0) {
        const long long rD = neg ? -f.rD : f.rD, y = neg ? f.y : -f.y;  // y: the update subtracts
        int2 a, c, d;
        fx_limbs(rD, a.x, a.y);
        fx_limbs(y, c.x, c.y);
        fx_limbs(-f.tq, d.x, d.y);
        sb[4 * b] = a;
        sb[4 * b + 1] = c;
        sb[4 * b + 2] = d;
        Rs[ro(jn) + jn] = fx_shift(neg ? f.P : -f.P, -f.sh);
        sr[jn] = rD;
        st[jn] = f.tq;
        ssh[jn] = f.sh;
      }
    };
    if (cb < nc && cb + GC > j0) rescale(j0);
    if (j0 >= cb && j0 < cb + GC) publish(j0);
    __syncthreads();

    const int jend = min(n, cb + GC - 1);  // this group's last step
    for (int j = j0; j < n; ++j) {
      if (j < jend && cb < nc) {
        const int b = j & 1;
        const longlong2 *xs = reinterpret_cast<const longlong2 *>(xb + b * kRows) + lr;
        if (ge) {  // the pivot row of a leaf tile is its own row j
          constexpr int kP = 2 * ((NW * GC + 2 * LR - 1) / (2 * LR)), kPr = RPL < kP ? RPL : kP;  // entries of rows < n
          const int rj = 2 * (j / (2 * LR)) + (j & 1);
          if (lr == (j % (2 * LR)) / 2)
#pragma unroll
            for (int t = 0; t < CPL; ++t) {
              const int c = cb + lc + LC * t;
              long long z = v[t][0];
#pragma unroll
              for (int r = 1; r < kPr; ++r)
                if (r == rj) z = v[t][r];
              if (c > j && c < nc) Rs[ro(j) + c] = z;
            }
          __syncwarp();
        }
        long long g[CPL], m[CPL];
#pragma unroll
        for (int t = 0; t < CPL; ++t) g[t] = 0, m[t] = 1ll << 28;
#pragma unroll
        for (int r = 0; r < RPL; r += 2) {
          const longlong2 q = xs[LR * (r >> 1)];
          const int xh[2] = {(int)q.x, (int)q.y}, xl[2] = {(int)(q.x >> 32), (int)(q.y >> 32)};
#pragma unroll
          for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int t = 0; t < CPL; ++t) {
              const long long w = v[t][r + e];
              const int ch = (int)(w >> 29), cl = (int)((unsigned)w & 0x1fffffffu);
              g[t] = fx_mad(xh[e], ch, g[t]);
              m[t] = fx_mad(xh[e], cl, m[t]);
              m[t] = fx_mad(xl[e], ch, m[t]);
            }
        }
#pragma unroll
        for (int t = 0; t < CPL; ++t) g[t] += m[t] >> 29;  // x C / 2^58
        // sum over the LR lanes of a column; with two columns per lane the first exchange
        // leaves the upper half of the lanes with the second one, with three the first two
        // exchanges leave a quarter of them with each
        long long gt = g[0];
        if constexpr (CPL == 2) {
          const long long send = up ? g[0] : g[1];
          gt = (up ? g[1] : g[0]) + __shfl_xor_sync(kFull, send, kH);
        }
        if constexpr (CPL == 3) {
          const bool odd = (lr & kQ) != 0;
          const long long a = (up ? g[2] : g[0]) + __shfl_xor_sync(kFull, up ? g[0] : g[2], kH);
          const long long b1 = (up ? 0 : g[1]) + __shfl_xor_sync(kFull, up ? g[1] : 0, kH);
          gt = (odd ? b1 : a) + __shfl_xor_sync(kFull, odd ? a : b1, kQ);
        }
#pragma unroll
        for (int s = CPL == 3 ? kQ / 2 : CPL == 2 ? kH / 2 : kH; s >= 1; s >>= 1) gt += __shfl_xor_sync(kFull, gt, s);
        const int c = cs;
        const bool on = c > j && c < nc;
        const int2 rD = sb[4 * b], y = sb[4 * b + 1], tq = sb[4 * b + 2];
        const float qsc = __int_as_float((99 - pick(cur)) << 23);  // 2^(-28 - cur)
        const long long p0 = on ? Rs[ro(j) + c] : 0;
        int h, l;
        fx_limbs((gt + 1) >> 1, h, l);
        const long long w = p0 + fx_mul<60>(h, l, rD);
        fx_limbs(w, h, l);
        const long long nq = fx_mul<61>(h, l, y);
        const long long pk = p0 + fx_mul<59>(h, l, tq);
        const float fk = __int2float_rn((int)(pk >> 32)) * qsc;
        qrem = fmaf(-fk, fk, qrem);
        h = (int)((nq + (1ll << 28)) >> 29);  // -x's coefficient, / 2^58
        l = (int)((unsigned)nq - ((unsigned)h << 29));
        if (!on) h = l = 0;  // columns up to j are reflectors now
        __syncwarp();        // every lane of a column has read p0
        if (on && (CPL == 3 ? lr % kQ : CPL == 2 ? lr % kH : lr) == 0) Rs[ro(j) + c] = pk;
        int qh[CPL], ql[CPL];
        qh[0] = h;
        ql[0] = l;
        if constexpr (CPL == 2) {
          const int oh = __shfl_xor_sync(kFull, h, kH), ol = __shfl_xor_sync(kFull, l, kH);
          qh[0] = up ? oh : h;
          ql[0] = up ? ol : l;
          qh[1] = up ? h : oh;
          ql[1] = up ? l : ol;
        }
        if constexpr (CPL == 3) {
#pragma unroll
          for (int t = 0; t < CPL; ++t) {
            qh[t] = __shfl_sync(kFull, h, lane - lr + t * kQ);
            ql[t] = __shfl_sync(kFull, l, lane - lr + t * kQ);
          }
        }
#pragma unroll
        for (int r = 0; r < RPL; r += 2) {
          const longlong2 q = xs[LR * (r >> 1)];
          const int xh[2] = {(int)q.x, (int)q.y}, xl[2] = {(int)(q.x >> 32), (int)(q.y >> 32)};
#pragma unroll
          for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int t = 0; t < CPL; ++t) {
              const long long z = fx_mad(xl[e], qh[t], fx_mad(xh[e], ql[t], 1ll << 28));
              v[t][r + e] = fx_mad(xh[e], qh[t], v[t][r + e]) + (long long)(int)(z >> 29);
            }
        }
        if (((j + 1) & (rb - 1)) == 0 && j + 1 < n) rescale(j + 1);
        if (j + 1 < n && j + 1 >= cb && j + 1 < cb + GC) publish(j + 1);
      }
      __syncthreads();
    }

    if (!KEEP) continue;
    // the reflectors' scalars: v = [1; scale x], H = I - tau v v^T, as the apply kernels read
    // them; identities for the rows a piece of a triangle does not reach
    for (int j = tid; j < n; j += 32 * NW) {
      p.tau[td.refl + j] = j < j0 ? 0.0 : fx_to_double(st[j], -59);
      p.scl[td.refl + j] = j < j0 ? 0.0 : fx_to_double(sr[j], ssh[j] + 60 - (exp_of(Es[j]) - Sc[(j >> rbl) * lds + j]) - 119);
    }
    // write the tile back: the leaf tile's reflectors below its diagonal (R goes out at the
    // chain's end), dense tails, or the child's triangle only
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
      const int c = cb + lc + LC * t;
      if (c >= nc) continue;
      double *dst = gptr(r0, c);
      const int lim = tri && c < n ? min(ht, c + 1 - off) : ht;
      const int beg = ge ? (c < n ? c + 1 : n) : 0;
      const int sh = exp_of(Es[c]) - 60 - cur[t];
      const bool al = (reinterpret_cast<uintptr_t>(dst) & 15) == 0;
#pragma unroll
      for (int r = 0; r < RPL; r += 2) {
        const int i = row_of(r);
        const double2 d = make_double2(fx_to_double(v[t][r], sh), fx_to_double(v[t][r + 1], sh));
        if (al && i >= beg && i + 1 < lim) {
          *reinterpret_cast<double2 *>(dst + i) = d;
        } else {
          if (i >= beg && i < lim) dst[i] = d.x;
          if (i + 1 >= beg && i + 1 < lim) dst[i + 1] = d.y;
        }
      }
    }
    __syncthreads();
  }
  write_r();
  __syncthreads();
  return job.tile_count;
}

}  // namespace
}  // namespace tsqr

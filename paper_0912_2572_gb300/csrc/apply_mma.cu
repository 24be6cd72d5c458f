// Application of the TSQR orthogonal factor to blocks of columns on the tensor cores
// (sm_103a): B <- Q^T B, B <- Q B and the thin Q, the same jobs and tiles as the kernels of
// apply.cu, with the reflectors taken eight at a time in compact-WY form,
//   H_j..H_j+7 = I - V T V^T,  C <- C - V (T^T (V^T C))   (T for Q),
// and both products done on 16-bit tensor-core instructions without rounding inside them.
//
// FP64 arithmetic on GB300 is one warp instruction per 64 cycles and SM sub-partition; a
// 16x8x16 half-precision MMA takes 8. A 64-bit fixed-point number is eight base-256 digits
// (signed, so adding 0x80..80 makes them its bytes), a half holds a digit exactly, and an
// FP32 accumulator holds the sum of digit products of equal weight exactly (4 pairs x 256
// rows x 2^14 = 2^24), so the 43 digit pairs of weight 256^6 and up take 43 MMA-shares, 5.4
// cycles per entry and product against 64 (the exact splitting of Ozaki, Ogita, Oishi and
// Rump, 2012). The 21 pairs left out are below 0.05 units of 2^-60 of ||v|| ||c|| a row (24
// units in the worst case of 512 rows, signs alike); T is made in FP64.
//
// A tile whose entries are small beside their column, or a reflector with many entries small
// beside 1, would lose digits at a fixed unit of the column: from there on the job goes through
// FP64 (apply_rest_fp64). Forward, a column that becomes short is shifted up.
//
// A warp holds 8 columns x up to 144 rows of C in registers: lane 4g + t holds column g,
// rows 8 b + 2t and 8 b + 2t + 1. That is at once the B fragment of V^T C (its digits are cut
// out of the registers) and, with columns and rows exchanged, the accumulator fragment of
// the update C^T -= Y^T V^T, so C never passes through shared memory. An 8-column, 8-row
// output would use half of an MMA; instead the two halves of M hold two digits of V (or Y)
// and the two halves of K two digits of Y and V, so 43 pairs take 23 and 14 instructions.
// V's digits (eight planes of rows x 8 reflectors, read by ldmatrix in either orientation)
// are prepared two panels ahead, and T one panel ahead, by four more warps.
//
// Measured on GB300 against the FP64 tile kernel it replaced: thin Q of 4,194,304 x 64
// 36.3 -> 12.0 ms (chains), Q^T B with 64 columns 16.1 ms, thin Q of 8M x 32 20.7 -> 9.4, of
// 16M x 16 9.7 -> 7.2 (8 columns 5.2 -> 7.1: those keep the warp kernel); a tree level of one
// 64-column node 82 -> 50 us. A panel step of a 144 x 64 tile took 17,600 cycles: V^T C
// 5,000 and the update 7,000 (MMA floor 3,300 and 4,000 for the two warps of a sub-partition),
// Y 2,000, conversions of the tile 2,800 (an eighth of them each step). Cutting V and making T
// on the eight main warps and one helper took 24,000. The loop is bound by its code, which does
// not fit the instruction caches (stalls on instruction fetch lead): the checks for small rows
// and short columns cost Q^T B of 1M x 64 with 32 columns 5.6 -> 7.1 ms, and 29 KB less of it in
// cut_v gave 6.3 back (thin Q of 1M x 64 5.6, 6.3, 5.7).
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "fixed_point.cuh"
#include "tsqr_internal.h"

namespace tsqr {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMagic = 0x4B400000;  // the bits of 1.5 2^23: a float there has unit 1

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}
__device__ __forceinline__ void mma16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                      uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// the same on top of constant accumulators (no copies into d first)
__device__ __forceinline__ void mma16_init(float (&d)[4], float c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                           uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c));
}
__device__ __forceinline__ void bar_main(int count) { asm volatile("bar.sync 1, %0;" ::"r"(count) : "memory"); }
constexpr int kHelpers = 4;  // warps that cut V into digits and make T
__device__ __forceinline__ void bar_helpers() { asm volatile("bar.sync 2, %0;" ::"n"(32 * kHelpers) : "memory"); }

// The eight base-256 digits of two numbers as half pairs, d[i] of weight 256^i: bytes of
// x + 0x80..80 placed under the exponent of 1024 (0x6400 | u = 1024 + u), minus 1152.
__device__ __forceinline__ void digits2(long long x0, long long x1, uint32_t (&d)[8]) {
  const unsigned long long u0 = (unsigned long long)x0 + 0x8080808080808080ull;
  const unsigned long long u1 = (unsigned long long)x1 + 0x8080808080808080ull;
  const uint32_t w0[2] = {(uint32_t)u0, (uint32_t)(u0 >> 32)}, w1[2] = {(uint32_t)u1, (uint32_t)(u1 >> 32)};
  const __half2 off = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));  // 1152
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t lo = __byte_perm(w0[h], w1[h], 0x5140), hi = __byte_perm(w0[h], w1[h], 0x7362);
    const uint32_t q[4] = {__byte_perm(lo, 0x64646464u, 0x4140), __byte_perm(lo, 0x64646464u, 0x4342),
                           __byte_perm(hi, 0x64646464u, 0x4140), __byte_perm(hi, 0x64646464u, 0x4342)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __half2 z = __hsub2(*reinterpret_cast<const __half2 *>(&q[i]), off);
      d[4 * h + i] = *reinterpret_cast<const uint32_t *>(&z);
    }
  }
}

// sum_d S_d 256^d / 2^61, d = 6..14, from the accumulators of V^T C: acc[e - 5] holds weight
// e in its first half of rows (entries 0, 1) and e + 1 in its second (2, 3).
__device__ __forceinline__ long long combine_w(const float (&acc)[9][4], int c) {
  int S[9];
#pragma unroll
  for (int d = 6; d <= 14; ++d)
    S[d - 6] = (d <= 13 ? __float2int_rn(acc[d <= 13 ? d - 5 : 0][c]) : 0) + __float2int_rn(acc[d - 6][2 + c]);
  long long w = fx_mad(S[1], 256, (long long)S[0] + (1ll << 12)) >> 13;
  w = fx_mad(S[2], 1 << 3, w);
  w = fx_mad(S[3], 1 << 11, w);
  w = fx_mad(S[4], 1 << 19, w);
  w = fx_mad(S[5], 1 << 27, w);
  const long long top = fx_mad(S[8], 1 << 16, fx_mad(S[7], 1 << 8, (long long)S[6]));
  return w + (long long)((unsigned long long)top << 35);
}

// One block of 16 rows of V^T C: digit planes of V at a lane's address `base` (matrices 0..3
// of a load: plane 2ip rows 0-7, plane 2ip+1 rows 0-7, the same for rows 8-15).
__device__ __forceinline__ uint32_t vt_base(uint32_t planes, uint32_t plane_bytes, int lane) {
  return planes + ((lane >> 3) & 1) * plane_bytes + (uint32_t)(8 * (lane >> 4) + (lane & 7)) * 16u;
}
__device__ __forceinline__ void vt_block(float (&acc)[9][4], int ip, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         const uint32_t (&b0)[8], const uint32_t (&b1)[8]) {
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (2 * ip + j >= 5) mma16(acc[2 * ip + j >= 5 ? 2 * ip + j - 5 : 0], a0, a1, a2, a3, b0[j], b1[j]);
}

__device__ __noinline__ double to_double_any(long long x, int sh) {
  return scalbn(__ll2double_rn(x), sh);
}

// The job from tile q0 (in its order of application) on, from reflector j0 of that tile (mid:
// the tile is under way), in FP64 with a warp per column: the tile in registers, V from global
// memory. For tiles of rows that are small beside their column, or reflectors small beside 1,
// which fixed point would round to a fixed fraction of the column's norm.
__device__ __noinline__ void apply_rest_fp64(const ApplyParamsT<double> p, const JobDesc job, int q0, int j0, bool mid,
                                             int c0, int kc) {
  const int lane = threadIdx.x & 31, n = p.n;
  for (int c = threadIdx.x >> 5; c < kc; c += blockDim.x >> 5) {
    double *Bc = p.B + (int64_t)(c0 + c) * p.ldb, *P = Bc + job.piv_row;
    for (int q = q0; q < job.tile_count; ++q) {
      const TileDesc td = p.tiles[job.tile_begin + (p.trans ? q : job.tile_count - 1 - q)];
      const double *Vt = p.V + td.row0;
      double *Bt = Bc + td.row0;
      // forming Q there is no input but the pivot block, which is a leaf's first n rows
      const bool ge = td.kind == GEQRT, zero = p.formq && !(mid && q == q0);
      double x[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const int i = lane + 32 * r;
        x[r] = i < td.nrows && (!zero || (ge && i < n)) ? __ldcg(Bt + i) : 0.0;
      }
      const int first = q == q0 ? j0 : p.trans ? 0 : n - 1;
      for (int j = first; j >= 0 && j < n; j += p.trans ? 1 : -1) {
        if (p.formq && j > c0 + c) continue;  // reflector j touches columns >= j only
        int lo, hi;
        refl_rows(td.kind, j, td.nrows, lo, hi, td.off);
        const double tau = __ldg(p.tau + td.refl + j), sc = __ldg(p.scl + td.refl + j);
        const double *Vj = Vt + (int64_t)j * p.ldv;
        double y[16], a = 0.0, piv = 0.0;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
          const int i = lane + 32 * r;
          y[r] = i >= lo && i < hi ? __ldg(Vj + i) : 0.0;
          a = fma(y[r], x[r], a);
          if (ge && i == j) piv = x[r];
        }
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) a += __shfl_xor_sync(kFull, a, m);
        if (!ge && lane == (j & 31)) piv = __ldcg(P + j);
        piv = __shfl_sync(kFull, piv, j & 31);
        const double w = fma(sc, a, piv), np = fma(-tau, w, piv), cf = tau * sc * w;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
          x[r] = fma(-cf, y[r], x[r]);
          if (ge && lane + 32 * r == j) x[r] = np;
        }
        if (!ge && lane == (j & 31)) P[j] = np;
      }
#pragma unroll
      for (int r = 0; r < 16; ++r)
        if (lane + 32 * r < td.nrows) Bt[lane + 32 * r] = x[r];
    }
  }
}

// |x| / 2^32, to its bit length
__device__ __forceinline__ unsigned fx_bits(long long x) {
  const int h = (int)(x >> 32);
  return (unsigned)(h ^ (h >> 31));
}

struct MmaParams {
  ApplyParamsT<double> a;
  int rg, cg;  // row groups and column groups of a CTA's warps
};

// Shared memory: three buffers of V's digit planes, the pivot block, partial products, T
// (two), G, column exponents and norms, exchange of the row groups' norms, counts and lengths,
// flags, V's light entries, the scales of the pivot block's panels.
__host__ __device__ inline size_t mma_smem_bytes(int n, int rg, int cg, int nb) {
  const size_t rows = (size_t)16 * nb * rg, kc = 8 * (size_t)cg, np = (size_t)(n + 7) / 8;
  return 3 * 8 * rows * 16 + np * 8 * (kc + 2) * 8 + (size_t)rg * 8 * (kc + 2) * 8 + 2 * 64 * 8 + 64 * 8 +
         kHelpers * 64 * 8 + kc * 12 + (size_t)rg * kc * 16 + np * kc * 2 + 3 * 8 * 4 + 64;
}

template <int NB>
__global__ void __launch_bounds__(384, 1) k_apply_mma(const MmaParams mp) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const ApplyParamsT<double> &p = mp.a;
  const int RG = mp.rg, CG = mp.cg;
  const int n = p.n, NP = (n + 7) >> 3;
  const int rows = 16 * NB * RG, kc8 = 8 * CG, kcp = kc8 + 2;
  const int MT = 32 * RG * CG;
  const uint32_t plane_bytes = (uint32_t)rows * 16u;
  // smraw: V's digit planes, three buffers of [8][rows][8] halves
  long long *Ps = reinterpret_cast<long long *>(smraw + 3 * 8 * (size_t)plane_bytes);  // [8 NP][kcp]
  long long *Wp = Ps + (size_t)8 * NP * kcp;                                // [RG][8][kcp]
  int2 *Ts = reinterpret_cast<int2 *>(Wp + (size_t)RG * 8 * kcp);           // [2][8][8]
  double *Gs = reinterpret_cast<double *>(Ts + 128);                        // [8][8]
  long long *Gp = reinterpret_cast<long long *>(Gs + 64);                   // [kHelpers][8][8]
  int *Es = reinterpret_cast<int *>(Gp + 64 * kHelpers);                               // [kc8]
  float *nbs = reinterpret_cast<float *>(Es + kc8);
  int *cbad = reinterpret_cast<int *>(nbs + kc8);
  int2 *xn = reinterpret_cast<int2 *>(cbad + kc8);                          // [RG][kc8] exponent, norm
  int2 *xl = xn + (size_t)RG * kc8;                                         // [RG][kc8] counts; bit length
  int *vbad = reinterpret_cast<int *>(xl + (size_t)RG * kc8);               // [4] by tile: first
                                                                            // reflector not finite
  int *vlt = vbad + 4;                                                      // [2] step's V is light
  int *blt = vlt + 2;                                                       // a tile of B is light
  int *vst = vbad + 8;                                                      // [3][8] V's light entries
  short *Sc = reinterpret_cast<short *>(vst + 24);  // [NP][kc8]: panel b of Ps is x 2^(60 - E + Sc)

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const bool helper = warp >= RG * CG;
  const int rg = warp / CG, cw = warp - rg * CG;
  // SM sub-partition w mod 4 gets column groups from both ends (forming the thin Q, the lower
  // groups finish early)
  const int cg = (CG == 8 && (cw & 4)) ? 11 - cw : cw;
  const int c0 = p.col0 + (int)blockIdx.y * kc8;    // first column of this CTA
  const int kc = min(kc8, p.col0 + p.k - c0);       // its columns
  const int col = 8 * cg + g;                       // this lane's column of the CTA
  const bool cin = col < kc;
  TSQR_CHECK_OR_SKIP(p.njobs == 0 || p.job0 + (int)blockIdx.x < p.njobs, p.err)
  const JobDesc job = p.jobs[p.job0 + blockIdx.x];
  const int64_t pr = job.piv_row;
  TSQR_CHECK_OR_SKIP(pr >= 0 && (p.rows == 0 || pr + n <= p.rows) &&
                         (p.ntiles == 0 || job.tile_begin + job.tile_count <= p.ntiles),
                     p.err)
#ifdef TSQR_CHECK
  for (int q = 0; q < job.tile_count; ++q) {
    const TileDesc td = p.tiles[job.tile_begin + q];
    TSQR_CHECK_OR_SKIP(td.row0 >= 0 && td.nrows >= 1 && td.nrows <= rows && (p.rows == 0 || td.row0 + td.nrows <= p.rows) &&
                           td.refl >= 0 && (p.nrefl == 0 || td.refl + n <= p.nrefl),
                       p.err)
  }
#endif
  double *Bc = p.B + (int64_t)(c0 + (cin ? col : 0)) * p.ldb;  // this lane's column
  const int nt = job.tile_count, S = nt * NP;
  auto tile_at = [&](int s) { return p.tiles[job.tile_begin + (p.trans ? s / NP : nt - 1 - s / NP)]; };
  auto panel_at = [&](int s) { return p.trans ? s % NP : NP - 1 - s % NP; };

  // V's digits of step s into buffer s mod 3, a row and two reflectors per thread and turn: v =
  // scale * tail in units of 2^-61, 1 on a leaf tile's diagonal, 0 above it. A thread's
  // entries of kTurns turns are loaded together, a round ahead (six turns in one round were
  // a tenth of the kernel's code, which its loop streams through the instruction cache).
  constexpr int kTurns = 2;
  auto cut_v = [&](int s, int id, int count) {
    const TileDesc td = tile_at(s);
    const int b = panel_at(s);
    unsigned char *buf = smraw + (size_t)(s % 3) * 8 * plane_bytes;
    int light[2] = {0, 0};  // light entries of a reflector
    const int h = id & 3;  // count is a multiple of 4: the same reflectors every turn
    double sc[2], xn2[kTurns][2];
#pragma unroll
    for (int q = 0; q < 2; ++q) sc[q] = 8 * b + 2 * h + q < n ? __ldg(p.scl + td.refl + 8 * b + 2 * h + q) : 0.0;
    auto load = [&](int e0) {
#pragma unroll
      for (int k = 0; k < kTurns; ++k)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int r = (e0 + k * count) >> 2, j = 8 * b + 2 * h + q;
          int lo, hi;
          refl_rows(td.kind, j, td.nrows, lo, hi, td.off);
          xn2[k][q] = (j < n && r >= lo && r < hi) ? __ldg(p.V + td.row0 + r + (int64_t)j * p.ldv) : 0.0;
        }
    };
    load(id);
#pragma unroll 1
    for (int e0 = id; e0 < 4 * rows; e0 += kTurns * count) {
      double x[kTurns][2];
#pragma unroll
      for (int k = 0; k < kTurns; ++k)
#pragma unroll
        for (int q = 0; q < 2; ++q) x[k][q] = xn2[k][q];
      load(e0 + kTurns * count);
#pragma unroll
      for (int k = 0; k < kTurns; ++k) {
        const int r = (e0 + k * count) >> 2;
        if (r >= rows) break;
        long long w[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int j = 8 * b + 2 * h + q;
          const double z = x[k][q] * sc[q];
          w[q] = (td.kind == GEQRT && r == j && j < n) ? 1ll << 61 : fx_of_double(__double_as_longlong(z), 61);
          // |v| <= 1 but for rounding; anything else is not a reflector
          const unsigned hz = (unsigned)__double2hiint(z) & 0x7fffffffu;
          if (hz > (1023u << 20 | 0x80000u)) atomicMin(vbad + ((s / NP) & 3), j);
          if (hz - 1u < ((1023u - kFxLightBits) << 20)) ++light[q];
        }
        uint32_t d[8];
        digits2(w[0], w[1], d);
        unsigned char *dst = buf + (size_t)r * 16 + 4 * h;
#pragma unroll
        for (int i = 0; i < 8; ++i) *reinterpret_cast<uint32_t *>(dst + (size_t)i * plane_bytes) = d[i];
      }
    }
    if (!p.trans) {  // (a warp's lanes take the same turns)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
#pragma unroll
        for (int m = 4; m <= 16; m <<= 1) light[q] += __shfl_xor_sync(kFull, light[q], m);
        if (lane < 4 && light[q] > 0) atomicAdd(vst + (s % 3) * 8 + 2 * lane + q, light[q]);
      }
    }
  };
  // T of step s (the coefficients of W_i in Y_j) from its digit planes. All helper warps:
  // partial products V^T V, every fourth block of 16 rows each; the first: T.
  auto gram = [&](int s) {
    const uint32_t vb = vt_base(smem_addr(smraw) + (uint32_t)(s % 3) * 8 * plane_bytes, plane_bytes, lane);
    float acc[9][4];
#pragma unroll
    for (int e = 0; e < 9; ++e)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[e][c] = 0.f;
    for (int kb = warp - RG * CG; kb < RG * NB; kb += kHelpers) {
      uint32_t b0[8], b1[8];
#pragma unroll
      for (int ip = 0; ip < 4; ++ip) {
        uint32_t q[4];
        ldsm4t(q, vb + 2 * ip * plane_bytes + kb * 256u);
        b0[2 * ip] = q[0];
        b0[2 * ip + 1] = q[1];
        b1[2 * ip] = q[2];
        b1[2 * ip + 1] = q[3];
      }
#pragma unroll
      for (int ip = 0; ip < 4; ++ip)
        vt_block(acc, ip, b0[2 * ip], b0[2 * ip + 1], b1[2 * ip], b1[2 * ip + 1], b0, b1);
    }
    *reinterpret_cast<longlong2 *>(Gp + (warp - RG * CG) * 64 + 8 * g + 2 * t) =
        make_longlong2(combine_w(acc, 0), combine_w(acc, 1));
  };
  auto make_t = [&](int s) {
    const TileDesc td = tile_at(s);
    const int b = panel_at(s);
    const double tl = (lane < 8 && 8 * b + lane < n) ? __ldg(p.tau + td.refl + 8 * b + lane) : 0.0;
    if (!p.trans) {
      // light: a quarter of a reflector's entries, or all of them (its column of Q falls off
      // along the rows as A's does; one to three rows may be small by chance)
      bool light = false;
      if (lane < 8) {
        const int l = vst[(s % 3) * 8 + lane];
        int lo, hi;
        refl_rows(td.kind, 8 * b + lane, td.nrows, lo, hi, td.off);
        light = l > 0 && td.off == 0 && (4 * (l - 4) > hi - lo || (l == hi - lo && (td.kind != TSQRT || l > 3)));
        vst[(s % 3) * 8 + lane] = 0;
      }
      light = __any_sync(kFull, light);
      if (lane == 0) vlt[s & 1] = light;
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int i = lane + 32 * e;
      long long a = 0;
#pragma unroll
      for (int h = 0; h < kHelpers; ++h) a += Gp[64 * h + i];
      Gs[i] = __ll2double_rn(a) * 0x1p-61;
    }
    __syncwarp();
    double T[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {  // T[0:j, j] = -tau_j T[0:j, 0:j] G[0:j, j], lane i has row i
      const double tau = __shfl_sync(kFull, tl, j);
      double a = 0.0;
#pragma unroll
      for (int l = 0; l < j; ++l) a = fma(T[l], Gs[8 * l + j], a);
      T[j] = lane == j ? tau : (lane < j ? -tau * a : 0.0);
    }
    if (lane < 8) {
      int2 *To = Ts + (s & 1) * 64;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (!(fabs(T[j]) <= 4.0)) atomicMin(vbad + ((s / NP) & 3), 8 * b + j);
        int2 q;
        fx_limbs(__double2ll_rn(T[j] * 0x1p59), q.x, q.y);
        To[p.trans ? 8 * lane + j : 8 * j + lane] = q;
      }
    }
    __syncwarp();
  };

  if (tid < 4) vbad[tid] = n;
  if (tid < 3) vlt[tid] = 0;  // and blt
  if (tid < 24) vst[tid] = 0;
  for (int e = tid; e < NP * kc8; e += blockDim.x) Sc[e] = 0;
  for (int c = tid; c < kc8; c += blockDim.x) {
    Es[c] = kFxNone;
    nbs[c] = 0.f;
    cbad[c] = 0;
  }
  for (int e = tid; e < 8 * NP * kcp; e += blockDim.x) Ps[e] = 0;
  __syncthreads();
  if (helper) {
    cut_v(0, tid - MT, 32 * kHelpers);
  } else {
    if (S > 1) cut_v(1, tid, MT);
    // the pivot block, unless the first tile holds it (a leaf, forward)
    if (rg == 0 && !(p.trans && tile_at(0).kind == GEQRT)) {
      unsigned mx = 0;
      for (int i = t; i < n; i += 4) mx = max(mx, cin ? (unsigned)__double2hiint(__ldcg(Bc + pr + i)) & 0x7fffffffu : 0u);
      mx = max(mx, __shfl_xor_sync(kFull, mx, 1));
      mx = max(mx, __shfl_xor_sync(kFull, mx, 2));
      const unsigned e = mx >> 20;
      int E = kFxNone;
      float nb = 0.f, sq = 0.f;
      const bool fin = e != 2047u;
      if (mx != 0 && fin)
        for (int i = t; i < n; i += 4) sq += fx_square_rel((unsigned)__double2hiint(__ldcg(Bc + pr + i)) & 0x7fffffffu, e);
      sq += __shfl_xor_sync(kFull, sq, 1);
      sq += __shfl_xor_sync(kFull, sq, 2);
      if (e != 0 && fin) fx_grow(E, nb, (int)e - 1022, sq);
      if (!p.trans && E != kFxNone)
        for (int i = t; i < n; i += 4) Ps[i * kcp + col] = fx_of_double(__double_as_longlong(__ldcg(Bc + pr + i)), 60 - E);
      // forward, each panel at its own scale, its largest entry below 2^56
      for (int b = 0; p.trans && b < NP; ++b) {
        long long x[2];
        int eb = 0;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int i = 8 * b + t + 4 * q;
          x[q] = E != kFxNone && cin && i < n ? __double_as_longlong(__ldcg(Bc + pr + i)) : 0;
          eb = max(eb, (int)((x[q] >> 52) & 0x7ff));
        }
        eb = max(eb, __shfl_xor_sync(kFull, eb, 1));
        eb = max(eb, __shfl_xor_sync(kFull, eb, 2));
        const int sc = eb == 0 ? 0 : min(max(E - (eb - 1022) - 4, 0), 400);
#pragma unroll
        for (int q = 0; q < 2; ++q)
          if (8 * b + t + 4 * q < n) Ps[(8 * b + t + 4 * q) * kcp + col] = fx_of_double(x[q], 60 - E + sc);
        if (t == 0) Sc[b * kc8 + col] = (short)sc;
      }
      if (t == 0) {
        Es[col] = E;
        nbs[col] = nb;
        if (!fin) cbad[col] = 1;
      }
    }
  }
  __syncthreads();
  if (helper) {
    gram(0);
    bar_helpers();
    if (warp == RG * CG) make_t(0);
  }
  __syncthreads();

  long long v[4 * NB];
  int cur = 0;   // this lane's column of the tile is x 2^(60 - E + cur)
  int ttop = 0;  // bit length of the tile's entries at its start, above 32
  int pdom = -1; // the last panel of the pivot block found not short in this tile
  auto store_tile = [&](const TileDesc &td) {
    const int E = Es[col];
    const int sh = (E == kFxNone ? 0 : E) - 60 - cur, ht = td.nrows;
    const bool bad = cbad[col] != 0, wide = sh < -900 || sh > 900;
    double *dst = Bc + td.row0;
    const bool al = (reinterpret_cast<uintptr_t>(dst) & 15) == 0;
    const int beg = td.kind == GEQRT && p.trans ? n : 0;
#pragma unroll
    for (int q = 0; q < 2 * NB; ++q) {
      const int i = 16 * NB * rg + 2 * t + 8 * q;
      if (beg > 0) {  // the pivot block leaves the leaf tile
        if (i < n) Ps[i * kcp + col] = v[2 * q];
        if (i + 1 < n) Ps[(i + 1) * kcp + col] = v[2 * q + 1];
      }
      double2 d;
      if (wide)
        d = make_double2(to_double_any(v[2 * q], sh), to_double_any(v[2 * q + 1], sh));
      else
        d = make_double2(fx_to_double(v[2 * q], sh), fx_to_double(v[2 * q + 1], sh));
      if (bad) d.x = d.y = __longlong_as_double(0x7ff8000000000000ll);
      if (cin && al && i >= beg && i + 1 < ht) {
        *reinterpret_cast<double2 *>(dst + i) = d;
      } else if (cin) {
        if (i >= beg && i < ht) dst[i] = d.x;
        if (i + 1 >= beg && i + 1 < ht) dst[i + 1] = d.y;
      }
    }
  };
  int s = 0;
  // the rest of the job goes on in FP64 when a step's V is light (from that step on) or a tile of
  // B is (from the tile on); both are the same for the whole CTA
  for (; s < S; ++s) {
    if (vlt[s & 1]) break;
    const TileDesc td = tile_at(s);
    const int pi = s % NP, b = panel_at(s);
    const int ht = td.nrows;
    const bool ge = td.kind == GEQRT;
    const int64_t r0 = td.row0;
    const int rbase = 16 * NB * rg + 2 * t;  // row of v[2 q + e]: rbase + 8 q + e
    if (helper) {
      if (s + 1 < S) {
        gram(s + 1);
        bar_helpers();
        if (warp == RG * CG) make_t(s + 1);
        else if (s + 2 < S) cut_v(s + 2, tid - MT - 32, 32 * (kHelpers - 1));
      }
    } else {
      bool skip = false;
      if (pi == 0) {  // a new tile: its rows, exponents, integers
        cur = 0;
        if (p.formq) {
#pragma unroll
          for (int r = 0; r < 4 * NB; ++r) v[r] = 0;
        } else {
          const double *src = Bc + r0;
          const bool al = (reinterpret_cast<uintptr_t>(src) & 15) == 0;
          const int beg = ge && !p.trans ? n : 0, lim = cin ? ht : 0;
#pragma unroll
          for (int q = 0; q < 2 * NB; ++q) {
            const int i = rbase + 8 * q;
            double2 d = make_double2(0.0, 0.0);
            if (al && i >= beg && i + 1 < lim) {
              d = *reinterpret_cast<const double2 *>(src + i);
            } else {
              if (i >= beg && i < lim) d.x = src[i];
              if (i + 1 >= beg && i + 1 < lim) d.y = src[i + 1];
            }
            v[2 * q] = __double_as_longlong(d.x);
            v[2 * q + 1] = __double_as_longlong(d.y);
          }
          unsigned mx = 0;
#pragma unroll
          for (int r = 0; r < 4 * NB; ++r) mx = max(mx, (unsigned)(v[r] >> 32) & 0x7fffffffu);
          mx = max(mx, __shfl_xor_sync(kFull, mx, 1));
          mx = max(mx, __shfl_xor_sync(kFull, mx, 2));
          const unsigned e = mx >> 20;
          float sq = 0.f;
#pragma unroll
          for (int r = 0; r < 4 * NB; ++r) sq += fx_square_rel((unsigned)(v[r] >> 32) & 0x7fffffffu, e);
          sq += __shfl_xor_sync(kFull, sq, 1);
          sq += __shfl_xor_sync(kFull, sq, 2);
          if (t == 0) xn[rg * kc8 + col] = make_int2((int)e, __float_as_int(sq));
          bar_main(MT);
          int E = Es[col];
          float nb = nbs[col];
          const int E0 = E;
          bool bad = false;
          for (int r = 0; r < RG; ++r) {
            const int2 x = xn[r * kc8 + col];
            if (x.x == 2047) bad = true;
            else if (x.x != 0) fx_grow(E, nb, x.x - 1022, __int_as_float(x.y));
          }
          {
            // light entries are counted in leaves and nodes; under a chain's triangle heavy rows
            // mix with light pivot rows in FP64 too
            if (td.kind != TSQRT) {
              const int lim = (E + 1023 - kFxLightBits) * (1 << 20);
              unsigned cnt = 0;
#pragma unroll
              for (int r = 0; r < 4 * NB; ++r) {
                const unsigned h = (unsigned)(v[r] >> 32) & 0x7fffffffu;
                if (h != 0) cnt += (int)h < lim ? 0x10001u : 1u;
              }
              cnt += __shfl_xor_sync(kFull, cnt, 1);
              cnt += __shfl_xor_sync(kFull, cnt, 2);
              if (t == 0) xl[rg * kc8 + col].x = (int)cnt;
            }
            const int sh = 60 - (E == kFxNone ? 0 : E);
#pragma unroll
            for (int r = 0; r < 4 * NB; ++r) v[r] = fx_of_double(v[r], sh);
          }
          bar_main(MT);  // the old exponents have been read
          int te = -100000;  // the tile's entries are below 2^(E + te)
          for (int r = 0; r < RG; ++r) {
            const int x = xn[r * kc8 + col].x;
            if (x != 0) te = max(te, x - 1022 - E);
          }
          ttop = 28 + te;
          // (a TSQRT tile with an entry above 2^(E - 7) is not light: 512 rows)
          if (te > -100000 && !bad && (td.kind != TSQRT || te < -6)) {
            unsigned cnt = td.kind == TSQRT ? (unsigned)ht : 0;
            float sum = 0.f;
            for (int r = 0; r < RG; ++r) {
              const int2 x = xn[r * kc8 + col];
              if (td.kind != TSQRT) cnt += (unsigned)xl[r * kc8 + col].x;
              if (x.x != 0) sum += __int_as_float(x.y) * exp2f((float)max(2 * (x.x - 1022 - E), -100));
            }
            if (td.off == 0 && fx_light(cnt & 0xffff, cnt >> 16, sum, 0, td.kind == TTQRT)) *blt = 1;
          }
          if (rg == 0) {
            if (E != E0 && E0 != kFxNone) {
              if (p.trans) {  // the panels' scales are relative to the exponent
                for (int b2 = t; b2 < NP; b2 += 4) Sc[b2 * kc8 + col] = (short)min(Sc[b2 * kc8 + col] + E - E0, 30000);
              } else {
                for (int i = t; i < n; i += 4) Ps[i * kcp + col] = fx_shift(Ps[i * kcp + col], E0 - E);
              }
            }
            if (t == 0) {
              Es[col] = E;
              nbs[col] = nb;
              if (bad) cbad[col] = 1;
            }
            __syncwarp();
          }
          bar_main(MT);
          skip = *blt != 0;  // light: the rest in FP64
        }
        if (ge && !p.trans) {  // the pivot block moves into the leaf tile
#pragma unroll
          for (int q = 0; q < 2 * NB; ++q)
#pragma unroll
            for (int e2 = 0; e2 < 2; ++e2) {
              const int i = rbase + 8 * q + e2;
              if (i < n) v[2 * q + e2] = Ps[i * kcp + col];
            }
        }
      }
      const uint32_t pl = smem_addr(smraw) + (uint32_t)(s % 3) * 8 * plane_bytes + (uint32_t)(16 * NB * rg) * 16u;
      // forming the thin Q, reflector j touches columns >= j only
      const bool act = !skip && (!p.formq || (c0 >> 3) + cg >= b);
      // Forward, a column whose remainder (the panels of the pivot block from b on, the tile)
      // has become short is shifted up to fill its bits again, as in the factorization: where
      // R is ill-conditioned the components of Q^T B fall off like R's rows, and R^-1 magnifies
      // what they lost (X of consistent systems of 4M x 64 at condition number 1e4 by Q^T B and the
      // solve 8.9e-15, with it 3.2e-15, in FP64 2.8e-15). Entries of the remainder stay below
      // 2^55, its norm below 2^60.
      if (p.trans && act) {
        int top = ttop;  // the tile's entries are below 2^(32 + top)
        if (pi != 0) {
          unsigned len = 0;
          for (int r = 0; r < RG; ++r) len |= (unsigned)xl[r * kc8 + col].y;
          top = 32 - __clz((int)len);
        } else {
          pdom = -1;
        }
        // the pivot block's panels from b on, the last first: on long chains they are far above the
        // tile, and while one that is not short is to come the column stays as it is
        bool look = top < 21 && b > pdom;
        for (int b2 = ge ? b - 1 : NP - 1; b2 >= b && __any_sync(kFull, look); --b2) {
          int pt = -100000;
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int i = 8 * b2 + t + 4 * q;
            const long long x = i < n ? Ps[i * kcp + col] : 0;
            if (x != 0) pt = max(pt, 32 - __clz((int)fx_bits(x)) + cur - Sc[b2 * kc8 + col]);
          }
          pt = max(pt, __shfl_xor_sync(kFull, pt, 1));
          pt = max(pt, __shfl_xor_sync(kFull, pt, 2));
          top = max(top, pt);
          if (look && pt >= 21) pdom = b2, look = false;
        }
        if (__any_sync(kFull, look)) {
          const int d = look ? min(23 - top, 23) : 0;
          cur += d;
#pragma unroll
          for (int q = 0; q < 2 * NB; ++q)
            if (!ge || 16 * NB * rg + 8 * q >= 8 * b) {
              v[2 * q] = (long long)((unsigned long long)v[2 * q] << d);
              v[2 * q + 1] = (long long)((unsigned long long)v[2 * q + 1] << d);
            }
        }
      }
      if (act) {
        float acc[9][4];
#pragma unroll
        for (int e = 0; e < 9; ++e)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[e][c] = 0.f;
        const uint32_t vb = vt_base(pl, plane_bytes, lane);
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) {
          uint32_t b0[8], b1[8];
          digits2(v[4 * kb], v[4 * kb + 1], b0);
          digits2(v[4 * kb + 2], v[4 * kb + 3], b1);
#pragma unroll
          for (int ip = 0; ip < 4; ++ip) {
            uint32_t a[4];
            ldsm4t(a, vb + 2 * ip * plane_bytes + kb * 256u);
            vt_block(acc, ip, a[0], a[1], a[2], a[3], b0, b1);
          }
        }
        longlong2 w = make_longlong2(combine_w(acc, 0), combine_w(acc, 1));  // reflector g, columns 2t, 2t+1
        const int cu0 = __shfl_sync(kFull, cur, 8 * t), cu1 = __shfl_sync(kFull, cur, 8 * t + 4);  // of columns 2t, 2t+1
        if (rg == 0 && !ge) {
          const longlong2 q = *reinterpret_cast<const longlong2 *>(Ps + (8 * b + g) * kcp + 8 * cg + 2 * t);
          const short *sc = Sc + b * kc8 + 8 * cg + 2 * t;
          const int d0 = cu0 - sc[0], d1 = cu1 - sc[1];
          w.x += q.x;
          w.y += q.y;
          if (__any_sync(kFull, d0 != 0 || d1 != 0)) {
            w.x += fx_shift(q.x, d0) - q.x;
            w.y += fx_shift(q.y, d1) - q.y;
          }
        }
        *reinterpret_cast<longlong2 *>(Wp + (rg * 8 + g) * kcp + 8 * cg + 2 * t) = w;
      }
      if (RG > 1) bar_main(MT);
      else __syncwarp();
      if (act) {
        // Y_j = sum_i T(i, j) W_i for reflectors j = 2t, 2t + 1 of column g
        const int2 *To = Ts + (s & 1) * 64;
        long long h0 = 0, h1 = 0, m0 = 1ll << 28, m1 = 1ll << 28;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          long long w = Wp[i * kcp + col];
          for (int r = 1; r < RG; ++r) w += Wp[(r * 8 + i) * kcp + col];
          int wh, wl;
          fx_limbs(w, wh, wl);
          const int2 ta = To[8 * i + 2 * t], tb = To[8 * i + 2 * t + 1];
          h0 = fx_mad(wh, ta.x, h0);
          m0 = fx_mad(wh, ta.y, fx_mad(wl, ta.x, m0));
          h1 = fx_mad(wh, tb.x, h1);
          m1 = fx_mad(wh, tb.y, fx_mad(wl, tb.x, m1));
        }
        const long long y0 = -((h0 << 1) + (m0 >> 29)), y1 = -((h1 << 1) + (m1 >> 29));
        if (rg == 0 && !ge) {
          long long *P = Ps + (8 * b + 2 * t) * kcp + col;
          const int d = cur - Sc[b * kc8 + col];
          if (__any_sync(kFull, d != 0)) {
            P[0] = fx_shift(P[0], d);
            P[kcp] = fx_shift(P[kcp], d);
            __syncwarp();
            if (t == 0) Sc[b * kc8 + col] = (short)cur;
          }
          P[0] += y0;
          P[kcp] += y1;
        }
        uint32_t yd[8];
        digits2(y0, y1, yd);
        // C += V (-Y): per block of 8 rows, accumulator a of weights 6 + 2a (columns' first copy)
        // and 7 + 2a (second copy); K's halves hold V's digits 2q and 2q + 1
        const uint32_t base = pl + (uint32_t)(lane >> 3) * plane_bytes + (uint32_t)(lane & 7) * 16u;
#pragma unroll
        for (int q = 0; q < 2 * NB; ++q) {
          uint32_t vd[8];
          {
            uint32_t x[4];
            ldsm4(x, base + q * 128u);
            vd[0] = x[0], vd[1] = x[1], vd[2] = x[2], vd[3] = x[3];
            ldsm4(x, base + 4 * plane_bytes + q * 128u);
            vd[4] = x[0], vd[5] = x[1], vd[6] = x[2], vd[7] = x[3];
          }
          float d[5][4];
#pragma unroll
          for (int h = 3; h >= 0; --h)
#pragma unroll
            for (int a = 0; a < 5; ++a) {
              const int w = 6 + 2 * a, i0 = w - 2 * h, i1 = i0 - 1, i2 = i0 + 1, i3 = i0;
              if (i1 > 7 || i2 < 0) continue;
              const uint32_t a0 = i0 >= 0 && i0 <= 7 ? yd[i0 & 7] : 0u, a1 = i2 >= 0 && i2 <= 7 ? yd[i2 & 7] : 0u,
                             a2 = i1 >= 0 && i1 <= 7 ? yd[i1 & 7] : 0u, a3 = i3 >= 0 && i3 <= 7 ? yd[i3 & 7] : 0u;
              if (h == 3) mma16_init(d[a], __int_as_float(kMagic), a0, a1, a2, a3, vd[6], vd[7]);
              else mma16(d[a], a0, a1, a2, a3, vd[2 * h], vd[2 * h + 1]);
            }
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            // sum_w S_w 256^w / 2^61 from the accumulators' bits (2^23 + 2^22 + S_w)
            auto S = [&](int w) { return __float_as_int(d[(w - 6) >> 1][((w & 1) ? 2 : 0) + e]); };
            constexpr int K2 = (int)((unsigned)kMagic * 257u);
            const int t0 = S(6) + (S(7) << 8) - K2, t1 = S(8) + (S(9) << 8) - K2, t2 = S(10) + (S(11) << 8) - K2,
                      t3 = S(12) + (S(13) << 8) - K2, t4 = S(14) - kMagic;
            long long c = v[2 * q + e] + (long long)((t0 + (1 << 12)) >> 13);
            c = fx_mad(t1, 1 << 3, c);
            c = fx_mad(t2, 1 << 19, c);
            c += (long long)((unsigned long long)(unsigned)((t3 << 3) + (t4 << 19)) << 32);
            v[2 * q + e] = c;
          }
        }
        if (p.trans && __any_sync(kFull, b >= pdom)) {
          // of what remains of the column: a sample of its rows, all of them if those are short
          unsigned len = 0;
          auto all = [&](auto step) {
#pragma unroll
            for (int q = 0; q < 2 * NB; q += decltype(step)::value)
              if (!ge || 16 * NB * rg + 8 * q > 8 * b) len |= fx_bits(v[2 * q]) | fx_bits(v[2 * q + 1]);
            len |= __shfl_xor_sync(kFull, len, 1);
            len |= __shfl_xor_sync(kFull, len, 2);
          };
          all(std::integral_constant<int, 4>());
          if (__any_sync(kFull, len < (1u << 20))) all(std::integral_constant<int, 1>());
          if (t == 0) xl[rg * kc8 + col].y = (int)len;
        }
        if (p.trans && ge && rg == 0 && t == 0) Sc[b * kc8 + col] = (short)cur;  // a leaf's rows of the pivot block
      }
      if (pi == NP - 1 && !skip) {  // the tile is done
        // a reflector that is not finite spoils the columns it touches
        if (vbad[(s / NP) & 3] < (p.formq ? min(n, c0 + col + 1) : n) && t == 0 && rg == 0) cbad[col] = 1;
        if (RG > 1) bar_main(MT);
        else __syncwarp();
        store_tile(td);
      }
    }
    __syncthreads();
    if (*blt) break;
  }
  const bool rest = s < S, mid = rest && s % NP != 0;
  if (mid && !helper) store_tile(tile_at(s));
  // the pivot block, unless it has not changed, or a leaf tile holds it (backward, the last one or
  // one under way)
  const bool in_leaf = !p.trans && (!rest || mid) && tile_at(rest ? s : S - 1).kind == GEQRT;
  if (!helper && rg == 0 && cin && s > 0 && !in_leaf) {
    const int E = Es[col];
    const bool bad = cbad[col] != 0;
    for (int i = t; i < n; i += 4)
      Bc[pr + i] = bad ? __longlong_as_double(0x7ff8000000000000ll)
                       : to_double_any(Ps[i * kcp + col], (E == kFxNone ? 0 : E) - 60 - Sc[(i >> 3) * kc8 + col]);
  }
  if (rest) {
    __syncthreads();
    apply_rest_fp64(p, job, s / NP, p.trans ? 0 : min(n, 8 * panel_at(s) + 8) - 1, mid, c0, kc);
  }
}

template <int NB>
cudaError_t launch_mma_t(const MmaParams &mp, int njobs, cudaStream_t s) {
  const size_t bytes = mma_smem_bytes(mp.a.n, mp.rg, mp.cg, NB);
  cudaError_t e = cudaFuncSetAttribute(k_apply_mma<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  const dim3 grid(njobs, (mp.a.k + 8 * mp.cg - 1) / (8 * mp.cg));
  k_apply_mma<NB><<<grid, 32 * (mp.rg * mp.cg + kHelpers), bytes, s>>>(mp);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_apply_mma(const ApplyParamsT<double> &p, int njobs, int rows, int cols_per_cta, cudaStream_t s) {
  if (njobs <= 0 || p.k <= 0) return cudaSuccess;
  MmaParams mp{p, 1, 1};
  int cg = (std::min(p.k, cols_per_cta) + 7) / 8;  // up to 8 warps
  if (rows <= 64) {
    mp.cg = std::min(cg, 8);
    return launch_mma_t<4>(mp, njobs, s);
  }
  if (rows <= 144) {
    mp.cg = std::min(cg, 8);
    return launch_mma_t<9>(mp, njobs, s);
  }
  if (rows <= 288) {
    mp.rg = 2;
    mp.cg = std::min(cg, 4);
    return launch_mma_t<9>(mp, njobs, s);
  }
  if (rows > 512) return cudaErrorInvalidValue;
  mp.rg = 4;
  mp.cg = std::min(cg, 2);
  return launch_mma_t<8>(mp, njobs, s);
}

}  // namespace tsqr

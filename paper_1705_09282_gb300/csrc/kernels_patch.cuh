// Patch solves of the multiplicative Schwarz sweep (eq. MSM of Sec. 5.2) with the patch's
// neighbourhood staged in shared memory, and, for FP64 values, block fixed-point integer
// arithmetic in place of FP64 multiply-adds.
//
// What bounds the sweep on GB300: an FP64 instruction occupies its scheduler for 64 cycles
// whatever its active lanes or its dependences (measured: 64.2 cycles per warp instruction at 1
// to 4 warps per scheduler), a 32 x 32 + 64 bit integer multiply-add 2.3-2.6 cycles.  A patch row
// of degree p = 2 (27 stencil terms, 8 columns of the local inverse) costs some 45 FP64
// instructions, 2900 cycles per warp.  Here every value of a patch's neighbourhood is turned once
// into two integer limbs relative to the largest exponent of its component (u_x, u_y, u_z,
// pressure) there, and every product of a coefficient with a value is three integer multiply-adds:
//   value        v = (hi 2^28 + lo) 2^(e - 57),  |v| < 2^e, |hi| < 2^29, 0 <= |lo| < 2^28
//   coefficient  c = (hi 2^28 + lo) 2^(s - 59),  sum of the box |c| < 2^(s-1),  |lo| <= 2^27
//   sum_j c_j v_j = (HH + MID 2^-28) 2^(e + s - 60),  HH = sum hi hi, MID = sum (hi lo + lo hi)
// The sums are exact in 64-bit integers (|HH| <= 2^59, |MID| < 2^62).  A row's error is bounded per
// box, relative to M = (the component's largest value in the neighbourhood) x (sum of the box's
// |coefficients|), N terms: 2^-56 M for the values' cut, N 2^-58 M each for the coefficients' rounding
// and for the products lo lo left out, 2^-57 M for each rounding of a sum.  That is the bound of N
// FP64 multiply-adds on values of like size; unlike theirs it is relative to M, not to the single
// products: a value 2^k below its component's largest keeps 57 - k bits, a coefficient 2^k below its
// box's sum 59 - k.  Measured over all rows of a level, root mean square relative to the sum of the
// boxes' M, random values, components alike or 1e-4 to 1e-8 of the others: 2D p = 2 4.4e-18, FP64
// multiply-adds 1.5e-17; mapped p = 3 5e-18 and 2e-17; 3D p = 2 6e-18 and 2e-17, p = 3 1.3e-17 and 2e-17.
// (With one exponent for all velocity components, 1.4e-13 and 2e-9 in the rows of a component 1e4 and
// 1e8 times smaller than another.)
// The local residuals stay integers and go through the local inverse the same way, one exponent for
// the velocity rows, one for the pressure rows: the inverse mixes the velocity rows, so a small
// one's low bits are lost in FP64 too.  Emulated on interior and wall patches, components up to 1e8
// apart: the corrections' errors are 0.05 to 0.9 of those of FP64 multiply-adds, the same with an
// exponent for each component.  The correction is rounded once to FP64.
// Values that are not finite make the patch's unknowns NaN; where all of a component is below 2^-959 (biased
// exponent 64) its low bits go, denormals count as 0.
//
// The neighbourhood of the patch at position (a, b): with one set of rows for every patch,
//   UX [2p+1][2p]  u_x at x = a-p .. a+p (outer), y = b-p .. b+p-1
//   UY [2p+1][2p]  u_y at y = b-p .. b+p (outer), x = a-p .. a+p-1
//   PX [2p][2p], PY [2p][2p]  the pressure at a-p .. a+p-1, b-p .. b+p-1, x outer / y outer
// Every row's two boxes (and the third one of mapped domains) are then rectangles with compile-time
// strides inside these arrays, the same for all row kinds, once u_y rows store their coefficients
// with y outer.  Interior (8-DOF) patches use exactly the entries that exist; rows of the larger
// wall patches may reach outside the arrays, only with zero coefficients, into a margin.
//
// What bounded the small levels was a chain of dependent fetches into cold caches (patch list ->
// rows -> records -> values -> inverse) after each launch.  Here all tables are addressed from
// the launch's own indices, fetched first and before the wait for the previous kernel
// (programmatic dependent launch), so a colour's chain is: wait, one fetch of U and F, arithmetic.
// Measured per colour launch (graph replay; row kernels k_mult_colour -> these), FP64: p = 2
// 8^2-64^2 5.0-5.4 -> 1.9-2.1 us, 128^2 5.4 -> 2.4, 256^2 8.1 -> 5.0; p = 3 10-10.5 -> 2.5-2.7,
// 256^2 11.1 -> 7.4; generalized Oseen 512^2 V-cycle 2908 -> 1977 us.  FP32 (same staging, FP32
// arithmetic): p = 2 4.1 -> 1.5-1.8 us, p = 3 7.6 -> 1.3-1.6.
#pragma once
#include <cstdlib>

#include "kernels.cuh"

namespace igamg {
namespace dev {

template <int P>
struct PatchShape {
  static constexpr int Q = P - 1, W = 2 * P;                   // W: extent across
  static constexpr int A1 = 2 * P + 1, B1 = 2 * P, C1 = 2 * Q + 1;  // box extents (long, long, across)
  static constexpr int NA = A1 * C1, NB = B1 * C1, RU = NA + NB + 1;
  static constexpr int NUX = A1 * W, NP = W * W;
  // offsets of the arrays and of the next patch: chosen so that the two patches of a half-warp and
  // their eight rows read from different banks (entries of 8 bytes, offsets mod 16)
  static constexpr int UY = P == 2 ? 22 : 56, PX = P == 2 ? 48 : 112, PY = P == 2 ? 68 : 150, REG = P == 2 ? 88 : 196;
  static constexpr int NLOAD = 2 * NUX + NP;                   // distinct values
  static constexpr int MARGIN = (P + 1) * W;                   // on both sides of a wall patch's arrays
  // a row record: box A, box B from entry RA on (FP64: then the exponents of both), the lambda
  // coefficient at IL (FP64: then its exponent)
  static constexpr int RA = (NA + 3) / 4 * 4, IL = RA + NB + 1, NREC = (IL + 2 + 3) / 4 * 4;
  static constexpr int NEXT = (W * W + 1 + 3) / 4 * 4;         // third box: limbs + exponent
  static constexpr int LW = P == 2 ? 32 : 64;                  // threads per wall patch
  // most velocity and pressure rows of a wall patch; rows of its inverse: MV velocity columns, MP
  // pressure columns (zeros past the patch's own), the FP64 exponents, an odd length (banks)
  static constexpr int MV = P == 2 ? 12 : 24, MP = P == 2 ? 9 : 16, LDW = (MV + MP + 1) | 1;
};

// A staged value or coefficient: two limbs (FP64) or the value itself (FP32).
template <typename T> struct Limb { using type = T; };
template <> struct Limb<double> { using type = int2; };
template <typename T> using limb_t = typename Limb<T>::type;

// Tables of one level in the staged kernels' layout (built once at creation).
template <typename T>
struct PatchTab {
  const limb_t<T>* rec;             // row records, NREC entries each: by class (kind NC^2 + class) or by row
  const limb_t<T>* ext;             // third box by velocity row, NEXT entries each (mapped domains), or null
  const limb_t<T>* inv8;            // interior patches' local inverses: per row 8 entries, then (FP64) exponents
  const limb_t<T>* winv;            // the other patches' inverses
  const int* gcls;                  // interior patches: class in inv8 (PatchGrids)
  const int4 *wdesc, *wrow;         // the other patches (PatchGrids)
  int by_row;                       // rec is indexed by row
};
template <typename T> constexpr int inv8_ld() { return sizeof(T) == 8 ? 10 : 8; }
// row length of a packed inverse of nl rows: odd, so that the rows of a warp fall into different
// banks; the FP64 exponents are the entry after the nl-th (3D)
__host__ __device__ constexpr int wall_ld(int nl) { return (nl + 1) | 1; }

// The staged tables repeat a level's operator records (which the residual goes on reading) and its
// local inverses: 976 against 944 bytes a row in 3D at p = 2, 5008 against 3808 at p = 3, 640 against 512
// bytes per interior patch.  A level takes them only if as much device memory stays free as they fill, so that a
// problem that fits without them still does; it runs the row kernels then.  IGAMG_STAGED_FREE: the
// bytes taken as free (tests).
inline bool staged_fits(size_t bytes) {
  size_t left = 0, total = 0;
  if (const char* e = std::getenv("IGAMG_STAGED_FREE")) left = (size_t)std::strtoull(e, nullptr, 10);
  else if (cudaMemGetInfo(&left, &total) != cudaSuccess) { cudaGetLastError(); return true; }
  return bytes <= left / 2;
}

// One colour's patches (PatchGrid, igamg_internal.h).
struct ColourGrid {
  int a0, b0, na, n8, gfirst, wfirst, nwall;
};

constexpr int kExpFloor = 64;       // least exponent of a group: zeros and denormals (biased exponent 0) shift out

__device__ __forceinline__ int exp_of(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// |v| as an integer that orders as its magnitude does (exponent from bit 20 up)
__device__ __forceinline__ int top_of(double v) { return __double2hiint(v) & 0x7fffffff; }

// v != 0 without an FP64 comparison (64 cycles)
__device__ __forceinline__ bool nonzero(double v) { return (__double2hiint(v) << 1 | __double2loint(v)) != 0; }

__device__ __forceinline__ unsigned long long shr64(unsigned long long x, int s) {
  unsigned long long r;                                        // s >= 64 gives 0
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
}
__device__ __forceinline__ long long sar64(long long x, int s) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
}

// 57-bit magnitude X with sign s (+-1) as limbs
__device__ __forceinline__ int2 limbs_of(unsigned long long X, int s) {
  const int hi = (int)(X >> 28), lo = (int)((unsigned)X & 0xfffffffu);
  return make_int2(hi * s, lo * s);
}

// v as limbs relative to the exponent e (biased, >= exp_of(v), >= kExpFloor)
__device__ __forceinline__ int2 to_limbs(double v, int e) {
  const int h = __double2hiint(v);
  const unsigned long long M = ((unsigned long long)(unsigned)((h & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
  return limbs_of(shr64(M << 4, e - ((h >> 20) & 0x7ff)), (h >> 31) | 1);
}

struct Acc {
  long long hh = 0, m1 = 1ll << 27, m2 = 0;                    // three independent chains (2^27: sum rounds)
  __device__ __forceinline__ void mac(int2 x, int2 c) {
    hh += (long long)x.x * c.x;
    m1 += (long long)x.x * c.y;
    m2 += (long long)x.y * c.x;
  }
  __device__ __forceinline__ long long sum() const { return hh + ((m1 + m2) >> 28); }
};

// integer S in units of 2^(a - 1142), rounded to FP64
__device__ __forceinline__ double to_double(long long S, int a) {
  const unsigned long long m = S < 0 ? 0ull - (unsigned long long)S : (unsigned long long)S;
  const int z = __clzll((long long)m);
  const unsigned long long n = m << z;
  const int ex = a - z - 56;                                   // biased exponent of the leading bit
  const unsigned long long mant = (n >> 11) + ((n >> 10) & 1);
  unsigned long long bits = ((unsigned long long)(unsigned)(ex - 1) << 52) + mant;
  if (ex <= 0 || m == 0) bits = 0;
  if (ex >= 2047) bits = 0x7ff0000000000000ull;
  if (S < 0) bits |= 0x8000000000000000ull;
  return __longlong_as_double((long long)bits);
}

// Table entries straight into registers, 16 bytes a load, issued where they stand (they do not
// depend on the previous kernel's results and are fetched while it still runs).
__device__ __forceinline__ void ld_table(const int2* p, int2* r) {
  asm volatile("ld.global.nc.v4.s32 {%0,%1,%2,%3}, [%4];" : "=r"(r[0].x), "=r"(r[0].y), "=r"(r[1].x), "=r"(r[1].y) : "l"(p));
}
__device__ __forceinline__ void ld_table(const float* p, float* r) {
  asm volatile("ld.global.nc.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]) : "l"(p));
}
template <int N, typename E>
__device__ __forceinline__ void ld_entries(const E* __restrict__ p, E* r) {   // N entries, p 16-byte aligned
  constexpr int V = 16 / sizeof(E);
  static_assert(N % V == 0, "whole 16-byte loads");
#pragma unroll
  for (int i = 0; i < N; i += V) ld_table(p + i, r + i);
}

// The same where they are used, for the compiler to schedule.
template <int N, typename E>
__device__ __forceinline__ void ld_entries_lazy(const E* __restrict__ p, E* r) {
  constexpr int V = 16 / sizeof(E);
  static_assert(N % V == 0, "whole 16-byte loads");
#pragma unroll
  for (int i = 0; i < N; i += V) {
    const int4 q = __ldg(reinterpret_cast<const int4*>(p + i));
    if constexpr (V == 2) { r[i] = make_int2(q.x, q.y); r[i + 1] = make_int2(q.z, q.w); }
    else {
      r[i] = __int_as_float(q.x); r[i + 1] = __int_as_float(q.y);
      r[i + 2] = __int_as_float(q.z); r[i + 3] = __int_as_float(q.w);
    }
  }
}

// Waits until the kernels before this one in the stream have finished and their results are
// visible, then lets the next kernel of the stream start its own table loads.  Without the
// launch attribute both are no-ops.
__device__ __forceinline__ void dependency_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A row's local residual: FP64 as an integer in units of 2^(a - 1082), FP32 as its value.
template <typename T> struct Resid { T v; };
template <> struct Resid<double> { long long v; int a; };

// R = F - (box A) - (box B) - (third box) - m lambda for one row whose boxes start at sA, sB, sE.
// exA, exB, exE: exponents of the staged values in the three boxes; st: the row's record.
// PRE: in registers; else in global memory, read box by box (boxes begin on 16 bytes: RA).
template <int P, typename T, bool EXT, bool PRE>
__device__ __forceinline__ Resid<T> row_resid(const limb_t<T>* sA, const limb_t<T>* sB, const limb_t<T>* sE,
                                              const limb_t<T>* st, const limb_t<T>* __restrict__ se,
                                              bool is_p, int exA, int exB, int exE, T f, T lam) {
  using S = PatchShape<P>;
  if constexpr (sizeof(T) == 8) {
    Acc A, B;
    int2 ec;
    if constexpr (PRE) {
      // both boxes in one loop: a dependent 64-bit multiply-add takes some 12 cycles, and a warp that is
      // alone on its scheduler needs the six chains
#pragma unroll
      for (int j = 0; j < S::NA; ++j) {
        const int at = (j / S::C1) * S::W + j % S::C1;
        A.mac(sA[at], st[j]);
        if (j < S::NB) B.mac(sB[at], st[S::RA + j]);
      }
      ec = st[S::RA + S::NB];
    } else {
      limb_t<T> ka[S::RA], kb[S::NREC - S::RA];
      ld_entries_lazy<S::RA>(st, ka);
#pragma unroll
      for (int j = 0; j < S::NA; ++j) A.mac(sA[(j / S::C1) * S::W + j % S::C1], ka[j]);
      ld_entries_lazy<S::NREC - S::RA>(st + S::RA, kb);
#pragma unroll
      for (int j = 0; j < S::NB; ++j) B.mac(sB[(j / S::C1) * S::W + j % S::C1], kb[j]);
      ec = kb[S::NB];
    }
    const int aA = exA + ec.x, aB = exB + ec.y, exF = exp_of(f);
    int a = max(max(aA, aB), max(exF, kExpFloor));
    long long sE_ = 0, sL = 0;
    int aE = 0, aL = 0;
    if (EXT && !is_p) {
      Acc E;
#pragma unroll
      for (int d = 0; d < S::W; ++d)
#pragma unroll
        for (int e = 0; e < S::W; ++e) E.mac(sE[d * S::W + e], se[d * S::W + e]);
      aE = exE + se[S::W * S::W].x;
      sE_ = E.sum();
      a = max(a, aE);
    }
    if (is_p && nonzero(lam)) {                                  // (lam is the same for the whole grid)
      const int exL = max(exp_of(lam), kExpFloor);
      Acc Lm;
      Lm.mac(to_limbs(lam, exL), st[S::IL]);
      aL = exL + st[S::IL + 1].x;
      sL = Lm.sum();
      a = max(a, aL);
    }
    const int h = __double2hiint(f);
    const unsigned long long M = ((unsigned long long)(unsigned)((h & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(f);
    long long r = (long long)shr64(M << 7, a - exF);
    if (h < 0) r = -r;
    r -= sar64(A.sum(), a - aA);
    r -= sar64(B.sum(), a - aB);
    if (EXT) r -= sar64(sE_, a - aE);
    if (is_p && nonzero(lam)) r -= sar64(sL, a - aL);
    return {r, a};
  } else {
    T a0 = T(0), a1 = T(0), b0 = T(0), b1 = T(0);
    limb_t<T> own[PRE ? 4 : S::NREC];
    if constexpr (!PRE) ld_entries_lazy<S::NREC>(st, own);
    const limb_t<T>* k = PRE ? st : own;
#pragma unroll
    for (int j = 0; j < S::NA; ++j) {
      const T v = sA[(j / S::C1) * S::W + j % S::C1];
      if (j & 1) a1 = fma(k[j], v, a1);
      else a0 = fma(k[j], v, a0);
    }
#pragma unroll
    for (int j = 0; j < S::NB; ++j) {
      const T v = sB[(j / S::C1) * S::W + j % S::C1];
      if (j & 1) b1 = fma(k[S::RA + j], v, b1);
      else b0 = fma(k[S::RA + j], v, b0);
    }
    if (is_p) b1 = fma(k[S::IL], lam, b1);
    if (EXT && !is_p) {
#pragma unroll
      for (int j = 0; j < S::W * S::W; ++j) {
        if (j & 1) b1 = fma(se[j], sE[j], b1);
        else b0 = fma(se[j], sE[j], b0);
      }
    }
    return {f - ((a0 + a1) + (b0 + b1))};
  }
}

__device__ __forceinline__ double resid_value(const Resid<double>& r) { return to_double(r.v, r.a + 60); }
__device__ __forceinline__ float resid_value(const Resid<float>& r) { return r.v; }

// exponent of a local residual on the scale of its unit (|r| < 2^(exponent - 1082)); 0 for r = 0
__device__ __forceinline__ int resid_exp(const Resid<double>& r) {
  const unsigned long long m = r.v < 0 ? 0ull - (unsigned long long)r.v : (unsigned long long)r.v;
  return m ? r.a + 64 - __clzll((long long)m) : 0;
}
// local residual as limbs relative to the exponent e of its group
__device__ __forceinline__ int2 resid_limbs(const Resid<double>& r, int er, int e) {
  const unsigned long long m = r.v < 0 ? 0ull - (unsigned long long)r.v : (unsigned long long)r.v;
  const unsigned long long Z = er ? m << (64 - (er - r.a)) : 0ull;   // leading bit at 63
  return limbs_of(shr64(Z, 7 + e - er), r.v < 0 ? -1 : 1);
}

// maxima over eight lanes of two exponents (16 bits each)
__device__ __forceinline__ unsigned max16x2(unsigned x, unsigned y) {
  unsigned r;
  asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(y));
  return r;
}
__device__ __forceinline__ unsigned group_max8(unsigned v) {
  v = max16x2(v, __shfl_xor_sync(0xffffffffu, v, 1));
  v = max16x2(v, __shfl_xor_sync(0xffffffffu, v, 2));
  return max16x2(v, __shfl_xor_sync(0xffffffffu, v, 4));
}

// ---- interior patches: four per warp, lane = (patch, local row) -----------------------------
// tables(): everything that does not depend on U or F, into registers (one memory round trip that
// overlaps the previous kernel); solve(): the neighbourhood, the residual rows, the inverse.
// All 32 lanes call together.
template <int P, typename T, bool EXT, bool PRE>
struct Patch8 {
  using S = PatchShape<P>;
  using E = limb_t<T>;
  E st_[PRE ? S::NREC : 4], A[PRE ? inv8_ld<T>() : 4];
  const E *st, *Ap;
  int a, b, g, nx, ny, np;          // nx, ny, np: the lane's first entries of the three arrays in U
  int ex, ey, ep;                   // exponents of the staged u_x, u_y and pressures
  T f, lam, u_own;
  bool active;

  __device__ __forceinline__ void tables(const LevelTab<T>& L, const PatchTab<T>& X, const ColourGrid& C, int w, int lane) {
    constexpr int TC = 2 * P + 1, NC = 2 * TC + 1;
    const int wpr = (C.na + 3) >> 2, j = w / wpr, i = (w - j * wpr) * 4 + (lane >> 3);
    active = i < C.na;
    const int ii = active ? i : C.na - 1, row = lane & 7;
    const int icls = X.gcls[C.gfirst + j * C.na + ii];
    a = C.a0 + ii * (P + 1);
    b = C.b0 + j * (P + 1);
    const bool is_p = row >= 4, is_y = row == 2 || row == 3;
    const int o = row & 1, o2 = (row >> 1) & 1;                // pressure rows: x offset o, y offset o2
    const int ix = is_p || is_y ? a - 1 + o : a, iy = is_p ? b - 1 + o2 : (is_y ? b : b - 1 + o);
    g = is_p ? L.n_ux + L.n_uy + iy * L.npd + ix : (is_y ? L.n_ux + (iy - 1) * L.npd + ix : iy * L.nxu + ix - 1);
    const int k = X.by_row ? g
                           : (is_p ? 2 : (is_y ? 1 : 0)) * NC * NC +
                                 cls1d<P>(ix, is_p || is_y ? L.lastq : L.lastp) * NC + cls1d<P>(iy, is_y ? L.lastp : L.lastq);
    {
      const int d = row / S::W, c = row - d * S::W;            // entry e = row + 8 k; k = 0
      nx = (b - P + c) * L.nxu + (a - P - 1) + d;
      ny = L.n_ux + (b - P - 1 + d) * L.npd + (a - P) + c;
      np = L.n_ux + L.n_uy + (b - P + c) * L.npd + (a - P) + d;
    }
    st = X.rec + (size_t)k * S::NREC;
    Ap = X.inv8 + ((size_t)icls * 8 + row) * inv8_ld<T>();
    if constexpr (PRE) {
      ld_entries<S::NREC>(st, st_);
      ld_entries<inv8_ld<T>()>(Ap, A);
    }
  }

  // stages the neighbourhood; the local residual of the lane's row
  __device__ __forceinline__ Resid<T> residual(const LevelTab<T>& L, const PatchTab<T>& X, const T* U, const T* F, int lane,
                                               E* sm) {
    constexpr int KU = (S::NUX + 7) / 8, KP = (S::NP + 7) / 8;
    const int row = lane & 7;
    E* reg = sm + (lane >> 3) * S::REG;
    const bool is_p = row >= 4, is_y = row == 2 || row == 3;
    const int o = row & 1, o2 = (row >> 1) & 1;
    // the neighbourhood: entry e = row + 8 k of each array
    T vx[KU], vy[KU], vp[KP];
    if constexpr (S::W == 4) {                                 // e -> e + 8: two steps along the long axis
#pragma unroll
      for (int k = 0; k < KU; ++k) {
        const bool in = S::NUX % 8 == 0 || k < KU - 1 || row + 8 * k < S::NUX;
        vx[k] = in ? U[nx + 2 * k] : T(0);
        vy[k] = in ? U[ny + 2 * k * L.npd] : T(0);
      }
#pragma unroll
      for (int k = 0; k < KP; ++k) vp[k] = U[np + 2 * k];
    } else {
      const int d0 = row / S::W, c0 = row - d0 * S::W;
#pragma unroll
      for (int k = 0; k < KU; ++k) {
        const int e = row + 8 * k, d = e / S::W - d0, c = e % S::W - c0;
        const bool in = S::NUX % 8 == 0 || k < KU - 1 || e < S::NUX;
        vx[k] = in ? U[nx + c * L.nxu + d] : T(0);
        vy[k] = in ? U[ny + d * L.npd + c] : T(0);
      }
#pragma unroll
      for (int k = 0; k < KP; ++k) {
        const int e = row + 8 * k, d = e / S::W - d0, c = e % S::W - c0;
        vp[k] = (S::NP % 8 == 0 || k < KP - 1 || e < S::NP) ? U[np + c * L.npd + d] : T(0);
      }
    }
    f = F[g];
    lam = U[L.n_total - 1];
    u_own = U[g];
    ex = ey = ep = kExpFloor << 20;
    if constexpr (sizeof(T) == 8) {
#pragma unroll
      for (int k = 0; k < KU; ++k) {
        ex = max(ex, top_of(vx[k]));
        ey = max(ey, top_of(vy[k]));
      }
#pragma unroll
      for (int k = 0; k < KP; ++k) ep = max(ep, top_of(vp[k]));
      const unsigned exy = group_max8((unsigned)(ex >> 20 | (ey >> 20) << 16));
      ex = (int)(exy & 0xffff);
      ey = (int)(exy >> 16);
      ep = (int)group_max8((unsigned)ep >> 20);
    }
    auto stage = [&](T v, int e) -> E {
      if constexpr (sizeof(T) == 8) return to_limbs(v, e);
      else return v;
    };
#pragma unroll
    for (int k = 0; k < KU; ++k) {
      const int e = row + 8 * k;
      if (S::NUX % 8 == 0 || k < KU - 1 || e < S::NUX) {
        reg[e] = stage(vx[k], ex);
        reg[S::UY + e] = stage(vy[k], ey);
      }
    }
#pragma unroll
    for (int k = 0; k < KP; ++k) {
      const int e = row + 8 * k, d = e / S::W, c = e - d * S::W;
      if (S::NP % 8 == 0 || k < KP - 1 || e < S::NP) {
        const E v = stage(vp[k], ep);
        reg[S::PX + e] = v;
        reg[S::PY + c * S::W + d] = v;
      }
    }
    if constexpr (sizeof(T) == 4) {                            // pressure rows read the gap after UX times zero
#pragma unroll
      for (int k = S::NUX; k < S::UY; k += 8)
        if (k + row < S::UY) reg[k + row] = T(0);
    }
    __syncwarp();
    const E* sA = reg + (is_p ? o * S::W + o2 : (is_y ? S::UY + o : o));
    const E* sB = reg + (is_p ? S::UY + o2 * S::W + o : (is_y ? S::PY + o : S::PX + o));
    const E* sE = reg + (is_y ? o * S::W : S::UY + o * S::W);
    const E* se = EXT ? X.ext + (size_t)(is_p ? 0 : g) * S::NEXT : nullptr;
    return row_resid<P, T, EXT, PRE>(sA, sB, sE, PRE ? st_ : st, se, is_p, is_y ? ey : ex, is_p ? ey : ep, is_y ? ex : ey, f, lam);
  }

  __device__ __forceinline__ void solve(const LevelTab<T>& L, const PatchTab<T>& X, T* U, const T* F, int lane, E* sm) {
    const int row = lane & 7;
    E* reg = sm + (lane >> 3) * S::REG;
    const bool is_p = row >= 4;
    const Resid<T> r = residual(L, X, U, F, lane, sm);
    __syncwarp();
    E A_[PRE ? 4 : inv8_ld<T>()];
    if constexpr (!PRE) ld_entries_lazy<inv8_ld<T>()>(Ap, A_);
    const E* A = PRE ? this->A : A_;
    if constexpr (sizeof(T) == 8) {
      const int er = resid_exp(r);
      int eg = max(er, __shfl_xor_sync(0xffffffffu, er, 1));
      eg = max(eg, __shfl_xor_sync(0xffffffffu, eg, 2));
      const int eo = __shfl_xor_sync(0xffffffffu, eg, 4);
      reg[row] = resid_limbs(r, er, eg);
      __syncwarp();
      Acc D0, D1;
#pragma unroll
      for (int s = 0; s < 4; ++s) { D0.mac(reg[s], A[s]); D1.mac(reg[4 + s], A[4 + s]); }
      const int a0 = (is_p ? eo : eg) + A[8].x, a1 = (is_p ? eg : eo) + A[8].y, am = max(a0, a1);
      double d = to_double(sar64(D0.sum(), am - a0) + sar64(D1.sum(), am - a1), am);
      // a value that is not finite in the neighbourhood or in F: the whole patch becomes NaN
      const bool bad = max(max(ex, ey), ep) == 0x7ff || exp_of(f) == 0x7ff || exp_of(lam) == 0x7ff;
      const unsigned any = __ballot_sync(0xffffffffu, bad);
      if ((any >> (lane & 24)) & 0xffu) d = __longlong_as_double(0x7ff8000000000000ll);
      if (active) U[g] = u_own + d;
    } else {
      T d[2] = {T(0), T(0)};
#pragma unroll
      for (int s = 0; s < 8; ++s) d[s & 1] = fma(A[s], __shfl_sync(0xffffffffu, r.v, (lane & ~7) + s), d[s & 1]);
      if (active) U[g] = u_own + (d[0] + d[1]);
    }
    __syncwarp();                                              // reg is free for the warp's next patches
  }
};

// Barrier of the LW threads that share a wall patch (a warp, or two with a named barrier of the
// block: barrier 1 + the pair's index).
template <int LW>
__device__ __forceinline__ void wall_sync() {
  if constexpr (LW == 32) __syncwarp();
  else asm volatile("bar.sync %0, 64;" ::"r"(1 + (int)(threadIdx.x >> 6)) : "memory");
}

// Shared-memory entries of one wall patch: margins, the arrays, the local residuals, reduction
// slots, and the inverse.
template <int P>
__host__ __device__ constexpr int wall_entries(int maxl) {
  return (2 * PatchShape<P>::MARGIN + PatchShape<P>::REG + PatchShape<P>::LW + 16 + maxl * PatchShape<P>::LDW + 3) / 4 * 4;
}
// Shared-memory entries per group of LW threads: one wall patch, or each warp's four patches.
template <int P>
__host__ __device__ constexpr int group_entries(int maxl) {
  return wall_entries<P>(maxl) > 4 * PatchShape<P>::REG * (PatchShape<P>::LW / 32)
             ? wall_entries<P>(maxl)
             : 4 * PatchShape<P>::REG * (PatchShape<P>::LW / 32);
}

// ---- the other patches (on or near a wall, up to LW rows): LW threads each, thread = row ----------
template <int P, typename T, bool EXT, bool PRE>
struct PatchWall {
  using S = PatchShape<P>;
  using E = limb_t<T>;
  static constexpr int K = (S::NLOAD + S::LW - 1) / S::LW;
  E st_[PRE ? S::NREC : 4];
  int at[K];                        // the thread's neighbourhood values in U, -1: outside
  int ex, ey, ep;                   // exponents of the staged u_x, u_y and pressures
  T u_own;
  bool bad;                         // a value that is not finite (in F, lambda: of this thread or its warp)
  int4 D, R;                        // D: a | b << 16, offset of the inverse (16 B), rows | velocity rows << 8
                                    // R: row, offset of box A | of box B << 16, of the third box, record

  // t: thread within the group; sm: the group's shared memory
  __device__ __forceinline__ void tables(const LevelTab<T>& L, const PatchTab<T>& X, int w, int t, E* sm) {
    D = X.wdesc[w];
    R = X.wrow[(size_t)w * S::LW + t];
    const int nl = D.z & 0xff;
    E* inv = sm + 2 * S::MARGIN + S::REG + S::LW + 16;
    const char* src = reinterpret_cast<const char*>(X.winv) + (size_t)D.y * 16;
    const int n16 = (int)((nl * S::LDW * sizeof(E) + 15) / 16);
    const unsigned dst = (unsigned)__cvta_generic_to_shared(inv);
    for (int i = t; i < n16; i += S::LW)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * i), "l"(src + 16 * (size_t)i) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
    if constexpr (PRE) ld_entries<S::NREC>(X.rec + (size_t)R.w * S::NREC, st_);   // threads past the last row: record 0
    const int a = D.x & 0xffff, b = D.x >> 16, nu = L.n_ux + L.n_uy;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int e = t + S::LW * k;
      const bool uy = e >= S::NUX, pr = e >= 2 * S::NUX;
      const int e1 = e - (pr ? 2 * S::NUX : (uy ? S::NUX : 0)), d = e1 / S::W, cc = e1 - d * S::W;
      // u_y: y outer; u_x and pressure: x outer
      const int x = a - P + (uy && !pr ? cc : d), y = b - P + (uy && !pr ? d : cc);
      const int xlo = uy ? 0 : 1, xhi = uy ? L.lastq : L.nint, ylo = uy && !pr ? 1 : 0, yhi = uy && !pr ? L.nint : L.lastq;
      const bool in = e < S::NLOAD && x >= xlo && x <= xhi && y >= ylo && y <= yhi;
      at[k] = in ? (pr ? nu : (uy ? L.n_ux : 0)) + (y - ylo) * (uy ? L.npd : L.nxu) + x - xlo : -1;
    }
  }

  // stages the neighbourhood; the local residual of the thread's row
  __device__ __forceinline__ Resid<T> residual(const LevelTab<T>& L, const PatchTab<T>& X, const T* U, const T* F, int t, E* sm) {
    const int nl = D.z & 0xff, g = R.x, nu = L.n_ux + L.n_uy;
    E* reg = sm + S::MARGIN;
    int* red = reinterpret_cast<int*>(reg + S::REG + S::MARGIN + S::LW);   // LW = 64: maxima of the two warps
    T v[K];
    ex = ey = ep = kExpFloor;
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = at[k] >= 0 ? U[at[k]] : T(0);
    const bool has = t < nl, is_p = g >= nu;
    const T f = has ? F[g] : T(0), lam = U[L.n_total - 1];
    u_own = has ? U[g] : T(0);
    bad = false;
    if constexpr (sizeof(T) == 8) {
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (t + S::LW * k >= 2 * S::NUX) ep = max(ep, exp_of(v[k]));
        else if (t + S::LW * k >= S::NUX) ey = max(ey, exp_of(v[k]));
        else ex = max(ex, exp_of(v[k]));
      }
      ex = __reduce_max_sync(0xffffffffu, ex);
      ey = __reduce_max_sync(0xffffffffu, ey);
      ep = __reduce_max_sync(0xffffffffu, ep);
      bad = exp_of(f) == 0x7ff || exp_of(lam) == 0x7ff;
      if constexpr (S::LW == 64) {
        const int any = __any_sync(0xffffffffu, bad);
        if ((t & 31) == 0) { red[t >> 5] = ex; red[2 + (t >> 5)] = ep; red[4 + (t >> 5)] = any; red[6 + (t >> 5)] = ey; }
        wall_sync<S::LW>();
        ex = max(red[0], red[1]);
        ey = max(red[6], red[7]);
        ep = max(red[2], red[3]);
        bad = red[4] | red[5];
      }
    } else {
      // what rows read with zero coefficients must be finite: the margins and the gaps
      for (int i = t; i < 2 * S::MARGIN + S::REG; i += S::LW) sm[i] = T(0);
      wall_sync<S::LW>();
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int e = t + S::LW * k;
      if (e >= S::NLOAD) continue;
      E w;
      if constexpr (sizeof(T) == 8) w = to_limbs(v[k], e >= 2 * S::NUX ? ep : (e >= S::NUX ? ey : ex));
      else w = v[k];
      const int e1 = e - (e >= 2 * S::NUX ? 2 * S::NUX : (e >= S::NUX ? S::NUX : 0));
      reg[e1 + (e >= 2 * S::NUX ? S::PX : (e >= S::NUX ? S::UY : 0))] = w;
      if (e >= 2 * S::NUX) {
        const int d = e1 / S::W;
        reg[S::PY + (e1 - d * S::W) * S::W + d] = w;
      }
    }
    wall_sync<S::LW>();
    const E* sA = reg + (short)(R.y & 0xffff);
    const E* sB = reg + (R.y >> 16);
    const E* se = EXT ? X.ext + (size_t)(is_p || !has ? 0 : g) * S::NEXT : nullptr;
    const bool is_y = g >= L.n_ux && !is_p;
    return row_resid<P, T, EXT, PRE>(sA, sB, reg + R.z, PRE ? st_ : X.rec + (size_t)R.w * S::NREC, se, is_p, is_y ? ey : ex,
                                     is_p ? ey : ep, is_y ? ex : ey, f, lam);
  }

  __device__ __forceinline__ void solve(const LevelTab<T>& L, const PatchTab<T>& X, T* U, const T* F, int t, E* sm) {
    const int nl = D.z & 0xff, nv = D.z >> 8, g = R.x;
    const bool has = t < nl, is_p = g >= L.n_ux + L.n_uy;
    E* rl = sm + 2 * S::MARGIN + S::REG;
    int* red = reinterpret_cast<int*>(rl + S::LW);
    const E* inv = rl + S::LW + 16;
    const Resid<T> r = residual(L, X, U, F, t, sm);
    asm volatile("cp.async.wait_all;" ::: "memory");
    const E* Ak = inv + (has ? t : 0) * S::LDW;
    const int slot = t < nv ? t : S::MV + t - nv;              // the row's column in the inverses
    // columns that the patch does not have (their entries in the inverse are zero)
    if (t < S::MV + S::MP && (t < S::MV ? t >= nv : t - S::MV >= nl - nv)) {
      if constexpr (sizeof(T) == 8) rl[t] = make_int2(0, 0);
      else rl[t] = T(0);
    }
    if constexpr (sizeof(T) == 8) {
      const int er = has ? resid_exp(r) : 0;
      int gu = __reduce_max_sync(0xffffffffu, is_p ? 0 : er), gp = __reduce_max_sync(0xffffffffu, is_p ? er : 0);
      bad = bad || max(max(ex, ey), ep) == 0x7ff;
      if constexpr (S::LW == 64) {
        if ((t & 31) == 0) { red[8 + (t >> 5)] = gu; red[10 + (t >> 5)] = gp; }
        wall_sync<S::LW>();
        gu = max(red[8], red[9]);
        gp = max(red[10], red[11]);
      } else {
        bad = __any_sync(0xffffffffu, bad);
      }
      if (has) rl[slot] = resid_limbs(r, er, is_p ? gp : gu);
      wall_sync<S::LW>();                                      // (also makes every thread's cp.async visible)
      Acc D0, D1;
#pragma unroll
      for (int s = 0; s < S::MV; ++s) {
        D0.mac(rl[s], Ak[s]);
        if (s < S::MP) D1.mac(rl[S::MV + s], Ak[S::MV + s]);
      }
      const int2 ec = Ak[S::MV + S::MP];
      const int a0 = gu + ec.x, a1 = gp + ec.y, am = max(a0, a1);
      double d = to_double(sar64(D0.sum(), am - a0) + sar64(D1.sum(), am - a1), am);
      if (bad) d = __longlong_as_double(0x7ff8000000000000ll);
      if (has) U[g] = u_own + d;
    } else {
      if (has) rl[slot] = r.v;
      wall_sync<S::LW>();
      T d[3] = {T(0), T(0), T(0)};
#pragma unroll
      for (int s = 0; s < S::MV + S::MP; ++s) d[s % 3] = fma(Ak[s], rl[s], d[s % 3]);
      if (has) U[g] = u_own + ((d[0] + d[1]) + d[2]);
    }
    wall_sync<S::LW>();                                        // the shared memory is free again
  }
};

// Group w of LW threads of one colour's work: the wall patches first (their chains are the
// longest), then the interior patches, four to a warp along x.  WAIT: the kernel's dependency wait
// stands between the table loads and the solve, in a loop of `once` (always 1) rounds that the
// compiler cannot unroll: it then computes every address and table value that does not depend on U
// before the loop, ahead of the wait, instead of sinking them to their uses.  Measured per colour
// with and without the loop: p = 3 64^2 2.65 and 3.08 us, 128^2 3.1 and 3.8, p = 2 128^2 2.5 and 2.9,
// 256^2 5.0-5.5 and 5.0 (more registers); V-cycle p = 3 72^2 614 and 697 us.
// ROWS: no solve; U is read only, and the rows' local residuals go to R.
template <int P, typename T, bool EXT, bool PRE, bool WAIT, bool ROWS = false>
__device__ __forceinline__ void colour_group(const LevelTab<T>& L, const PatchTab<T>& X, T* U, const T* F,
                                             const ColourGrid& C, int w, int t, limb_t<T>* sm, int once, T* R = nullptr) {
  using S = PatchShape<P>;
  if (w < C.nwall) {
    PatchWall<P, T, EXT, PRE> W;
    W.tables(L, X, C.wfirst + w, t, sm);
#pragma unroll 1
    for (int k = 0; k < (WAIT ? once : 1); ++k) {
      if (WAIT) dependency_wait();
      if constexpr (ROWS) {
        const Resid<T> r = W.residual(L, X, U, F, t, sm);
        if (t < (W.D.z & 0xff)) R[W.R.x] = resid_value(r);
        asm volatile("cp.async.wait_all;" ::: "memory");
      } else {
        W.solve(L, X, U, F, t, sm);
      }
    }
  } else {
    const int wp = (w - C.nwall) * (S::LW / 32) + (t >> 5);
    if (wp >= C.n8 / max(C.na, 1) * ((C.na + 3) >> 2)) return;
    Patch8<P, T, EXT, PRE> I;
    I.tables(L, X, C, wp, t & 31);
#pragma unroll 1
    for (int k = 0; k < (WAIT ? once : 1); ++k) {
      if (WAIT) dependency_wait();
      limb_t<T>* smw = sm + (t >> 5) * 4 * S::REG;
      if constexpr (ROWS) {
        const Resid<T> r = I.residual(L, X, U, F, t & 31, smw);
        if (I.active) R[I.g] = resid_value(r);
      } else {
        I.solve(L, X, U, F, t & 31, smw);
      }
    }
  }
}
template <int P>
__host__ __device__ inline int colour_groups(const ColourGrid& C) {
  constexpr int wpg = PatchShape<P>::LW / 32;
  return C.nwall + (C.n8 ? (C.n8 / C.na * ((C.na + 3) >> 2) + wpg - 1) / wpg : 0);
}

// One colour of the sweep.  Threads per block: 64 (two groups at p = 2, one at p = 3).  The records
// are fetched into registers before the dependency wait: reading them in place instead (twice the
// warps per SM) measured 2.75 against 2.2 us on 64^2, 6.4 against 6.5 on 256^2 (p = 2).
template <int P, typename T, bool EXT>
__global__ void __launch_bounds__(64) k_patch_colour(const __grid_constant__ LevelTab<T> L, const __grid_constant__ PatchTab<T> X,
                                                     T* U, const T* F, const ColourGrid C, int ngroups, int smg, int once) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int LW = PatchShape<P>::LW;
  const int gib = threadIdx.x / LW, w = blockIdx.x * (64 / LW) + gib;
  if (w >= ngroups) return;
  colour_group<P, T, EXT, true, true>(L, X, U, F, C, w, threadIdx.x % LW, reinterpret_cast<limb_t<T>*>(smem_raw) + gib * smg,
                                      once);
}

// The local residuals F - K U of the rows of one colour's patches as the colour kernel forms them
// (a measuring hook: what its arithmetic makes of a row before the local inverse mixes the rows).
template <int P, bool EXT>
__global__ void __launch_bounds__(64) k_patch_rows(const __grid_constant__ LevelTab<double> L,
                                                   const __grid_constant__ PatchTab<double> X, double* U, const double* F,
                                                   double* R, const ColourGrid C, int ngroups, int smg) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int LW = PatchShape<P>::LW;
  const int gib = threadIdx.x / LW, w = blockIdx.x * (64 / LW) + gib;
  if (w >= ngroups) return;
  colour_group<P, double, EXT, true, false, true>(L, X, U, F, C, w, threadIdx.x % LW,
                                                  reinterpret_cast<int2*>(smem_raw) + gib * smg, 1, R);
}

// ---- building the tables (once, at creation) ---------------------------------------------------

// exponent s with sum |c| < 2^(s-1) (s = -4096 for zeros), and c as limbs on that scale
__device__ __forceinline__ int sum_exp(double sum) { return sum > 0.0 ? ilogb(sum) + 2 : -4096; }
__device__ __forceinline__ int2 coef_limbs(double c, int s) {
  const long long C = s < -4000 ? 0 : __double2ll_rn(ldexp(c, 59 - s));
  const long long hi = (C + (1ll << 27)) >> 28;
  return make_int2((int)hi, (int)(C - (hi << 28)));
}

// Box entry j of the staged layout (long axis outer) -> index in the stored record (x outer).
template <int P>
__device__ __forceinline__ int box_src(int kind, bool boxB, int j) {
  using S = PatchShape<P>;
  const int d = j / S::C1, e = j % S::C1;                      // d along, e across
  if (!boxB) return kind == 1 ? e * S::A1 + d : j;             // u_y rows: stored x (across) outer
  if (kind == 0) return S::NA + j;
  return S::NA + e * S::B1 + d;                                // u_y and pressure rows: y is the long axis
}

// Row records: src has RU entries per record; kind 0/1/2 = u_x / u_y / pressure rows, or -1: rows
// of a level in order (n_ux u_x rows, n_uy u_y rows, then pressure rows).
template <int P, typename T>
__global__ void k_patch_records(int n, int kind, int n_ux, int n_uy, const T* __restrict__ src, limb_t<T>* __restrict__ dst) {
  using S = PatchShape<P>;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int k = kind >= 0 ? kind : (i < n_ux ? 0 : (i < n_ux + n_uy ? 1 : 2));
  const T* s = src + (size_t)i * S::RU;
  limb_t<T>* d = dst + (size_t)i * S::NREC;
  if constexpr (sizeof(T) == 8) {
    double sa = 0, sb = 0;
    for (int j = 0; j < S::NA; ++j) sa += fabs(s[j]);
    for (int j = 0; j < S::NB; ++j) sb += fabs(s[S::NA + j]);
    const int ea = sum_exp(sa), eb = sum_exp(sb), el = sum_exp(fabs(s[S::RU - 1]));
    for (int j = 0; j < S::NA; ++j) d[j] = coef_limbs(s[box_src<P>(k, false, j)], ea);
    for (int j = S::NA; j < S::RA; ++j) d[j] = make_int2(0, 0);
    for (int j = 0; j < S::NB; ++j) d[S::RA + j] = coef_limbs(s[box_src<P>(k, true, j)], eb);
    d[S::RA + S::NB] = make_int2(ea, eb);
    d[S::IL] = coef_limbs(s[S::RU - 1], el);
    d[S::IL + 1] = make_int2(el, 0);
    for (int j = S::IL + 2; j < S::NREC; ++j) d[j] = make_int2(0, 0);
  } else {
    for (int j = 0; j < S::NA; ++j) d[j] = s[box_src<P>(k, false, j)];
    for (int j = S::NA; j < S::NREC; ++j) d[j] = T(0);
    for (int j = 0; j < S::NB; ++j) d[S::RA + j] = s[box_src<P>(k, true, j)];
    d[S::IL] = s[S::RU - 1];
  }
}

// Third box of mapped domains per velocity row (stored x outer): u_x rows read u_y with y outer.
template <int P, typename T>
__global__ void k_patch_ext(int n, int n_ux, const T* __restrict__ src, limb_t<T>* __restrict__ dst) {
  using S = PatchShape<P>;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const T* s = src + (size_t)i * S::NP;
  limb_t<T>* d = dst + (size_t)i * S::NEXT;
  auto at = [&](int j) { return i < n_ux ? (j % S::W) * S::W + j / S::W : j; };
  if constexpr (sizeof(T) == 8) {
    double sum = 0;
    for (int j = 0; j < S::NP; ++j) sum += fabs(s[j]);
    const int e = sum_exp(sum);
    for (int j = 0; j < S::NP; ++j) d[j] = coef_limbs(s[at(j)], e);
    d[S::NP] = make_int2(e, 0);
    for (int j = S::NP + 1; j < S::NEXT; ++j) d[j] = make_int2(0, 0);
  } else {
    for (int j = 0; j < S::NP; ++j) d[j] = s[at(j)];
    for (int j = S::NP; j < S::NEXT; ++j) d[j] = T(0);
  }
}

// One local inverse row of nl entries (the first nv the velocity columns) with its exponents.
template <typename T>
__device__ __forceinline__ void inverse_row(const T* s, int nl, int nv, limb_t<T>* d) {
  if constexpr (sizeof(T) == 8) {
    double su = 0, sp = 0;
    for (int j = 0; j < nl; ++j) (j < nv ? su : sp) += fabs(s[j]);
    const int eu = sum_exp(su), ep = sum_exp(sp);
    for (int j = 0; j < nl; ++j) d[j] = coef_limbs(s[j], j < nv ? eu : ep);
    d[nl] = make_int2(eu, ep);
  } else {
    for (int j = 0; j < nl; ++j) d[j] = s[j];
  }
}

// Interior patches: 8 rows of 8 per class.
template <typename T>
__global__ void k_patch_inv8(int ncls, const T* __restrict__ src, limb_t<T>* __restrict__ dst) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < ncls * 8) inverse_row<T>(src + (size_t)i * 8, 8, 4, dst + (size_t)i * inv8_ld<T>());
}

// The other patches: one block per class c of spec (x: class in cinv8 (-1 - x) or cinv, y: offset of
// the result in 16 bytes, z: rows | velocity rows << 8), threads over its rows.
template <int P, typename T>
__global__ void k_patch_winv(int maxl, const int4* __restrict__ spec, const T* __restrict__ cinv, const T* __restrict__ cinv8,
                             limb_t<T>* __restrict__ dst) {
  const int4 s = spec[blockIdx.x];
  const int nl = s.z & 0xff, nv = s.z >> 8, r = threadIdx.x;
  if (r >= nl) return;
  const T* src = s.x < 0 ? cinv8 + ((size_t)(-1 - s.x) * 8 + r) * 8 : cinv + ((size_t)s.x * maxl + r) * maxl;
  using S = PatchShape<P>;
  limb_t<T>* d = reinterpret_cast<limb_t<T>*>(reinterpret_cast<char*>(dst) + (size_t)s.y * 16) + r * S::LDW;
  limb_t<T> row[S::MV + S::MP + 1];
  inverse_row<T>(src, nl, nv, row);
  for (int j = 0; j < S::LDW; ++j) {
    limb_t<T> v{};
    if (j < nv) v = row[j];
    else if (j >= S::MV && j - S::MV < nl - nv) v = row[nv + j - S::MV];
    else if (sizeof(T) == 8 && j == S::MV + S::MP) v = row[nl];
    d[j] = v;
  }
}

// ---- lockstep batches of any mesh sizes: one launch per V-cycle step over every solve -------
// The solves of a batch share p and the cycle shape but may differ in mesh size and number
// of grids.  Their V-cycles are aligned from the finest grid down: at depth t (0 = finest) a
// solve with L grids is on its level L - 1 - t.  A launch covers up to kMixChunk solves of any
// sizes (blockIdx.y = solve), their descriptors for that depth in the kernel parameters;
// larger batches are cut into chunks that run as parallel branches of one graph.  A block
// whose solve is converged, past its coarsest level, not on a level that takes part in the
// step, or beyond that solve's work, returns at once.
template <typename T>
struct MixLevel {
  int level;                      // level index in the solve's hierarchy, -1 past its coarsest
  int lpr;                        // lanes per 8-DOF patch row of the level's colour kernel
  int staged;                     // 1: staged patch solves (X, grid)
  LevelTab<T> L, Lc;              // this level and (level >= 1) the next coarser one
  Xfer<T> tp, tq;                 // transfers between Lc and L
  const T *cinv, *cinv8, *kinv;   // local inverses; kinv: the coarsest level's dense inverse
  T *U, *F, *R, *Uc, *Fc;
  const int *dofs, *cls, *nloc;
  int maxl;
  int first[kMaxColours], n8[kMaxColours], cnt[kMaxColours];
  PatchTab<T> X;
  ColourGrid grid[kMaxColours];
  double* part;                   // residual partials (two per block of 256 rows)
  double* norm2;                  // ||F - K U||^2 of the finest level
  const int* active;              // 1 while the solve is iterating
};

constexpr int kMixChunk = 24;     // solves per launch (descriptors in the kernel parameters)

template <typename T>
struct MixArgs {
  int count;
  MixLevel<T> s[kMixChunk];
};

template <int P, typename T, bool EXT>
__global__ void __launch_bounds__(128) k_mix_colour(const __grid_constant__ MixArgs<T> A, int c, int smg) {
  const MixLevel<T>& d = A.s[blockIdx.y];
  if (d.level < 1 || !*d.active) return;
  if (d.staged) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const ColourGrid C = d.grid[c];
    constexpr int LW = PatchShape<P>::LW;
    const int gib = threadIdx.x / LW, w = blockIdx.x * (blockDim.x / LW) + gib;
    if (w >= colour_groups<P>(C)) return;
    const LevelTab<T> L = d.L;
    const PatchTab<T> X = d.X;
    colour_group<P, T, EXT, false, false>(L, X, d.U, d.F, C, w, threadIdx.x % LW,
                                   reinterpret_cast<limb_t<T>*>(smem_raw) + gib * smg, 1);
    return;
  }
  const int wpb = blockDim.x >> 5, ppw = d.lpr == 2 ? 2 : 4;
  const int n8 = d.n8[c], ngen = d.cnt[c] - n8;
  const int nb8 = (n8 + ppw * wpb - 1) / (ppw * wpb), nbg = (ngen + wpb - 1) / wpb;
  if ((int)blockIdx.x >= nb8 + nbg) return;
  const LevelTab<T> L = d.L;
  T* U = d.U;
  const T* F = d.F;
  const int *dofs = d.dofs, *cls = d.cls, *nloc = d.nloc;
  const T *cinv = d.cinv, *cinv8 = d.cinv8;
  const int maxl = d.maxl, first = d.first[c];
  // the block walks the solve's blocks with the grid's stride (a descriptor read serves
  // several rounds of patches)
  for (int b = blockIdx.x; b < nb8 + nbg; b += gridDim.x) {
    if (d.lpr == 2)
      mult_colour_block<P, T, 2>(L, U, F, dofs, cls, cinv, cinv8, nloc, maxl, first, n8, ngen, nb8, b);
    else
      mult_colour_block<P, T, 1, 2>(L, U, F, dofs, cls, cinv, cinv8, nloc, maxl, first, n8, ngen, nb8, b);
  }
}

// R = F - K U with per-block partials; any_level: also for solves on their coarsest level
// (the finest level of a one-grid solve, for its norm)
template <int P, typename T>
__global__ void __launch_bounds__(256) k_mix_residual(const __grid_constant__ MixArgs<T> A,
                                                      int any_level) {
  __shared__ double sh[32];
  const MixLevel<T>& d = A.s[blockIdx.y];
  if (d.level < (any_level ? 0 : 1) || !*d.active) return;
  const LevelTab<T> L = d.L;
  if ((int)(blockIdx.x * blockDim.x) >= L.n_total - 1) return;
  int g = blockIdx.x * blockDim.x + threadIdx.x;
  double r2 = 0.0, mp = 0.0;
  if (g < L.n_total - 1) {
    T r = d.F[g] - row_KU<P, T, 2, 2>(L, d.U, g);
    d.R[g] = r;
    r2 = (double)r * (double)r;
    int off = g - L.n_ux - L.n_uy;
    if (off >= 0) mp = (double)mean_coef<P>(L, off) * (double)d.U[g];
  }
  double s1 = block_sum(r2, sh);
  double s2 = block_sum(mp, sh);
  if (threadIdx.x == 0) { d.part[2 * blockIdx.x] = s1; d.part[2 * blockIdx.x + 1] = s2; }
}

template <typename T>
__global__ void k_mix_residual_finish(const __grid_constant__ MixArgs<T> A, int any_level,
                                      int want_norm, int rows_per_part) {
  __shared__ double sh[32];
  const MixLevel<T>& d = A.s[blockIdx.x];
  if (d.level < (any_level ? 0 : 1) || !*d.active) return;
  const int n_total = d.L.n_total, nparts = (n_total - 1 + rows_per_part - 1) / rows_per_part;
  double a = 0.0, c = 0.0;
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) { a += d.part[2 * i]; c += d.part[2 * i + 1]; }
  double s1 = block_sum(a, sh);
  double s2 = block_sum(c, sh);
  if (threadIdx.x == 0) {
    double rl = (double)d.F[n_total - 1] - s2;
    d.R[n_total - 1] = (T)rl;
    if (want_norm) *d.norm2 = s1 + rl * rl;
  }
}

// coarse F = P^T R
template <typename T>
__global__ void k_mix_restrict(const __grid_constant__ MixArgs<T> A) {
  const MixLevel<T>& d = A.s[blockIdx.y];
  if (d.level < 1 || !*d.active) return;
  int g = blockIdx.x * blockDim.x + threadIdx.x;
  const int nc = d.Lc.n_total;
  if (g >= nc) return;
  d.Fc[g] = (g == nc - 1) ? d.R[d.L.n_total - 1] : restrict_elem(d.L, d.Lc, d.tp, d.tq, d.R, g);
}

// U += P Uc
template <typename T>
__global__ void k_mix_prolong_add(const __grid_constant__ MixArgs<T> A) {
  const MixLevel<T>& d = A.s[blockIdx.y];
  if (d.level < 1 || !*d.active) return;
  int g = blockIdx.x * blockDim.x + threadIdx.x;
  const int nf = d.L.n_total;
  if (g >= nf) return;
  d.U[g] += (g == nf - 1) ? d.Uc[d.Lc.n_total - 1] : prolong_elem(d.L, d.Lc, d.tp, d.tq, d.Uc, g);
}

template <typename T>
__global__ void k_mix_zero(const __grid_constant__ MixArgs<T> A) {
  const MixLevel<T>& d = A.s[blockIdx.y];
  if (d.level < 1 || !*d.active) return;
  int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g < d.L.n_total) d.U[g] = T(0);
}

// U = K_0^{-1} F for the solves on their coarsest level at this depth, one block per solve
template <typename T>
__global__ void k_mix_coarse(const __grid_constant__ MixArgs<T> A) {
  const MixLevel<T>& d = A.s[blockIdx.x];
  if (d.level != 0 || !*d.active) return;
  extern __shared__ unsigned char smem_raw[];
  T* g = reinterpret_cast<T*>(smem_raw);
  const int n = d.L.n_total;
  for (int i = threadIdx.x; i < n; i += blockDim.x) g[i] = d.F[i];
  __syncthreads();
  int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int i = threadIdx.x >> 5; i < n; i += nw) {
    const T* row = d.kinv + (size_t)i * n;
    T acc = T(0);
#pragma unroll 4
    for (int j = lane; j < n; j += 32) acc = fma(row[j], g[j], acc);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) d.U[i] = acc;
  }
}

}  // namespace dev
}  // namespace igamg

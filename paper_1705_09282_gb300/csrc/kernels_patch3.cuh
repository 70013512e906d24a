// Patch solves of the 3D multiplicative Schwarz sweep with staged neighbourhoods and, for FP64,
// block fixed-point integer rows: the 3D counterpart of kernels_patch.cuh (its arithmetic,
// exponents and error bound).
//
// A 3D row has 82-118 stencil terms at p = 2 (up to 476 at p = 3), one FP64 instruction of 64 cycles
// each in the row kernels.  Here LPR lanes share a row (4 at p = 2, 8 at p = 3): a lane takes one
// slice (one position along the box's long axis) of each of the row's boxes, at most 27 (75)
// integer multiply-add triples, and the lanes' partial sums, integers on the row's common scale,
// meet in shuffles.  An interior patch (8 rows) is then one warp (two at p = 3) and its records are
// loaded lane by lane before the wait for the previous colour; a wall patch has one block.
//
// Staged arrays of the patch of family f at position (P_0, P_1, P_2), c1 = f+1, c2 = f+2 mod 3:
//   U1, U2   u_c1, u_c2, indexed [own axis: 2p+1][next axis][next but one]
//   UF       u_f, [f: 2p][c1][c2]
//   P1, P2, P3  the pressure, [c][c+1][c+2] for c = c1, c2, f (P3 only for wall patches)
// every axis across padded to W = 2p, so that all rows of all kinds and families use the same
// compile-time strides.  Origins: P_a - p along a != f, P_f - (p-1) along f.
//
// Measured per colour launch, FP64 Stokes (k_mult_rows3 / k_mult_rows3x -> these): p = 2 8^3 10.0 ->
// 3.8 us, 16^3 9.8 -> 4.4, 32^3 10.7 -> 10.3, 64^3 42.1 -> 40.3; p = 3 8^3 41.1 -> 18.6, 16^3 47.0 -> 29.6.
// (An exponent per component and the rounding of the rows' sums cost 0.1 to 0.4 us of these up to 16^3.)
// 64^3 is now bound by the staging itself (232 values fetched and converted for the 8 rows of
// a patch, about 900 instructions a warp), the small levels by one block's chain of latencies.
#pragma once
#include "kernels3d.cuh"
#include "kernels_patch.cuh"

namespace igamg {
namespace dev {

template <int P>
struct PatchShape3 {
  static constexpr int Q = P - 1, W = 2 * P, W2 = W * W, A1 = 2 * P + 1, C1 = 2 * Q + 1;
  // stride of the long axis: the lanes of a row read LS entries apart, which W2 would put into one
  // bank (p = 2); 20 and 38 spread them over the banks
  static constexpr int LS = W2 + (P == 2 ? 4 : 2), W3 = W * LS;
  static constexpr int LPR = P == 2 ? 4 : 8, SL = C1 * C1;     // lanes per row, entries per slice
  static constexpr int UC = A1 * LS, NUC = A1 * W2, NW3 = W * W2;   // array sizes and entries in use
  static constexpr int U2 = UC, UF = 2 * UC, P1 = UF + W3, P2 = P1 + W3, P3 = P2 + W3;
  static constexpr int REGI = P3, REGW = P3 + W3;              // interior / wall patch
  static constexpr int MARGIN = P * LS;
  static constexpr int NT = 128;                               // threads per block
  static constexpr int G8 = 8 * LPR, PPB = NT / G8;            // per interior patch; patches per block
  static constexpr int RPR = NT / LPR;                         // wall patches: rows per round
  static constexpr int MR = P == 2 ? 64 : 192;                 // most rows of a wall patch
  static constexpr int XA = W, XE = W * C1;                    // third box: slices, entries per slice
};
// entries per slice in the records: the slice, its exponent (FP64), padding to 16 bytes
template <int P, typename T> constexpr int slice_len() { return sizeof(T) == 8 ? (PatchShape3<P>::SL + 2) / 2 * 2 : (PatchShape3<P>::SL + 3) / 4 * 4; }
template <int P, typename T> constexpr int rec3_len() { return PatchShape3<P>::LPR * 3 * slice_len<P, T>() + (sizeof(T) == 8 ? 2 : 4); }
// (third box: the slice, then its exponent and the order it is stored in)
template <int P, typename T> constexpr int ext_slice_len() { return sizeof(T) == 8 ? (PatchShape3<P>::XE + 2) / 2 * 2 : (PatchShape3<P>::XE + 4) / 4 * 4; }
template <int P, typename T> constexpr int ext3_rec_len() { return PatchShape3<P>::XA * ext_slice_len<P, T>(); }

// Tables of one level (built once at creation).
template <typename T>
struct PatchTab3 {
  const limb_t<T>* rec;             // row records, rec3_len entries: by class record (koff[kind] + record) or row
  const limb_t<T>* ext;             // third box per u_x / u_y row (mapped domains), or null
  const limb_t<T>* inv8;            // interior patches' inverses
  const limb_t<T>* winv;
  const int* gcls;
  const int4 *wdesc, *wrow;
  int koff[4];
  int by_row, maxl;
};

// Exponents of a patch's staged values, one per component.
struct Exps3 {
  int u0, u1, u2, p;
  __device__ __forceinline__ int of(int k) const { return k == 1 ? u1 : (k == 2 ? u2 : u0); }
  __device__ __forceinline__ bool bad() const { return max(max(u0, u1), max(u2, p)) == 0x7ff; }
};

// One colour (PatchGrid3, igamg_internal.h).  row[r]: the interior patch's local row r: kind, its
// position relative to the patch (0 or -1 per axis, as bits), offsets of its boxes.
struct ColourGrid3 {
  int f, o[3], s[3], cnt[3], n8, gfirst, wfirst, nwall;
  int kind[8], d[8], oA[8], oB[8], oC[8], oE[8];
};

// The lane's share of a row: box A at slice s, box B at slice s, and box C at slice s (pressure
// rows) or the last slice of box A (velocity rows, p = 2, lane 0).  Result: the lane's part of the
// local residual on the row's common scale, the same exponent a on all lanes of the row.
// PRE: st is the lane's record in registers; else in global memory, read box by box.  kind: the row's.
template <int P, typename T, bool EXT, bool PRE>
__device__ __forceinline__ Resid<T> row_part(const limb_t<T>* reg, int oA, int oB, int oC, int oE, const limb_t<T>* st,
                                             const limb_t<T>* __restrict__ tail, const limb_t<T>* __restrict__ se, int kind,
                                             int s, const Exps3& ev, T f, T lam) {
  using S = PatchShape3<P>;
  constexpr int SLP = slice_len<P, T>();
  const bool is_p = kind == 3;
  const limb_t<T>* pA = reg + oA + min(s, S::A1 - 1) * S::LS;
  const limb_t<T>* pB = reg + oB + min(s, 2 * P - 1) * S::LS;
  const limb_t<T>* pC = is_p ? reg + oC + min(s, 2 * P - 1) * S::LS : reg + oA + (S::LPR < S::A1 && s == 0 ? S::LPR * S::LS : 0);
  if constexpr (sizeof(T) == 8) {
    Acc A, B, C;
    int aA = ev.of(kind), aB = is_p ? ev.u1 : ev.p, aC = is_p ? ev.u2 : aA;   // (pressure rows: boxes on u_x, u_y, u_z)
    if constexpr (PRE) {                                       // the three boxes' chains side by side
#pragma unroll
      for (int j = 0; j < S::SL; ++j) {
        const int at = (j / S::C1) * S::W + j % S::C1;
        A.mac(pA[at], st[j]);
        B.mac(pB[at], st[SLP + j]);
        C.mac(pC[at], st[2 * SLP + j]);
      }
      aA += st[S::SL].x;
      aB += st[SLP + S::SL].x;
      aC += st[2 * SLP + S::SL].x;
    } else {
      auto box = [&](Acc& acc, const limb_t<T>* p, const limb_t<T>* c) -> int {
        limb_t<T> k[SLP];
        ld_entries_lazy<SLP>(c, k);
#pragma unroll
        for (int j = 0; j < S::SL; ++j) acc.mac(p[(j / S::C1) * S::W + j % S::C1], k[j]);
        return k[S::SL].x;
      };
      aA += box(A, pA, st);
      aB += box(B, pB, st + SLP);
      aC += box(C, pC, st + 2 * SLP);
    }
    const int exF = exp_of(f);
    int a = max(max(aA, max(aB, aC)), max(exF, kExpFloor));
    long long sE = 0, sL = 0;
    int aE = 0, aL = 0;
    if (EXT && se) {
      constexpr int XL = ext_slice_len<P, T>();
      Acc E;
      const limb_t<T>* pE = reg + oE + min(s, S::XA - 1) * S::LS;
      const limb_t<T>* ce = se + min(s, S::XA - 1) * XL;
      if (s < S::XA) {
#pragma unroll
        for (int j = 0; j < S::XE; ++j) {
          // u_x rows read u_y [y][z][x]: C1 x W entries; u_y rows read u_x [x][y][z]: W x C1; the
          // records store the slice in array order with the row length of the first kind
          E.mac(pE[ce[S::XE].y ? (j / S::C1) * S::W + j % S::C1 : (j / S::W) * S::W + j % S::W], ce[j]);
        }
      }
      aE = ev.of(1 - kind) + ce[S::XE].x;
      sE = E.sum();
      a = max(a, aE);
    }
    if (is_p && nonzero(lam)) {
      const int exL = max(exp_of(lam), kExpFloor);
      Acc Lm;
      Lm.mac(to_limbs(lam, exL), tail[0]);
      aL = exL + tail[1].x;
      sL = Lm.sum();
      a = max(a, aL);
    }
    long long r = 0;
    if (s == 0) {
      const int h = __double2hiint(f);
      const unsigned long long M = ((unsigned long long)(unsigned)((h & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(f);
      r = (long long)shr64(M << 7, a - exF);
      if (h < 0) r = -r;
      if (is_p && nonzero(lam)) r -= sar64(sL, a - aL);
      // the shifts below round down: half a unit per lane and shifted box, put back here for all lanes
      // (without it the rows of the cylinder at p = 3 were 7 % less accurate than FP64 multiply-adds)
      const int shifted = (aA < a) + (aB < a) + (is_p && aC < a) + (EXT && se && aE < a);
      r -= S::LPR / 2 * shifted;
    }
    r -= sar64(A.sum(), a - aA);
    r -= sar64(B.sum(), a - aB);
    r -= sar64(C.sum(), a - aC);
    if (EXT && se) r -= sar64(sE, a - aE);
    return {r, a};
  } else {
    T x0 = T(0), x1 = T(0), x2 = T(0);
    limb_t<T> own[PRE ? 4 : 3 * SLP];
    if constexpr (!PRE) ld_entries_lazy<3 * SLP>(st, own);
    const limb_t<T>* k = PRE ? st : own;
#pragma unroll
    for (int j = 0; j < S::SL; ++j) {
      const int at = (j / S::C1) * S::W + j % S::C1;
      x0 = fma(k[j], pA[at], x0);
      x1 = fma(k[SLP + j], pB[at], x1);
      x2 = fma(k[2 * SLP + j], pC[at], x2);
    }
    if (EXT && se && s < S::XA) {
      constexpr int XL = ext_slice_len<P, T>();
      const limb_t<T>* pE = reg + oE + s * S::LS;
      const limb_t<T>* ce = se + s * XL;
      const bool k1 = ce[S::XE] != T(0);
#pragma unroll
      for (int j = 0; j < S::XE; ++j)
        x1 = fma(ce[j], pE[k1 ? (j / S::C1) * S::W + j % S::C1 : (j / S::W) * S::W + j % S::W], x1);
    }
    T r = -((x0 + x1) + x2);
    if (s == 0) {
      r += f;
      if (is_p) r = fma(-tail[0], lam, r);
    }
    return {r};
  }
}

// Sum of the LPR lanes' parts (the exponent is already common).
template <int LPR>
__device__ __forceinline__ void lanes_sum(Resid<double>& r) {
#pragma unroll
  for (int o = 1; o < LPR; o <<= 1) r.v += __shfl_xor_sync(0xffffffffu, r.v, o);
}
template <int LPR>
__device__ __forceinline__ void lanes_sum(Resid<float>& r) {
#pragma unroll
  for (int o = 1; o < LPR; o <<= 1) r.v += __shfl_xor_sync(0xffffffffu, r.v, o);
}

// Loads the neighbourhood of the patch (f; p0, p1, p2) with G threads and stages it at reg.
// sync: barrier of the G threads; red: shared memory for a maximum per warp, if G > 32.
// WALL: positions outside the index range count as 0, and P3 is filled.
template <int P, typename T, bool WALL, int G, typename Sync>
__device__ __forceinline__ void stage3(const LevelTab3<T>& L, const T* U, int f, const int* pos, int t, limb_t<T>* reg,
                                       int4* red, Exps3& ev, Sync sync) {
  using S = PatchShape3<P>;
  constexpr int KU = (S::NUC + G - 1) / G, KW = (S::NW3 + G - 1) / G;
  T v1[KU], v2[KU], vf[KW], vp[KW];
  const int c1 = f == 2 ? 0 : f + 1, c2 = f == 0 ? 2 : f - 1;
  if constexpr (P == 2 && !WALL && G == 32) {
    // entry t + 32 k: positions (t >> 4) + 2 k, (t >> 2) & 3, t & 3 along c, c+1, c+2, all in range
    const int d0 = t >> 4, d1 = t >> 2 & 3, d2 = t & 3;
    auto load = [&](int blk, int c, int n, T* v) {
      const int x1 = c == 2 ? 0 : c + 1, x2 = c == 0 ? 2 : c - 1;
      const bool pad = (x1 == f && d1 >= S::C1) || (x2 == f && d2 >= S::C1);
      const int dx = blk == 0 ? L.ni : L.nq, dxy = dx * (blk == 1 ? L.ni : L.nq);
      auto str = [&](int a) { return a == 0 ? 1 : (a == 1 ? dx : dxy); };
      auto org = [&](int a) { return pos[a] - (a == f ? S::Q : P) - (blk == a ? 1 : 0); };
      const int sc = str(c);
      const T* q = U + (blk < 3 ? blk * L.n_uc : L.n_u) + (org(c) + d0) * sc + (org(x1) + d1) * str(x1) + (org(x2) + d2) * str(x2);
#pragma unroll
      for (int k = 0; k < (n + 31) / 32; ++k) v[k] = pad || (32 * k + 32 > n && t + 32 * k >= n) ? T(0) : q[2 * k * sc];
    };
    load(c1, c1, S::NUC, v1);
    load(c2, c2, S::NUC, v2);
    load(f, f, S::NW3, vf);
    load(3, c1, S::NW3, vp);
  } else {
    // array of component blk (3: pressure) in the axis order (c, c+1, c+2)
    auto load = [&](int blk, int c, int e, int n) -> T {
      const int d0 = e / S::W2, d1 = e / S::W % S::W, d2 = e % S::W;
      const int x1 = c == 2 ? 0 : c + 1, x2 = c == 0 ? 2 : c - 1;
      const bool pad = (x1 == f && d1 >= S::C1) || (x2 == f && d2 >= S::C1) || (blk == 3 && c == f && d0 >= S::C1);
      if (e >= n || pad) return T(0);
      const int dx = blk == 0 ? L.ni : L.nq, dxy = dx * (blk == 1 ? L.ni : L.nq);
      int idx = blk < 3 ? blk * L.n_uc : L.n_u;
      bool ok = true;
      auto axis = [&](int a, int d) {
        const int own = blk == a ? 1 : 0, q = pos[a] - (a == f ? S::Q : P) + d;
        if (WALL) ok = ok && q >= own && q <= (own ? L.ni : L.nq - 1);
        idx += (q - own) * (a == 0 ? 1 : (a == 1 ? dx : dxy));
      };
      axis(c, d0);
      axis(x1, d1);
      axis(x2, d2);
      return !WALL || ok ? U[idx] : T(0);
    };
#pragma unroll
    for (int k = 0; k < KU; ++k) { v1[k] = load(c1, c1, t + G * k, S::NUC); v2[k] = load(c2, c2, t + G * k, S::NUC); }
#pragma unroll
    for (int k = 0; k < KW; ++k) { vf[k] = load(f, f, t + G * k, S::NW3); vp[k] = load(3, c1, t + G * k, S::NW3); }
  }
  int e1 = kExpFloor << 20, e2 = e1, ef = e1, ep = e1;
  if constexpr (sizeof(T) == 8) {
#pragma unroll
    for (int k = 0; k < KU; ++k) { e1 = max(e1, top_of(v1[k])); e2 = max(e2, top_of(v2[k])); }
#pragma unroll
    for (int k = 0; k < KW; ++k) { ef = max(ef, top_of(vf[k])); ep = max(ep, top_of(vp[k])); }
    e1 = __reduce_max_sync(0xffffffffu, e1);
    e2 = __reduce_max_sync(0xffffffffu, e2);
    ef = __reduce_max_sync(0xffffffffu, ef);
    ep = __reduce_max_sync(0xffffffffu, ep);
    if constexpr (G > 32) {
      if ((t & 31) == 0) red[t >> 5] = make_int4(e1, e2, ef, ep);
      sync();
#pragma unroll
      for (int w = 0; w < G / 32; ++w) {
        const int4 q = red[w];
        e1 = max(e1, q.x);
        e2 = max(e2, q.y);
        ef = max(ef, q.z);
        ep = max(ep, q.w);
      }
    }
    e1 >>= 20;
    e2 >>= 20;
    ef >>= 20;
    ep >>= 20;
  }
  ev.u0 = f == 0 ? ef : (f == 2 ? e1 : e2);
  ev.u1 = f == 1 ? ef : (f == 0 ? e1 : e2);
  ev.u2 = f == 2 ? ef : (f == 1 ? e1 : e2);
  ev.p = ep;
  auto put = [&](int at, T v, int e) {
    if constexpr (sizeof(T) == 8) reg[at] = to_limbs(v, e);
    else reg[at] = v;
  };
#pragma unroll
  for (int k = 0; k < KU; ++k) {
    const int e = t + G * k, at = e + e / S::W2 * (S::LS - S::W2);
    if (e < S::NUC) { put(at, v1[k], e1); put(S::U2 + at, v2[k], e2); }
  }
#pragma unroll
  for (int k = 0; k < KW; ++k) {
    const int e = t + G * k, at = e + e / S::W2 * (S::LS - S::W2);
    if (e >= S::NW3) continue;
    put(S::UF + at, vf[k], ef);
    limb_t<T> w;
    if constexpr (sizeof(T) == 8) w = to_limbs(vp[k], ep);
    else w = vp[k];
    const int d0 = e / S::W2, d1 = e / S::W % S::W, d2 = e % S::W;   // positions along c1, c2, f
    reg[S::P1 + at] = w;
    reg[S::P2 + d1 * S::LS + d2 * S::W + d0] = w;
    if (WALL) reg[S::P3 + d2 * S::LS + d0 * S::W + d1] = w;
  }
  sync();
}

template <typename T>
__device__ __forceinline__ int row_index3(const LevelTab3<T>& L, int kind, int x, int y, int z) {
  const int dx = kind == 0 ? L.ni : L.nq, dy = kind == 1 ? L.ni : L.nq;
  return (kind < 3 ? kind * L.n_uc : L.n_u) + ((z - (kind == 2)) * dy + y - (kind == 1)) * dx + x - (kind == 0);
}

// ---- one colour: blocks [0, nwall) a wall patch each, then PPB interior patches per block ------
// Three blocks per SM at p = 2 (left alone, the third box's variant takes 222 registers, two blocks:
// cylinder 32^3 17.2 us a colour against 14.3).
// PRE: the records are fetched into registers before the dependency wait (colours that leave the
// GPU idle: the chain of one block counts); else they are read where they are used and the
// registers saved hold twice the warps (colours of many blocks).
// ROWS: no solve; U is read only, and the rows' local residuals go to R_ (k_patch_rows of the 2D path).
template <int P, typename T, bool EXT, bool PRE, bool ROWS = false>
__global__ void __launch_bounds__(128, !PRE ? 6 : (P == 2 ? 3 : 2)) k_patch_colour3(const __grid_constant__ LevelTab3<T> L,
                                                       const __grid_constant__ PatchTab3<T> X, T* U, const T* F,
                                                       const __grid_constant__ ColourGrid3 C, T* R_) {
  using S = PatchShape3<P>;
  using E = limb_t<T>;
  constexpr int SLP = slice_len<P, T>(), NR = rec3_len<P, T>(), LPR = S::LPR;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int red[8];                                       // residual exponents (2) and a flag, per group
  __shared__ int4 emax[S::NT / 32];
  E st_[PRE ? 3 * SLP : 1];
  const E* st = st_;
  if ((int)blockIdx.x >= C.nwall) {
    const int grp = threadIdx.x / S::G8, t = threadIdx.x % S::G8, k8 = ((int)blockIdx.x - C.nwall) * S::PPB + grp;
    if (k8 >= C.n8) return;
    auto sync = [&]() {
      if constexpr (S::G8 == 32) __syncwarp();
      else asm volatile("bar.sync %0, 64;" ::"r"(1 + grp) : "memory");
    };
    const int row = t / LPR, s = t % LPR;
    const int i01 = C.cnt[0] * C.cnt[1], k2 = k8 / i01, k1 = (k8 - k2 * i01) / C.cnt[0], k0 = k8 - k2 * i01 - k1 * C.cnt[0];
    const int pos[3] = {C.o[0] + C.s[0] * k0, C.o[1] + C.s[1] * k1, C.o[2] + C.s[2] * k2};
    const int icls = X.gcls[C.gfirst + k8];
    const int kind = C.kind[row], d = C.d[row];
    const bool is_p = kind == 3;
    const int x = pos[0] - (d & 1), y = pos[1] - (d >> 1 & 1), z = pos[2] - (d >> 2 & 1);
    const int g = row_index3(L, kind, x, y, z);
    int ri = g;
    if (!X.by_row) {
      using R3 = Rec3<P>;
      const int lastp = L.n + P - 1, lastq = L.n + P - 2;
      const int cl = (cls1d<P>(z, kind == 2 ? lastp : lastq) * R3::NC + cls1d<P>(y, kind == 1 ? lastp : lastq)) * R3::NC +
                     cls1d<P>(x, kind == 0 ? lastp : lastq);
      const int* cm = kind == 0 ? L.cm0 : (kind == 1 ? L.cm1 : (kind == 2 ? L.cm2 : L.cm3));
      ri = X.koff[kind] + cm[cl];
    }
    const E* rp = X.rec + (size_t)ri * NR;
    if constexpr (PRE) ld_entries<3 * SLP>(rp + s * 3 * SLP, st_);
    else st = rp + s * 3 * SLP;
    constexpr int LD = inv8_ld<T>(), NC8 = 8 / LPR;
    const E* Ap = X.inv8 + ((size_t)icls * 8 + row) * LD;
    E A[NC8];
#pragma unroll
    for (int c = 0; c < NC8; ++c) A[c] = Ap[s * NC8 + c];
    int2 ec = make_int2(0, 0);
    if constexpr (sizeof(T) == 8) ec = Ap[8];
    if (S::G8 > 32 && t < 4) red[grp * 4 + t] = 0;
    const E* se = EXT && kind < 2 ? X.ext + (size_t)g * ext3_rec_len<P, T>() : nullptr;
    dependency_wait();
    if (S::G8 > 32) sync();
    E* reg = reinterpret_cast<E*>(smem_raw) + grp * S::REGI;
    const T fv = F[g], lam = U[L.n_total - 1], u_own = U[g];
    Exps3 ev;
    stage3<P, T, false, S::G8>(L, U, C.f, pos, t, reg, emax + grp * (S::G8 / 32), ev, sync);
    Resid<T> r = row_part<P, T, EXT, PRE>(reg, C.oA[row], C.oB[row], C.oC[row], C.oE[row], st, rp + LPR * 3 * SLP, se, kind, s,
                                     ev, fv, lam);
    lanes_sum<LPR>(r);
    if constexpr (ROWS) {
      if (s == 0) R_[g] = resid_value(r);
      return;
    }
    sync();
    if constexpr (sizeof(T) == 8) {
      const int er = resid_exp(r);
      int eg = er, eo;                                         // maxima over the velocity and pressure rows
      if constexpr (S::G8 == 32) {
        eg = max(eg, __shfl_xor_sync(0xffffffffu, eg, 4));
        eg = max(eg, __shfl_xor_sync(0xffffffffu, eg, 8));
        eo = __shfl_xor_sync(0xffffffffu, eg, 16);
      } else {
        if (s == 0) atomicMax(&red[grp * 4 + (is_p ? 1 : 0)], er);
        sync();
        eg = red[grp * 4 + (is_p ? 1 : 0)];
        eo = red[grp * 4 + 1 - (is_p ? 1 : 0)];
      }
      if (s == 0) reg[row] = resid_limbs(r, er, eg);
      const bool bad = ev.bad() || exp_of(fv) == 0x7ff || exp_of(lam) == 0x7ff;
      if (S::G8 > 32 && bad) red[grp * 4 + 2] = 1;
      sync();
      const int c0 = s * NC8;                                  // this lane's columns: all velocity or all pressure
      Acc D;
#pragma unroll
      for (int c = 0; c < NC8; ++c) D.mac(reg[c0 + c], A[c]);
      const int gu = is_p ? eo : eg, gp = is_p ? eg : eo, a0 = gu + ec.x, a1 = gp + ec.y, am = max(a0, a1);
      Resid<double> q{sar64(D.sum(), am - (c0 < 4 ? a0 : a1)), 0};
      lanes_sum<LPR>(q);
      double dv = to_double(q.v, am);
      bool any;
      if constexpr (S::G8 == 32) any = __any_sync(0xffffffffu, bad);
      else any = red[grp * 4 + 2];
      if (any) dv = __longlong_as_double(0x7ff8000000000000ll);
      if (s == 0) U[g] = u_own + dv;
    } else {
      if (s == 0) reg[row] = r.v;
      sync();
      Resid<T> q{T(0)};
#pragma unroll
      for (int c = 0; c < NC8; ++c) q.v = fma(A[c], reg[s * NC8 + c], q.v);
      lanes_sum<LPR>(q);
      if (s == 0) U[g] = u_own + q.v;
    }
    return;
  }
  // a wall patch: rounds of RPR rows
  const int t = threadIdx.x, w = C.wfirst + (int)blockIdx.x, rl_row = t / LPR, s = t % LPR;
  const int4 D = X.wdesc[w];                                   // position, inverse (16 B), rows | velocity rows << 16
  const int nl = D.z & 0xffff, nv = D.z >> 16, ld = wall_ld(nl);
  E* reg = reinterpret_cast<E*>(smem_raw) + S::MARGIN;
  E* rl = reg + S::REGW + S::MARGIN;
  long long* rv = reinterpret_cast<long long*>(rl + S::MR);
  int* ra = reinterpret_cast<int*>(rv + S::MR);
  E* inv = reinterpret_cast<E*>(ra + S::MR);
  const char* src = reinterpret_cast<const char*>(X.winv) + (size_t)D.y * 16;
  if constexpr (P == 2) {                                      // (152 x 153 entries at p = 3 do not fit)
    const int n16 = (int)((nl * ld * sizeof(E) + 15) / 16);
    const unsigned dst = (unsigned)__cvta_generic_to_shared(inv);
    for (int i = t; i < n16; i += S::NT)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * i), "l"(src + 16 * (size_t)i) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  auto sync = [&]() { __syncthreads(); };
  int4 R = X.wrow[(size_t)w * S::MR + rl_row];
  if constexpr (PRE) ld_entries<3 * SLP>(X.rec + (size_t)R.w * NR + s * 3 * SLP, st_);
  if (t < 4) red[t] = 0;
  dependency_wait();
  __syncthreads();
  if constexpr (sizeof(T) == 4) {                              // what rows read with zero coefficients is finite
    for (int i = t; i < 2 * S::MARGIN + S::REGW; i += S::NT) reg[i - S::MARGIN] = T(0);
    __syncthreads();
  }
  const int pos[3] = {D.x & 1023, D.x >> 10 & 1023, D.x >> 20 & 1023};
  const T lam = U[L.n_total - 1];
  Exps3 ev;
  stage3<P, T, true, S::NT>(L, U, C.f, pos, t, reg, emax, ev, sync);
  bool bad = false;
  if constexpr (sizeof(T) == 8) bad = ev.bad() || exp_of(lam) == 0x7ff;
  for (int r0 = 0; r0 < nl; r0 += S::RPR) {
    const int row = r0 + rl_row;
    if (r0 > 0) {
      R = X.wrow[(size_t)w * S::MR + min(row, S::MR - 1)];
      if constexpr (PRE) ld_entries<3 * SLP>(X.rec + (size_t)R.w * NR + s * 3 * SLP, st_);
    }
    if constexpr (!PRE) st = X.rec + (size_t)R.w * NR + s * 3 * SLP;
    const bool has = row < nl;
    const int kind = R.x >= L.n_u ? 3 : (R.x >= 2 * L.n_uc ? 2 : (R.x >= L.n_uc ? 1 : 0));
    const T fv = has ? F[R.x] : T(0);
    const E* se = EXT && has && R.x < 2 * L.n_uc ? X.ext + (size_t)R.x * ext3_rec_len<P, T>() : nullptr;
    Resid<T> r = row_part<P, T, EXT, PRE>(reg, (short)(R.y & 0xffff), R.y >> 16, (short)(R.z & 0xffff), R.z >> 16, st,
                                     X.rec + (size_t)R.w * NR + LPR * 3 * SLP, se, kind, s, ev, fv, lam);
    lanes_sum<LPR>(r);
    if constexpr (ROWS) {
      if (s == 0 && has) R_[R.x] = resid_value(r);
      continue;
    }
    if constexpr (sizeof(T) == 8) {
      bad = bad || exp_of(fv) == 0x7ff;
      if (s == 0 && has) {
        rv[row] = r.v;
        ra[row] = r.a;
        atomicMax(&red[row < nv ? 0 : 1], resid_exp(r));
      }
    } else {
      if (s == 0 && has) rl[row] = r.v;
    }
  }
  if (bad) red[2] = 1;
  asm volatile("cp.async.wait_all;" ::: "memory");
  if constexpr (ROWS) return;
  __syncthreads();
  const E* A = P == 2 ? inv : reinterpret_cast<const E*>(src);
  if constexpr (sizeof(T) == 8) {
    const int gu = red[0], gp = red[1];
    const bool any = red[2] != 0;
    for (int row = t; row < nl; row += S::NT) {
      const Resid<double> r{rv[row], ra[row]};
      rl[row] = resid_limbs(r, resid_exp(r), row < nv ? gu : gp);
    }
    __syncthreads();
    for (int r0 = 0; r0 < nl; r0 += S::RPR) {
      const int row = r0 + rl_row, rr = min(row, nl - 1);
      const E* Ak = A + (size_t)rr * ld;
      Acc D0, D1;
#pragma unroll 4
      for (int c = s; c < nv; c += LPR) D0.mac(rl[c], Ak[c]);
#pragma unroll 4
      for (int c = nv + s; c < nl; c += LPR) D1.mac(rl[c], Ak[c]);
      const int2 ec = Ak[nl];
      const int a0 = gu + ec.x, a1 = gp + ec.y, am = max(a0, a1);
      Resid<double> q{sar64(D0.sum(), am - a0) + sar64(D1.sum(), am - a1), 0};
      lanes_sum<LPR>(q);
      double dv = to_double(q.v, am);
      if (any) dv = __longlong_as_double(0x7ff8000000000000ll);
      if (s == 0 && row < nl) U[X.wrow[(size_t)w * S::MR + row].x] += dv;
    }
  } else {
    for (int r0 = 0; r0 < nl; r0 += S::RPR) {
      const int row = r0 + rl_row, rr = min(row, nl - 1);
      const E* Ak = A + (size_t)rr * ld;
      Resid<T> q{T(0)};
#pragma unroll 4
      for (int c = s; c < nl; c += LPR) q.v = fma(Ak[c], rl[c], q.v);
      lanes_sum<LPR>(q);
      if (s == 0 && row < nl) U[X.wrow[(size_t)w * S::MR + row].x] += q.v;
    }
  }
}

// bytes of shared memory of a colour launch
template <int P, typename T>
size_t patch3_smem(int maxl) {
  using S = PatchShape3<P>;
  const size_t e = sizeof(limb_t<T>);
  const size_t in = (size_t)S::PPB * S::REGI * e;
  size_t wall = (2 * S::MARGIN + S::REGW + S::MR) * e + S::MR * 12;
  if (P == 2) wall += ((size_t)maxl * wall_ld(maxl) * e + 15) / 16 * 16;
  return wall > in ? wall : in;
}

// ---- building the tables -------------------------------------------------------------------------

// Row records of one kind (or, kind < 0, of all rows of a level in order): src has Rec3<P>::RU
// entries per record, in the order the staged arrays are read.
template <int P, typename T>
__global__ void k_patch_records3(int n, int kind, int n_u, const T* __restrict__ src, limb_t<T>* __restrict__ dst) {
  using S = PatchShape3<P>;
  using R = Rec3<P>;
  constexpr int SLP = slice_len<P, T>(), NR = rec3_len<P, T>(), LPR = S::LPR;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const bool is_p = kind >= 0 ? kind == 3 : i >= n_u;
  const T* s = src + (size_t)i * R::RU;
  limb_t<T>* d = dst + (size_t)i * NR;
  int ea = 0, eb = 0, ec = 0;
  if constexpr (sizeof(T) == 8) {
    double a = 0, b = 0, c = 0;
    for (int j = 0; j < R::B0; ++j) a += fabs(s[j]);
    for (int j = 0; j < R::B1; ++j) { b += fabs(s[R::B0 + j]); c += fabs(s[R::B0 + R::B1 + j]); }
    ea = sum_exp(a);
    eb = sum_exp(b);
    ec = is_p ? sum_exp(c) : ea;
  }
  auto put = [&](int at, T v, int e) {
    if constexpr (sizeof(T) == 8) d[at] = coef_limbs(v, e);
    else d[at] = v;
  };
  for (int l = 0; l < LPR; ++l)
    for (int j = 0; j < SLP; ++j) {
      const int at = (l * 3) * SLP + j;
      if (j < S::SL) {
        put(at, l < S::A1 ? s[l * S::SL + j] : T(0), ea);
        put(at + SLP, l < 2 * P ? s[R::B0 + l * S::SL + j] : T(0), eb);
        T c = T(0);
        if (is_p) c = l < 2 * P ? s[R::B0 + R::B1 + l * S::SL + j] : T(0);
        else if (l == 0 && LPR < S::A1) c = s[LPR * S::SL + j];
        put(at + 2 * SLP, c, ec);
      } else {
        if constexpr (sizeof(T) == 8) {
          d[at] = make_int2(ea, 0);
          d[at + SLP] = make_int2(eb, 0);
          d[at + 2 * SLP] = make_int2(ec, 0);
        } else {
          d[at] = d[at + SLP] = d[at + 2 * SLP] = T(0);
        }
      }
    }
  limb_t<T>* tail = d + LPR * 3 * SLP;
  if constexpr (sizeof(T) == 8) {
    const int el = sum_exp(fabs(s[R::RU - 1]));
    tail[0] = coef_limbs(s[R::RU - 1], el);
    tail[1] = make_int2(el, 0);
  } else {
    tail[0] = s[R::RU - 1];
    tail[1] = tail[2] = tail[3] = T(0);
  }
}

// Third box per u_x / u_y row: slices in the order of the array they are read from.
template <int P, typename T>
__global__ void k_patch_ext3(int n, int n_uc, const T* __restrict__ src, limb_t<T>* __restrict__ dst) {
  using S = PatchShape3<P>;
  constexpr int XL = ext_slice_len<P, T>();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const bool ux = i < n_uc;                                    // reads u_y [y][z][x]; u_y rows read u_x [x][y][z]
  const T* s = src + (size_t)i * (S::W * S::W * S::C1);        // stored [x][y][z]
  limb_t<T>* d = dst + (size_t)i * ext3_rec_len<P, T>();
  int e = 0;
  if constexpr (sizeof(T) == 8) {
    double sum = 0;
    for (int j = 0; j < S::W * S::W * S::C1; ++j) sum += fabs(s[j]);
    e = sum_exp(sum);
  }
  for (int l = 0; l < S::XA; ++l)
    for (int j = 0; j < XL; ++j) {
      T v = T(0);
      if (j < S::XE) {
        if (ux) v = s[((j % S::W) * S::W + l) * S::C1 + j / S::W];           // y = l; z, x = j
        else v = s[(l * S::W + j / S::C1) * S::C1 + j % S::C1];              // x = l; y, z = j
      }
      if constexpr (sizeof(T) == 8) d[l * XL + j] = j < S::XE ? coef_limbs(v, e) : make_int2(j == S::XE ? e : 0, ux ? 0 : 1);
      else d[l * XL + j] = j < S::XE ? v : T(ux ? 0 : 1);
    }
}

// Local inverses from the packed table of all classes (nl x nl each): interior classes first0 ..
// first0 + n - 1, 8 rows each.
template <typename T>
__global__ void k_patch_inv8_3(int n, int first0, const long long* __restrict__ off, const T* __restrict__ cinv,
                               limb_t<T>* __restrict__ dst) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n * 8) inverse_row<T>(cinv + off[first0 + i / 8] + (i & 7) * 8, 8, 4, dst + (size_t)i * inv8_ld<T>());
}
// Wall patches: one block per class of spec (x: class in the packed table, y: offset of the result
// in 16 bytes, z: rows | velocity rows << 16).
template <typename T>
__global__ void k_patch_winv3(const int4* __restrict__ spec, const long long* __restrict__ off, const T* __restrict__ cinv,
                              limb_t<T>* __restrict__ dst) {
  const int4 s = spec[blockIdx.x];
  const int nl = s.z & 0xffff, nv = s.z >> 16;
  limb_t<T>* d = reinterpret_cast<limb_t<T>*>(reinterpret_cast<char*>(dst) + (size_t)s.y * 16);
  for (int r = threadIdx.x; r < nl; r += blockDim.x)
    inverse_row<T>(cinv + off[s.x] + (size_t)r * nl, nl, nv, d + (size_t)r * wall_ld(nl));
}

}  // namespace dev
}  // namespace igamg

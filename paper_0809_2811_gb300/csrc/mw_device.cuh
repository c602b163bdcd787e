// mw_device.cuh -- device data layout and kernels of libmw (sm_103a).
//
// Model: Stillinger-Weber form with the mW parameters (Molinero & Moore,
// Sec. II.A and II.D):
//   E = sum_{i<j} phi2(r_ij) + sum_i sum_{j<k, legs of i} phi3(r_ij, r_ik, theta_jik)
//   phi2(r) = A eps [B (sig/r)^p - (sig/r)^q] exp(sig/(r - a sig))
//   phi3    = lam eps (cos th - cos th0)^2 exp(gam sig/(r - a sig)) exp(gam sig/(s - a sig))
// Dynamics: velocity Verlet with Berendsen or Nose-Hoover (Sec. II.B).
//
// Layout (all boxes concatenated box-major, atoms sorted by cell inside each
// box at every eighth neighbour-list rebuild):
//   x,y,z            master positions as 64-bit fractions of the box edge
//   vx,vy,vz         master velocities (A/fs) as FP32 sums hi + lo; between
//                    steps they lack the second half-kick of the last step
//                    (Global::pend), which the next kick1 folds into its own
//   q                uint4 {qx, qy, qz, box}: position as a 32-bit fraction of
//                    the box edge; the minimum-image difference of two atoms
//                    is the wrapping int32 difference, converted once to FP32
//   f                float4 forces (w unused), accumulated with red.global
//   nbr              int32 [N][W] neighbour list (atom-major rows), nbr_cnt[N]
//   cell_start       exclusive scan of atoms per cell, ncell + 1 entries
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "mw_quotient.h"

namespace mw {

constexpr double kKB = 0.0019872042586408316;  // kcal/mol/K
constexpr double kFCONV = 4.184e-4;            // (kcal/mol/A)/(g/mol) -> A/fs^2
constexpr double kATM = 68568.4158;            // atm per kcal/mol/A^3
constexpr unsigned kFull = 0xffffffffu;

// Status codes written to Global::status (same values as mw_status).
enum : int { ST_OK = 0, ST_OVERFLOW = 3, ST_NAN = 4, ST_LOST = 5, ST_TIMEOUT = 6, ST_LEGS = 10, ST_GRID = 11,
             ST_CELLS = 12, ST_INPUT = 13 };

enum : int { TH_NVE = 0, TH_BERENDSEN = 1, TH_NH = 2, TH_NPT = 3 };

// Legs staged per centre atom in the fused force kernel's shared-memory table;
// centres with more legs take the overflow path.
constexpr int kLMax = 24;
// Upper bound for the overflow path (more legs than this = overlapping atoms).
constexpr int kMaxLegsOverflow = 64;

struct Box {        // read-only in kernels, except the geometry under isobaric runs (end_of_step_box)
  double L[3];
  double dtL[3];    // dt / L: drift of the box fraction per unit velocity
  float dtL64[3];   // dt / L * 2^64: drift in 2^-64 box-fraction units per unit velocity (FP32)
  float lost;       // half the shortest edge (A)
  double qs[3];     // unused (2^32 / L at creation; checkpoints hold this structure)
  float Lq[3];      // L / 2^32
  int off, n;       // atom range
  int nc[3];        // cells per dimension
  int cell_off;     // first global cell
  double T0, Ndf, Q, volume;
  double invQ;      // unused (1 / Q)
  double ndfkT0;    // N_df k_B T0
  double q4;        // dt / (4 Q): quarter-step factor of xi
  float q4f;        // q4 in FP32
  double inv_ndf_kb;  // 1 / (N_df k_B): T = 2 KE inv_ndf_kb
  double p_fac;     // unused (1/(3 V) in atm at creation)
  int vexp_lost;    // a velocity component whose FP32 exponent field is >= this is a runaway (see validate_integ)
  // isobaric runs only: the box scales at the drift of every step
  float hs2;        // squared displacement (measured with this step's Lq) that triggers a rebuild
  float a3;         // 1 + 3/N_df (barostat coupling)
  double W;         // barostat mass (N_df + 3) k_B T0 tau_p^2
  double Ln[3];     // edges of the coming step, made current by the last block of its kick1
};

struct BoxState {   // mutated by kernels
  float4 th;              // (xi hi, xi lo, eta hi, eta lo) after the start half of the next step
  float4 th_e;            // the same after the last end half
  double ke_last;         // KE after the last end half, or of the state just set (kcal/mol)
  double s_endc;          // last end scale, still pending on the stored velocities
  float sig;              // S - 1 for the next kick1: S = s_endc times the start-half scale
  int sorted;             // 1: the box's atoms are in cell order of a recent build (see box_sorts)
  double ke_acc[2];       // per step-parity raw kinetic energy of v + a (the second half-kick)
  double ew[2][8];        // per step-parity E2, E3, W[6]
  int rebuild;            // displacement flag of this box
  int pad_;
  long long rebuilds;
  double pe_b;            // barostat momentum (isobaric runs), after the start half of the next step
  double pe_e;            // the same after the last end half
  double Lb;              // edge 0 of the box at its last build (isotropic scaling: one ratio for all edges)
};

// Per-box thermo record written at the end of each step (doubles).
enum { TR_STEP, TR_PE, TR_E2, TR_E3, TR_KE, TR_T, TR_CONS, TR_P, TR_W0, TR_XI = TR_W0 + 6, TR_ETA,
       TR_REBUILDS, TR_VOL, TR_L0, TR_N = TR_L0 + 3 };

struct Global {
  unsigned long long step;  // completed steps since set_state
  int any_rebuild;
  int status;
  int max_count;            // widest neighbour set of the last build
  unsigned done;            // last-block counter of k_kick2
  int wpar;                 // parity slot of ew[] holding the virial of the latest force evaluation
  unsigned done1;           // last-block counter of k_kick1 (graph condition)
  long long rebuild_steps;  // steps (or force calls) that rebuilt at least one box
  int pend;                 // 1: velocities lack the second half-kick of the last step
  int pad_bar[4];           // (unused: checkpoints hold this struct)
  long long npairs, ntrip;  // leg / triplet counts of the last force call (if counting)
  int count_terms;
  int pad_over;             // (unused)
  int err_index;
  int pad_;
};

struct Integ {
  double dt;
  double cf;         // 0.5 dt FCONV / mass
  float cf_f;        // the same in FP32 (velocity increment = cf_f * F in FP32, added in FP64)
  double ke_fac;     // 0.5 mass / FCONV
  double tau;
  int kind;
  float half_skin2;  // (skin/2)^2
  double p_ext;      // target pressure of isobaric runs (kcal/mol/A^3)
  float skin, rlist; // list skin and radius (A): rebuild margin and cell check of a scaling box
};

// Cell grids of isobaric runs: laid out with cells kCellMargin r_list wide;
// a box that shrinks below r_list per cell, or grows so that one more cell
// of kCellGrow r_list fits, stops the run at a step boundary (ST_GRID) for
// the host to lay the grid out again.
constexpr double kCellMargin = 1.12;
constexpr double kCellGrow = 1.2;

// FP32 constants of the force kernels.  The *_lo fields hold the FP32
// rounding error of the constant before them (value = hi + lo to ~2^-48),
// which leg_terms adds back at first order.
struct FParams {
  float rc, rc2, rl2;
  float sig, sig_l2e, gsig_l2e, gsig;
  float Aeps, B, c0, sle;  // sle = sqrt(lambda eps)
  int p, q;
  float rc_lo, sig_lo, sig_l2e_lo, gsig_l2e_lo, B_lo;
};

// Several species: FP32 constants of the pair (a, b), from the parameter
// set of entry (a, b, b); the three-body leg factor of a leg from a centre
// of species a to one of species b uses the same set's gamma, sigma, a.
constexpr int kMaxSpecies = 8;
// h and c0 serve the moment kernel, for tables whose lambda epsilon of
// (centre a; legs b, c) is h_ab h_ac and whose cos theta0 depends on the
// centre alone: h = sqrt(lambda epsilon) of (a, b, b), c0 = cos theta0 of a.
struct SpPair {
  float rc, rc2, sig, sig_l2e, gsig, gsig_l2e, Aeps, B;
  int p, q;
  float h, c0;
  float rc_lo, sig_lo, sig_l2e_lo, gsig_l2e_lo, B_lo;  // as in FParams
};



struct Dev {
  int N, W, ncell, nbox;
  // master state: positions as 64-bit box fractions (s 2^64, wrapping), velocities
  // (A/fs) as unevaluated FP32 sums hi + lo (about 48 significant bits)
  unsigned long long *x, *y, *z;
  float2 *vx, *vy, *vz;
  unsigned long long *tx, *ty, *tz;
  float2 *tvx, *tvy, *tvz;
  int4 *img, *timg;   // periodic images crossed per component since the state was set (x, y, z)
  uint4 *q, *qb, *tq;
  float4* f;
  int *id, *tid;
  int *cell, *rank;
  int *cell_cnt, *cell_start;
  int* cell_box;      // box of each global cell
  int *nbr, *nbr_cnt;
  unsigned long long* bar;  // grid barrier of the persistent engine: two counters, kBarStride apart
  int* chunk;         // per-block cell totals of the persistent engine's scan
  int chunk_cap;
  const Box* box;
  BoxState* bst;
  double* thermo;     // nbox * TR_N
  Global* g;
  const Integ* integ;
  double* stage;      // n*3 doubles staging (user order)
  double* stage2;
  // several species (null / 1 for one species): species of each sorted atom
  // and its staging copy, the caller-order species, and the tables
  int *typ, *ttyp;
  const int* utyp;
  const SpPair* sp_pair;  // nsp^2, (a, b) at a nsp + b
  const float2* sp_tri;   // nsp^3: (lambda epsilon, cos theta0) of (centre a; legs b, c)
  int nsp;
  // phase marks of the persistent engine (null unless enabled): clock64 of
  // block 0 at kPhaseMarks points of each of the first marks_cap steps
  unsigned long long* marks;
  int marks_cap;
  // owner-computes force mode (null unless selected): per-atom moments of the
  // three-body terms (S0, s; M xx yy zz xy; M xz yz), the staged legs and
  // their count (-1: a centre over the staged-leg limit, done by scatter)
  float4* mom;
  int* legs;
  int* nleg;
};

constexpr int kPhaseMarks = 16;  // 14 used

// ---------------------------------------------------------------------------
// small helpers

// 32-bit fixed-point coordinate of a 64-bit box fraction: round(s / 2^32)
// mod 2^32 (a fraction within half a unit of 1 wraps to 0).
__device__ __forceinline__ uint32_t q_of(unsigned long long s) {
  return (uint32_t)((s + 0x80000000ull) >> 32);
}

// Box fraction in [0, 1) (FP64) -> 64-bit fraction round(s 2^64) mod 2^64.
__device__ __forceinline__ unsigned long long frac64_of(double s) {
  const double t = s * 18446744073709551616.0;
  return (t >= 18446744073709551616.0) ? 0ull : __double2ull_rn(t);
}

// FP64 arithmetic on GB300 runs at 1/64 of the FP32 rate, conversions to and
// from it included, and a division is ten such instructions: loading a state
// of 2^20 atoms took 142 us for 22 us of memory traffic, reading it back 62 us.
// The state's conversions below therefore take integer instructions where the
// result is the same (61 and 36 us).

// Box fraction of the coordinate x in an edge L, rl = 1 / L: round(x / L 2^64)
// mod 2^64 (the quotient corrected by its own remainder, Markstein's form: to
// its last FP64 bit), and the whole edges below it.
__device__ __forceinline__ unsigned long long box_fraction(double x, double L, double rl, int& image) {
  double q = x * rl;
  q = fma(fma(-q, L, x), rl, q);
  const unsigned long long u = (unsigned long long)__double_as_longlong(q);
  const int ex = (int)((u >> 52) & 0x7ffull);
  const int sh = ex - 1011;  // |q| 2^64 = m 2^sh
  if (sh > 42) {  // 2^31 edges away or more
    const double fl = floor(q);
    image = (int)fl;
    const double f = q - fl;
    return f >= 1.0 ? 0ull : frac64_of(f);
  }
  const unsigned long long m = (u & 0xfffffffffffffull) | (ex ? 0x10000000000000ull : 0ull);
  unsigned long long f;
  int whole = 0;
  if (sh >= 0) {
    f = m << sh;
    if (sh > 11) whole = (int)(m >> (64 - sh));
  } else if (sh > -64) {  // round to nearest, ties to even
    const int r = -sh;
    f = m >> r;
    const unsigned long long rest = m & ((1ull << r) - 1ull), half = 1ull << (r - 1);
    f += rest > half || (rest == half && (f & 1ull)) ? 1ull : 0ull;
  } else {
    f = 0ull;
  }
  if ((long long)u >= 0) {
    image = whole;
    return f;
  }
  image = -whole - (f ? 1 : 0);
  return 0ull - f;
}

// f 2^-64 L of a 64-bit box fraction f, rounded once to FP64: the normalised
// fraction times L's mantissa, its high half with the rest as a sticky bit.
__device__ __forceinline__ double fraction_times(unsigned long long f, double L) {
  if (f == 0ull) return 0.0;
  const int lz = __clzll((long long)f);
  const unsigned long long u = (unsigned long long)__double_as_longlong(L);  // (L > 0, normal)
  const unsigned long long n = f << lz, m = ((u & 0xfffffffffffffull) | 0x10000000000000ull) << 11;
  const unsigned long long h = __umul64hi(n, m) | (n * m ? 1ull : 0ull);  // f L 2^(1086 + lz - exponent of L)
  const long long scale = (long long)(u >> 52) - 1086 - lz;
  return __longlong_as_double(__double_as_longlong(__ull2double_rn(h)) + (scale << 52));
}

// FP32 to FP64, exact (a subnormal, which hardly any call meets, by the
// conversion instruction).
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t ex = (u >> 23) & 0xffu;
  if (ex == 0u && (u & 0x7fffffu)) return (double)f;
  const uint32_t hi = ex == 0u ? 0u : ((ex == 255u ? 2047u : ex + 896u) << 20) | ((u & 0x7fffffu) >> 3);
  return __hiloint2double((int)((u & 0x80000000u) | hi), ex == 0u ? 0 : (int)(u << 29));
}

// Reciprocal edges of the boxes of a block's first and last atom, in shared
// memory (a block of atoms holds one box or two, but for tiny ones).  Called
// by all threads with their atom's box (b < 0: none; box ids never decrease
// along atoms); edge() then serves any box.
struct BlockEdges {
  double L[2][3], r[2][3];
  int box[2];
};
__device__ __forceinline__ void block_edges(BlockEdges& S, const Box* box, int b) {
  if (threadIdx.x == 0) {
    S.box[0] = b;
    S.box[1] = b;
  }
  __syncthreads();
  if (b >= 0) atomicMax(&S.box[1], b);
  __syncthreads();
  if (threadIdx.x < 6 && S.box[0] >= 0) {
    const int w = (int)threadIdx.x / 3, k = (int)threadIdx.x % 3;
    const double L = box[S.box[w]].L[k];
    S.L[w][k] = L;
    S.r[w][k] = 1.0 / L;
  }
  __syncthreads();
}
__device__ __forceinline__ unsigned long long edge_fraction(const BlockEdges& S, const Box* box, int b, int k, double x, int& image) {
  const int w = b == S.box[0] ? 0 : 1;
  if (b == S.box[w]) return box_fraction(x, S.L[w][k], S.r[w][k], image);
  const double L = box[b].L[k];
  return box_fraction(x, L, 1.0 / L, image);
}

// Exact conversion of an FP32 value to a 64-bit integer with integer
// operations only (no FP64 or 64-bit conversion instruction): |f| >= 2^23 is
// an integer already; smaller values round half away from zero; zero and
// subnormals give 0; magnitudes beyond 2^62 are clamped (a runaway atom,
// reported separately).
__device__ __forceinline__ long long f2ll_exact(float f) {
  const uint32_t u = __float_as_uint(f);
  const int ex = (int)((u >> 23) & 0xffu);
  const long long m = (long long)((u & 0x7fffffu) | 0x800000u);
  const int e = ex - 150;  // |f| = m 2^e
  long long r;
  if (ex == 0) r = 0;
  else if (e >= 0) r = m << min(e, 38);
  else if (e > -25) r = (m + (1ll << (-e - 1))) >> (-e);
  else r = 0;
  return (u >> 31) ? -r : r;
}

// Velocity as hi + lo (FP32 pair) <-> FP64 (set/get state and rare paths only).
__device__ __forceinline__ float2 split_df(double v) {
  const float hi = (float)v;
  return make_float2(hi, (float)(v - widen(hi)));
}
__device__ __forceinline__ double join_df(float2 v) { return widen(v.x) + widen(v.y); }

__device__ __forceinline__ float fix_diff(uint32_t a, uint32_t b, float lq) {  // b - a, minimum image
  return __int2float_rn((int)(b - a)) * lq;
}

__device__ __forceinline__ void red_add_v4(float4* addr, float a, float b, float c) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(0.0f)
               : "memory");
}

__device__ __forceinline__ float powi(float x, int n) {
  float r = 1.0f;
  for (int k = 0; k < n; ++k) r *= x;
  return r;
}

// ---------------------------------------------------------------------------
// One leg's terms (Sec. II.A) to about one FP32 ulp each.  The exponentials
// exp(sig/(r - a sig)) and exp(gam sig/(r - a sig)) amplify a relative error
// of their argument by the argument's size (about 2 at the first shell), and
// at the first shell the derivative of the pair term is a difference of two
// parts five to twenty times larger than itself (it vanishes at the phi2
// minimum).  So r, 1/r, 1/(r - a sig), the exponent arguments and the pair
// derivative carry their first-order corrections, which also absorb the
// error of the hardware approximations they start from:
//   r = r0 + dr, r0 = r2 rsqrt(r2), dr = (r2 - r0^2) / (2 r0) (residual by one FMA);
//   1/r = v (1 + ev), v = rsqrt(r2), ev = (1 - r0 v) - dr v;
//   x = r - a sig = (r0 - rc) + (dr - rc_lo) (r0 - rc exact for r0 >= rc / 2);
//   1/x = t (1 + tc), t ~ 1/(r0 - rc), tc = (1 - (r0 - rc) t) - (dr - rc_lo) t;
//   exp2(k / x) = exp2(k t) (1 + ln 2 (k t tc + RN residual of k t + k_lo t)).
// For the SW exponents (p, q) = (4, 0) the pair derivative
//   dphi2/dr = A eps e2 [(1 - y) sig / x^2 - 4 y / r],  y = B (sig / r)^4,
// is formed from hi + lo pairs (exact products by FMA, two-sum at the final
// difference); other exponents take the plain FP32 formula.  Returns false
// (nothing to add) when the leg is not inside a sig.
struct LegTerms {
  float r, invr;  // |d|, 1 / |d|
  float e3;       // exp(gam sig / (r - a sig))
  float nde;      // gam sig / (r - a sig)^2
  float phi;      // phi2(r)
  float dphi;     // dphi2 / dr
  float t, ae2;   // 1 / (r - a sig), A eps exp(sig / (r - a sig)) (the adjoint's second derivative)
  float invu;     // 1 / |d| of the unstretched d (kFine): u = d invu
};

// 1/x from the hardware approximation (rcp.approx.ftz: within one ulp); the
// callers correct it to first order or need no more.
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// 1/sqrt(x) and 2^x from the hardware approximations, subnormal inputs and
// results flushed to zero (the leg arithmetic corrects 1/sqrt to first order
// and the exponent's argument likewise; a 2^x below 2^-126 belongs to a leg at
// the cutoff, whose terms vanish there).
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 2^(a + al), a <= 0 and al its low part, by the Taylor series of 2^f at the
// nearest integer (|f| <= 1/2, seven terms: truncation 5e-9), without the
// hardware approximation's bias, which is the same sign for every leg and so
// survives a sum over all of them.  Below 2^-126: 0 (ex2_approx flushes too).
__device__ __forceinline__ float exp2_taylor(float a, float al) {
  const float n = rintf(a);
  const float f = (a - n) + al;
  float p = 1.5252734e-5f;  // (ln 2)^k / k!, k = 7 ... 1
  p = fmaf(p, f, 1.5403530e-4f);
  p = fmaf(p, f, 1.3333558e-3f);
  p = fmaf(p, f, 9.6181291e-3f);
  p = fmaf(p, f, 5.5504109e-2f);
  p = fmaf(p, f, 2.4022651e-1f);
  p = fmaf(p, f, 6.9314718e-1f);
  p = fmaf(p, f, 1.0f);
  return n < -125.0f ? 0.0f : p * __int_as_float(((int)n + 127) << 23);
}

// kFine (the adjoint, whose parameter derivatives are sums of one sign over
// all legs): the exponentials by exp2_taylor instead of the hardware
// approximation, and the leg's length stretched by the relative amount
// `stretch` (below an FP32 ulp, so it goes into the low part dr).
template <bool kFine = false, class C>
__device__ __forceinline__ bool leg_terms(float r2, const C& c, LegTerms& o, float stretch = 0.f) {
  constexpr float kLn2 = 0.693147180559945f;
  const float v = rsqrt_approx(r2);
  const float r = r2 * v;
  float dr = 0.5f * fmaf(-r, r, r2) * v;
  if constexpr (kFine) {
    o.invu = fmaf(v, fmaf(-r, v, 1.0f) - dr * v, v);
    dr = fmaf(r, stretch, dr);
  }
  // (r itself may still round to the cutoff, or past it, when r + dr does not:
  // 1/(r - a sig) would then be infinite)
  if (!(fmaxf(r, r + dr) < c.rc)) return false;
  const float ev = fmaf(-r, v, 1.0f) - dr * v;
  const float xh = r - c.rc;
  const float xl = dr - c.rc_lo;
  const float t = rcp_approx(xh);  // < 0
  const float tc = fmaf(-xh, t, 1.0f) - xl * t;
  const float a2 = c.sig_l2e * t;
  const float a2l = fmaf(c.sig_l2e, t, -a2) + fmaf(a2, tc, c.sig_l2e_lo * t);
  float e2;
  if constexpr (kFine) {
    e2 = exp2_taylor(a2, a2l);
  } else {
    e2 = ex2_approx(a2);
    e2 = fmaf(e2, kLn2 * a2l, e2);
  }
  const float a3 = c.gsig_l2e * t;
  const float a3l = fmaf(c.gsig_l2e, t, -a3) + fmaf(a3, tc, c.gsig_l2e_lo * t);
  if constexpr (kFine) {
    o.e3 = exp2_taylor(a3, a3l);
  } else {
    const float e3 = ex2_approx(a3);
    o.e3 = fmaf(e3, kLn2 * a3l, e3);
  }
  const float invr = fmaf(v, ev, v);
  const float t2 = t * t;
  const float t2l = fmaf(t, t, -t2) + 2.0f * t2 * tc;  // t^2 (1 + 2 tc) = t2 + t2l
  o.r = r + dr;
  o.invr = invr;
  o.nde = c.gsig * fmaf(t2, 2.0f * tc, t2);
  const float ae2 = c.Aeps * e2;
  o.t = fmaf(t, tc, t);
  o.ae2 = ae2;
  if (c.p == 4 && c.q == 0) {
    // u = sig / r, y = B u^4, each as hi + lo
    const float uh = c.sig * v;
    const float ul = fmaf(c.sig, v, -uh) + fmaf(uh, ev, c.sig_lo * v);
    const float u2 = uh * uh;
    const float u2l = fmaf(uh, uh, -u2) + 2.0f * uh * ul;
    const float u4 = u2 * u2;
    const float u4l = fmaf(u2, u2, -u4) + 2.0f * u2 * u2l;
    const float yh = c.B * u4;
    const float yl = fmaf(c.B, u4, -yh) + fmaf(c.B, u4l, c.B_lo * u4);
    // 1 - y by two-sum (y exceeds 1 only for atoms closer than 2.1 A)
    const float om = 1.0f - yh;
    const float ob = om - 1.0f;
    const float oml = ((1.0f - (om - ob)) + (-yh - ob)) - yl;
    // part 1: (1 - y) sig t^2
    const float qh = c.sig * t2;
    const float ql = fmaf(c.sig, t2, -qh) + fmaf(c.sig, t2l, c.sig_lo * t2);
    const float p1 = om * qh;
    const float p1l = fmaf(om, qh, -p1) + fmaf(om, ql, oml * qh);
    // part 2: -4 y / r
    const float p2 = -4.0f * (yh * v);
    const float p2l = -4.0f * (fmaf(yh, v, -yh * v) + fmaf(yh * v, ev, yl * v));
    // their sum by two-sum, the low parts added once
    const float sh = p1 + p2;
    const float bb = sh - p1;
    const float se = (p1 - (sh - bb)) + (p2 - bb);
    const float g = sh + (se + p1l + p2l);
    o.dphi = ae2 * g;
    o.phi = -ae2 * (om + oml);
  } else {
    const float sr = c.sig * invr;
    const float srp = powi(sr, c.p), srq = powi(sr, c.q);
    const float brk = fmaf(c.B, srp, -srq);
    o.phi = ae2 * brk;
    o.dphi = ae2 * (fmaf((float)(-c.p) * c.B, srp, (float)c.q * srq) * invr - brk * c.sig * fmaf(t2, 2.0f * tc, t2));
  }
  return true;
}

__device__ __forceinline__ int cell_of(const uint4& q, const Box& bx) {
  const int cx = (int)(((unsigned long long)q.x * (unsigned)bx.nc[0]) >> 32);
  const int cy = (int)(((unsigned long long)q.y * (unsigned)bx.nc[1]) >> 32);
  const int cz = (int)(((unsigned long long)q.z * (unsigned)bx.nc[2]) >> 32);
  return bx.cell_off + cx + bx.nc[0] * (cy + bx.nc[1] * cz);
}

// The block's own error flag, for the engine whose barriers carry it (the
// other kernels neither clear nor read it).
__device__ __forceinline__ int& block_error() {
  __shared__ int s_error;
  return s_error;
}
__device__ __forceinline__ void set_status(Global* g, int st) {
  block_error() = 1;
  atomicCAS(&g->status, 0, st);
}
// A NaN found together with the next kick1's checks: its status stands over
// the runaway velocity that the same NaN makes there.
__device__ __forceinline__ void set_status_nan(Global* g) {
  block_error() = 1;
  if (atomicCAS(&g->status, 0, (int)ST_NAN) == ST_LOST) atomicCAS(&g->status, (int)ST_LOST, (int)ST_NAN);
}

// Arrival on a block counter, acq_rel at gpu scope: after a __syncthreads it
// publishes the whole block's writes (the barrier orders them before thread
// 0's release) and, for the last block to arrive, acquires every other
// block's.  Returns the count including this arrival.
__device__ __forceinline__ unsigned bar_arrive(unsigned* p) {
  unsigned old;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(p) : "memory");
  return old + 1u;
}

// Rebuilds are per box.  On a rebuild step every atom is binned and the scan
// over all cells gives absolute cell starts (every box's counts add up to its
// atom range), but only boxes whose flag kick1 raised (or that the host
// flagged) are re-sorted and re-listed; the others keep their order and list
// and never read their recomputed starts.
__device__ __forceinline__ bool box_flagged(const Dev& d, int b) { return d.bst[b].rebuild != 0; }

// Whether a build moves a box's atoms into cell order, or only builds the
// list: every kSortEvery-th build, and the first after a new state or anything
// else that flags every box.  The list is built from the cell-sorted copy tq,
// whose records carry their atoms' indices, so it does not need the atoms
// themselves in that order; they are sorted only so that a force block's
// candidates lie close together, and in the 8 builds between (about 40 steps)
// an atom diffuses well under a cell's width.  A build without the sort saves
// moving each atom's 100 bytes twice: k_scatter + k_copyback 65 us at 2^20
// atoms, 17 without.
constexpr int kSortEvery = 8;
__device__ __forceinline__ bool sorts(const BoxState& st) { return !st.sorted || st.rebuilds % kSortEvery == 0; }
__device__ __forceinline__ bool box_sorts(const Dev& d, int b) { return sorts(d.bst[b]); }
// A build of box b done (its scatter and copy-back have read the above).
__device__ __forceinline__ void box_built(const Dev& d, int b) {
  BoxState& st = d.bst[b];
  st.sorted = 1;
  st.rebuilds += 1;
  st.Lb = d.box[b].L[0];
}

// Per-box accumulation of NV values held as FP32 by each thread; the sums
// across blocks are FP64.  Every thread of the block calls it (b < 0 for
// threads without a contribution, whose values must be 0); thread 0 must hold
// the block's first box.  Atoms are box-major, so box ids along a warp are
// non-decreasing.  A warp within one box (nearly all) reduces its NV values
// by a transpose-reduce butterfly (about NV + 5 shuffles in all); a warp that
// straddles boxes runs a segmented FP32 scan over each run of one box.  Sums
// of the block's first and last box are combined in shared memory (FP32) and
// widened to FP64 for one global atomic per value and block; sums of other
// boxes (small boxes only) go to global memory directly.
template <int NV, class Dst>
__device__ void box_accumulate(float (&v)[NV], int b, Dst dst) {
  static_assert(NV <= 16, "two slots of NV sums are flushed by warp 0");
  __shared__ float sacc[2][NV];
  __shared__ int sbox[2];
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    sbox[0] = b;
    sbox[1] = -1;
  }
  if (threadIdx.x < 2 * NV) (&sacc[0][0])[threadIdx.x] = 0.f;
  __syncthreads();
  if (b >= 0) atomicMax(&sbox[1], b);  // the block's last box (box ids never decrease along atoms)
  const int b0 = __shfl_sync(kFull, b, 0);
  constexpr bool kPow2 = (NV & (NV - 1)) == 0;
  if (kPow2 && __all_sync(kFull, b == b0 || b < 0)) {
    // the warp holds one box (the common case): transpose-reduce, each of the
    // NV sums ending on its own group of 32/NV lanes
    int off = 16;
#pragma unroll
    for (int n = NV; n > 1; n >>= 1) {
      const bool up = (lane & off) != 0;
#pragma unroll
      for (int k = 0; k < n / 2; ++k) {
        const float send = up ? v[k] : v[k + n / 2];
        const float keep = up ? v[k + n / 2] : v[k];
        v[k] = keep + __shfl_xor_sync(kFull, send, off);
      }
      off >>= 1;
    }
#pragma unroll
    for (; off > 0; off >>= 1) v[0] += __shfl_xor_sync(kFull, v[0], off);
    __syncthreads();
    constexpr int kGroup = 32 / NV;
    if (b0 >= 0 && lane % kGroup == 0) {
      const int k = lane / kGroup;
      const int slot = (b0 == sbox[0]) ? 0 : ((b0 == sbox[1]) ? 1 : -1);
      if (slot >= 0) atomicAdd(&sacc[slot][k], v[0]);
      else atomicAdd(dst(b0) + k, (double)v[0]);
    }
  } else {
    // segmented FP32 scan over the runs of one box in the warp
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int bo = __shfl_up_sync(kFull, b, off);
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const float vo = __shfl_up_sync(kFull, v[k], off);
        if (lane >= off && bo == b) v[k] += vo;
      }
    }
    const int bn = __shfl_down_sync(kFull, b, 1);
    __syncthreads();
    const bool tail = (b >= 0) && (lane == 31 || bn != b);
    if (tail) {
      const int slot = (b == sbox[0]) ? 0 : ((b == sbox[1]) ? 1 : -1);
      if (slot >= 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) atomicAdd(&sacc[slot][k], v[k]);
      } else {
        double* p = dst(b);
#pragma unroll
        for (int k = 0; k < NV; ++k) atomicAdd(p + k, (double)v[k]);
      }
    }
  }
  __syncthreads();
  // warp 0 alone reads the shared sums after the barrier, so a following call
  // (whose warp 0 resets them first) cannot race with these reads
  if (threadIdx.x < NV && sbox[0] >= 0) atomicAdd(dst(sbox[0]) + threadIdx.x, (double)sacc[0][threadIdx.x]);
  if (threadIdx.x >= 16 && threadIdx.x < 16 + NV && sbox[1] >= 0 && sbox[1] != sbox[0])
    atomicAdd(dst(sbox[1]) + (threadIdx.x - 16), (double)sacc[1][threadIdx.x - 16]);
}

// ---------------------------------------------------------------------------
// Thermostat (Sec. II.B: Nose-Hoover, tau = 1 ps; Berendsen as the option).
// GB300 issues an FP64 instruction at a small fraction of the FP32 rate, even
// for one active lane, so the per-step thermostat arithmetic is FP32: xi and
// eta are unevaluated FP32 pairs hi + lo (their increments are tiny against
// their values), the kinetic energy enters through d = 2 KE - N_df k_B T0,
// formed with one FP64 FMA from the FP64 sum, and a velocity scale s is
// carried as sig = s - 1 (expm1f): the kick applies v += sig v, and the
// relative FP32 error of sig (~1e-4 in size) is ~1e-12 of s.

// a += b for an unevaluated pair a = (hi, lo) and an FP32 b (two-sum).
__device__ __forceinline__ void df_add(float& hi, float& lo, float b) {
  const float s = hi + b;
  const float bb = s - hi;
  const float e = (hi - (s - bb)) + (b - bb);
  const float l = lo + e;
  hi = s + l;
  lo = l - (hi - s);
}

struct ThermoState {  // one box at a step boundary
  float xh, xl, eh, el;  // xi, eta as hi + lo
  float d;               // 2 KE - N_df k_B T0 (FP32)
  float ke;              // KE in FP32 (for the scale's effect on d)
};

// One Nose-Hoover half step (length dt/2) of a single thermostat: quarter step
// on xi, velocity scale exp(-xi dt/2), half step on eta, quarter step on xi.
// Returns sig = s - 1; KE and d follow the scale.
__device__ __forceinline__ float nh_half(const Integ& I, const Box& bx, ThermoState& t) {
  const float hdt = 0.5f * (float)I.dt;
  df_add(t.xh, t.xl, bx.q4f * t.d);
  const float sig = expm1f(-hdt * t.xh);
  const float f = sig * (2.0f + sig);  // s^2 - 1
  const float dke = t.ke * f;
  t.ke += dke;
  t.d = fmaf(2.0f, dke, t.d);
  df_add(t.eh, t.el, hdt * t.xh);
  df_add(t.xh, t.xl, bx.q4f * t.d);
  return sig;
}

// End-of-step half, after the second half-kick: Nose-Hoover half step, or
// the Berendsen scale s = sqrt(1 + dt/tau (T0/T - 1)) (sig = x / (s + 1) with
// x = dt/tau (T0/T - 1), free of cancellation); NVE changes nothing.
// (kNpt: the isobaric instantiation, whose thermostat is always Nose-Hoover)
template <bool kNpt = false>
__device__ __forceinline__ float end_half(const Integ& I, const Box& bx, ThermoState& t) {
  if (kNpt || I.kind == TH_NH) return nh_half(I, bx, t);
  if (I.kind == TH_BERENDSEN && t.ke > 0.f) {
    const float T = 2.0f * t.ke * (float)bx.inv_ndf_kb;
    const float x = (float)(I.dt / I.tau) * ((float)bx.T0 / T - 1.0f);
    const float sig = x / (sqrtf(1.0f + x) + 1.0f);
    const float f = sig * (2.0f + sig);
    t.ke += t.ke * f;
    return sig;
  }
  return 0.f;
}

// Start-of-step half, before the first half-kick (Nose-Hoover only).
template <bool kNpt = false>
__device__ __forceinline__ float start_half(const Integ& I, const Box& bx, ThermoState& t) {
  return (kNpt || I.kind == TH_NH) ? nh_half(I, bx, t) : 0.f;
}

__device__ __forceinline__ ThermoState thermo_in(const Box& bx, float4 th, double ke) {
  ThermoState t;
  t.xh = th.x;
  t.xl = th.y;
  t.eh = th.z;
  t.el = th.w;
  t.d = (float)fma(2.0, ke, -bx.ndfkT0);
  t.ke = (float)ke;
  return t;
}

// Thermo record of box b for the last completed step (parity pp): the
// thermostat state after its end half and the step's energies and virial.
// Written only when the host reads it (k_record).
__device__ void write_record(const Dev& d, const Integ& I, int b, int pp, unsigned long long step_done) {
  const BoxState* st = d.bst + b;
  const Box& bx = d.box[b];
  double* r = d.thermo + (size_t)b * TR_N;
  const double e2 = st->ew[pp][0], e3 = st->ew[pp][1];
  const double ke = st->ke_last;
  const double xi = (double)st->th_e.x + (double)st->th_e.y, eta = (double)st->th_e.z + (double)st->th_e.w;
  const double V = bx.volume;  // the box of the completed step (the next one is made current in its kick1)
  r[TR_STEP] = (double)step_done;
  r[TR_PE] = e2 + e3;
  r[TR_E2] = e2;
  r[TR_E3] = e3;
  r[TR_KE] = ke;
  r[TR_T] = 2.0 * ke * bx.inv_ndf_kb;
  double cons = ke + e2 + e3;
  if (I.kind == TH_NH || I.kind == TH_NPT) cons += 0.5 * bx.Q * xi * xi + bx.ndfkT0 * eta;
  if (I.kind == TH_NPT) cons += I.p_ext * V + 0.5 * st->pe_e * st->pe_e / bx.W;
  r[TR_CONS] = cons;
  r[TR_P] = (2.0 * ke + st->ew[pp][2] + st->ew[pp][3] + st->ew[pp][4]) / (3.0 * V) * kATM;
  for (int k = 0; k < 6; ++k) r[TR_W0 + k] = st->ew[pp][2 + k];
  r[TR_XI] = xi;
  r[TR_ETA] = eta;
  r[TR_REBUILDS] = (double)st->rebuilds;
  r[TR_VOL] = V;
  for (int k = 0; k < 3; ++k) r[TR_L0 + k] = bx.L[k];
}

// How the end-of-step tails read what an earlier phase wrote: with L2 loads
// from global memory (another block may have written it in the same launch),
// or plainly from the block's own shared copy (the cluster engine).
struct LdGlobal {
  template <class T>
  __device__ static T get(const T& v) { return __ldcg(&v); }
};
struct LdShared {
  template <class T>
  __device__ static T get(const T& v) { return v; }
};

// Isotropic barostat (Sec. II.B, read as the Martyna-Tobias-Klein form):
// half step on its momentum, pe += dt/2 [(1 + 3/N_df) 2 KE + tr(W) - 3 P V],
// and the friction on the velocities, v *= exp(-dt/2 (1 + 3/N_df) pe/W),
// returned as s - 1 (FP32).  pe and the volume stay FP64.
template <class Ld = LdGlobal>
__device__ __forceinline__ void baro_half(const Integ& I, const Box& bx, double ke, double trw, double& pe) {
  pe += 0.5 * I.dt * (bx.a3 * 2.0 * ke + trw - 3.0 * I.p_ext * Ld::get(bx.volume));
}
__device__ __forceinline__ float baro_friction(const Integ& I, const Box& bx, double pe) {
  return expm1f((float)quotient(-0.5 * I.dt * bx.a3 * pe, bx.W));
}

// The box of the coming step: every edge scaled by e^u, u = dt pe/W, during
// its drift.  A box fraction then advances by (v dt / L) (1 - e^-u)/u (the
// drift r -> r e^u + v dt e^(u/2) sinh(u/2)/(u/2) divided by the new edge),
// which the kick kernel's drift factor absorbs; the new edges (Ln) become
// current after that drift, in time for the list build and the force.
// Rebuild margin: a pair outside the list (r >= r_list at the build) is at
// least c r_list - 2 d apart, c = L/L_build, d the largest displacement
// since the build, so the list holds while 2 d <= r_list - r_c -
// r_list max(0, 1 - c); the displacement is measured with the current
// edges, e^-u of the new ones.  A margin below skin/2 rebuilds at once.
// Returns bit 0: the margin asks for a rebuild, bit 1: the box left its grid.
template <class Ld>
__device__ int npt_geometry_of(const Integ& I, Box& bx, BoxState& st, double pe) {
  const float u = (float)quotient(I.dt * pe, bx.W);
  const float eu = expm1f(u);
  const float fdr = fabsf(u) > 1e-3f ? -expm1f(-u) / u : fmaf(u, fmaf(u, 1.0f / 6.0f, -0.5f), 1.0f);
  const float dt64 = (float)(I.dt * 18446744073709551616.0);  // dt 2^64
  int out = 0;
  for (int k = 0; k < 3; ++k) {
    const double L = Ld::get(bx.L[k]);
    const double Ln = fma(L, (double)eu, L);
    bx.dtL64[k] = dt64 / (float)L * fdr;
    bx.Ln[k] = Ln;
    const int nc = bx.nc[k];
    if (Ln < 2.0 * I.rlist || (nc >= 4 && Ln < nc * (double)I.rlist) || Ln >= (nc + 1) * kCellGrow * I.rlist) out = 2;
  }
  const float c = (float)quotient(bx.Ln[0], Ld::get(st.Lb));
  const float m = I.skin - I.rlist * fmaxf(0.0f, 1.0f - c);
  if (m < 0.5f * I.skin) {
    st.rebuild = 1;
    out |= 1;
  }
  const float h = 0.5f * fmaxf(m, 0.0f) / (1.0f + eu);
  bx.hs2 = h * h;
  return out;
}
__device__ void npt_geometry(const Dev& d, const Integ& I, int b, double pe) {
  const int r = npt_geometry_of<LdGlobal>(I, const_cast<Box*>(d.box)[b], d.bst[b], pe);
  if (r & 2) set_status(d.g, ST_GRID);
  if (r & 1) d.g->any_rebuild = 1;
}

// The edges of the coming step made current (the last block of kick1, once
// every block has drifted with the old ones).
template <class Ld>
__device__ void npt_commit(Box& bx) {
  double vol = 1.0;
  for (int k = 0; k < 3; ++k) {
    const double Ln = Ld::get(bx.Ln[k]);
    bx.L[k] = Ln;
    bx.Lq[k] = (float)(Ln * 2.3283064365386963e-10);  // 2^-32
    vol *= Ln;
  }
  bx.volume = vol;
}
__device__ void npt_commit_box(const Dev& d, int b) { npt_commit<LdGlobal>(const_cast<Box*>(d.box)[b]); }

// Thermostat at the end of a step, for one box (after the step's kinetic-
// energy sum ke0 is complete): the end half of this step, then the start half
// of the next one; stores the state after each half and the combined scale
// S - 1 the next kick1 applies.  Isobaric (kNpt instantiations only, so that
// the FP64 barostat arithmetic does not raise the register count of the
// others; trw the trace of the step's virial): friction, barostat half,
// thermostat half end this step; thermostat half, barostat half, friction
// start the next; then the new box.  Returns npt_geometry_of's bits.
template <bool kNpt, class Ld>
__device__ int end_of_step(const Integ& I, Box& bx, BoxState& st, double ke0, double trw) {
  if constexpr (kNpt) {
    double pe = Ld::get(st.pe_b);
    const float f1 = baro_friction(I, bx, pe);
    double ke = fma(ke0, (double)(f1 * (2.0f + f1)), ke0);
    baro_half<Ld>(I, bx, ke, trw, pe);
    ThermoState t = thermo_in(bx, Ld::get(st.th), ke);
    const float se = end_half<true>(I, bx, t);
    ke = fma(ke, (double)(se * (2.0f + se)), ke);
    st.th_e = make_float4(t.xh, t.xl, t.eh, t.el);
    st.ke_last = ke;
    st.pe_e = pe;
    const float e1 = fmaf(f1, se, f1 + se);
    st.s_endc = 1.0 + (double)e1;
    const float ss = start_half<true>(I, bx, t);
    ke = fma(ke, (double)(ss * (2.0f + ss)), ke);
    st.th = make_float4(t.xh, t.xl, t.eh, t.el);
    baro_half<Ld>(I, bx, ke, trw, pe);
    const float f2 = baro_friction(I, bx, pe);
    const float e2 = fmaf(ss, f2, ss + f2);
    st.sig = fmaf(e1, e2, e1 + e2);
    st.pe_b = pe;
    return npt_geometry_of<Ld>(I, bx, st, pe);
  } else {
    ThermoState t = thermo_in(bx, Ld::get(st.th), ke0);
    const float se = end_half(I, bx, t);
    st.th_e = make_float4(t.xh, t.xl, t.eh, t.el);
    st.ke_last = fma(ke0, (double)(se * (2.0f + se)), ke0);
    st.s_endc = 1.0 + (double)se;
    const float ss = start_half(I, bx, t);
    st.th = make_float4(t.xh, t.xl, t.eh, t.el);
    st.sig = fmaf(se, ss, se + ss);
    return 0;
  }
}

// The same for box b of the step of parity par, from the global sums (one
// thread per box, in the last block to finish).
template <bool kNpt>
__device__ void end_of_step_box(const Dev& d, const Integ& I, int b, int par) {
  BoxState& st = d.bst[b];
  const double ke0 = __ldcg(&st.ke_acc[par]);
  const double trw = kNpt ? __ldcg(&st.ew[par][2]) + __ldcg(&st.ew[par][3]) + __ldcg(&st.ew[par][4]) : 0.0;
  const int r = end_of_step<kNpt, LdGlobal>(I, const_cast<Box*>(d.box)[b], st, ke0, trw);
  if (r & 2) set_status(d.g, ST_GRID);
  if (r & 1) d.g->any_rebuild = 1;
}

// Start half only, from the state after the last end half (a new state, or a
// changed integrator): the scale S - 1 includes the pending end scale.
__global__ void k_prime_thermostat(Dev d) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= d.nbox) return;
  const Integ I = *d.integ;
  BoxState* st = d.bst + b;
  const Box& bx = d.box[b];
  ThermoState t = thermo_in(bx, st->th_e, st->ke_last);
  const float se = (float)(st->s_endc - 1.0);
  const float ss = I.kind == TH_NPT ? start_half<true>(I, bx, t) : start_half(I, bx, t);
  st->th = make_float4(t.xh, t.xl, t.eh, t.el);
  float e2 = ss;
  if (I.kind == TH_NPT) {  // barostat half and friction with the latest virial
    const int wp = d.g->wpar;
    const double trw = st->ew[wp][2] + st->ew[wp][3] + st->ew[wp][4];
    const double ke = fma(st->ke_last, (double)(ss * (2.0f + ss)), st->ke_last);
    double pe = st->pe_e;
    baro_half(I, bx, ke, trw, pe);
    const float f2 = baro_friction(I, bx, pe);
    e2 = fmaf(ss, f2, ss + f2);
    st->pe_b = pe;
    npt_geometry(d, I, b, pe);
  }
  st->sig = fmaf(se, e2, se + e2);
}

// Uniform early exit of a block on a device error status (one read, shared),
// so that no warp skips a barrier the others wait at.
__device__ __forceinline__ bool block_stop(const Dev& d) {
  __shared__ int s_stop;
  if (threadIdx.x == 0) s_stop = *(volatile int*)&d.g->status;
  __syncthreads();
  return s_stop != 0;
}

// ---------------------------------------------------------------------------
// Phase bodies (one item each) shared by the per-phase kernels and the
// persistent kernel.

// a1 + a7 (first half): the second half-kick of the last step and the first
// of this one use the same force, so they are folded: v = S v + (S + 1) a
// when a half-kick is pending (S = thermostat scale of the step boundary,
// a = dt/2 F/m), else v = S v + a; then s += (dt/L) v on the box fraction,
// fixed-point copy, displacement check against the last build.  One thread
// per atom, its three components in turn: every array is read and written
// with one coalesced vector access per warp (the force and the fixed-point
// copies as 16-byte records, the velocity and fraction components as 8-byte
// words), and the box's constants are loaded once per atom.  No FP64
// instruction: v is the unevaluated sum hi + lo of two FP32 values, updated
// as hi + t with t = (S - 1) v + kick and the rounding error of that sum
// carried into lo (Knuth's two-sum); the drift (dt/L) v 2^64 is rounded once
// to FP32 and added exactly to the 64-bit box fraction, which wraps at the
// faces by itself.  The runaway check is an integer test of the FP32
// exponent.  Also zeroes f for this step.
constexpr int kKThreads = 256;  // threads per block of k_kick1 / k_kick2

struct Kick1In {  // one atom's inputs
  float4 F;
  uint4 qb;
  float2 v[3];
  unsigned long long s[3];
};
__device__ __forceinline__ Kick1In kick1_load(const Dev& d, int i) {
  return {d.f[i], d.qb[i], {d.vx[i], d.vy[i], d.vz[i]}, {d.x[i], d.y[i], d.z[i]}};
}

// The kick, drift and displacement check of atom i in box b, results stored;
// moved: the atom is further than the rebuild margin from its list position;
// lost: a velocity component at or above the runaway threshold, or NaN/inf.
template <bool kNpt>
__device__ __forceinline__ void kick1_apply(const Dev& d, const Integ& I, const Box& bx, float sig, int i, int b, int pend,
                                            const Kick1In& in, bool& moved, bool& lost) {
  const float kf = I.cf_f * (pend ? 2.0f + sig : 1.0f);
  const int vexp = bx.vexp_lost;
  const float Fc[3] = {in.F.x, in.F.y, in.F.z};
  const uint32_t qbc[3] = {in.qb.x, in.qb.y, in.qb.z};
  float2 vn[3];
  unsigned long long sn[3];
  uint32_t qn[3];
  float dd = 0.f;  // squared displacement since the last build
  lost = false;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    // v + t as hi + lo: two-sum of hi and t, its error added to lo, renormalised
    const float t = fmaf(sig, in.v[c].x, fmaf(sig, in.v[c].y, kf * Fc[c]));
    const float sh = in.v[c].x + t;
    const float bb = sh - in.v[c].x;
    const float er = (in.v[c].x - (sh - bb)) + (t - bb);
    const float lo1 = in.v[c].y + er;
    const float hi = sh + lo1;
    const float lo = lo1 - (hi - sh);
    const float k64 = bx.dtL64[c];
    const long long inc = f2ll_exact(fmaf(hi, k64, lo * k64));
    sn[c] = in.s[c] + (unsigned long long)inc;
    if (inc > 0 ? sn[c] < in.s[c] : sn[c] > in.s[c])  // the 64-bit fraction wrapped: the atom crossed a face
      reinterpret_cast<int*>(d.img + i)[c] += inc > 0 ? 1 : -1;
    vn[c] = make_float2(hi, lo);
    qn[c] = q_of(sn[c]);
    const float dc = fix_diff(qbc[c], qn[c], bx.Lq[c]);
    dd += __fmul_rn(dc, dc);
    // |v| at or above the box's runaway threshold (or NaN/inf): exponent field test
    lost |= (int)((__float_as_uint(hi) >> 23) & 0xffu) >= vexp;
  }
  d.f[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  d.vx[i] = vn[0];
  d.vy[i] = vn[1];
  d.vz[i] = vn[2];
  d.x[i] = sn[0];
  d.y[i] = sn[1];
  d.z[i] = sn[2];
  d.q[i] = make_uint4(qn[0], qn[1], qn[2], (unsigned)b);
  moved = dd > (kNpt ? bx.hs2 : I.half_skin2);
}

// The kinetic energy of v + a (FP32 per component and per atom).
__device__ __forceinline__ float kick2_energy(const Integ& I, const float4& F, const float2 (&v)[3]) {
  const float Fc[3] = {F.x, F.y, F.z};
  float ke = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float u = fmaf(I.cf_f, Fc[c], v[c].x) + v[c].y;
    ke += (float)I.ke_fac * u * u;
  }
  return ke;
}

// boxes, states: d.box and d.bst, or a block's own copies of the fields read
// here.  late: the step before left its NaN check to this one.
template <bool kNpt>
__device__ __forceinline__ void kick1_atom(const Dev& d, const Integ& I, int i, int par, int pend, const Box* boxes,
                                           const BoxState* states, bool late) {
  // every load first (nothing here is written by another atom's thread);
  // the fixed-point copy is read only for its box (one box: box 0)
  const int b = d.nbox == 1 ? 0 : (int)d.q[i].w;
  const Kick1In in = kick1_load(d, i);
  const Box& bx = boxes[b];
  bool moved, lost;
  kick1_apply<kNpt>(d, I, bx, states[b].sig, i, b, pend, in, moved, lost);
  if (i == bx.off) {  // this step's accumulators start from zero
    BoxState* sw = d.bst + b;
    sw->ke_acc[par] = 0.0;
#pragma unroll
    for (int k2 = 0; k2 < 8; ++k2) sw->ew[par][k2] = 0.0;
  }
  if (moved) {
    d.bst[b].rebuild = 1;
    d.g->any_rebuild = 1;
  }
  if (lost) {
    set_status(d.g, ST_LOST);
    d.g->err_index = i;
  }
  if (late && !(kick2_energy(I, in.F, in.v) < 1e30f)) {
    set_status_nan(d.g);
    d.g->err_index = i;
  }
}

// a7 (second half): the kinetic energy of atom i's v + a (FP32 per
// component and per atom; the sums over atoms are FP64).  The half-kick
// itself is left pending and folded into the next kick1 (or applied when the
// state is read).  b: the atom's box (-1 past the last atom).
__device__ __forceinline__ float kick2_atom(const Dev& d, const Integ& I, int i, int& b) {
  b = -1;
  if (i >= d.N) return 0.f;
  b = d.nbox == 1 ? 0 : (int)d.q[i].w;
  const float4 F = d.f[i];
  const float2 v[3] = {d.vx[i], d.vy[i], d.vz[i]};
  const float ke = kick2_energy(I, F, v);
  if (!(ke < 1e30f)) {
    set_status(d.g, ST_NAN);
    d.g->err_index = i;
  }
  return ke;
}

// ---------------------------------------------------------------------------
// Neighbour list (a3): one warp per cell.  The candidates of the stencil are
// staged, up to kNStage at a time, in the warp's slice of shared memory; then
// the centre atoms of the cell, kNeighCentres at a time, run over the staged
// candidates, and the hits of each batch go straight to their places in each
// centre's row (its running count plus the hits of lower lanes).  Bound by
// instruction issue.  Two forms:
//   neigh_rows_frame: every axis of the box has at least 4 cells;
//   neigh_rows_wrap: grids of 1-3 cells on an axis, where the stencil wraps
//     round the box: the (deduplicated) cells' fixed-point coordinates are
//     staged and each pair takes its own minimum-image difference.
constexpr int kNStage = 256;  // candidates staged per warp at a time (4 KB)
constexpr int kNSlice = kNStage + 8;  // float4 of shared memory a warp: the candidates, a mark per candidate, 18 runs
constexpr int kNeighCentres = 2;  // centres tested together against each staged batch
__device__ __forceinline__ int stencil_n(int nc) { return nc >= 3 ? 3 : nc; }
__device__ __forceinline__ int stencil_off(int nc, int o) { return nc >= 3 ? o - 1 : o; }

// Two FP32 values in a register pair: the packed instructions round each half
// as the scalar ones do, at one issue slot for both.
__device__ __forceinline__ unsigned long long pk2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void upk2(unsigned long long v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// One candidate per lane against one centre: its hit (r2 < rl2, not the centre
// itself) is stored as j at row[min(count + hits of lower lanes, last)], and
// the count of the warp's hits is added to count.  In one piece, so that the
// hit stays a predicate from the test to the store.
__device__ __forceinline__ void neigh_hit(float r2, float rl2, int j, int centre, unsigned below, int last, int* row, int& count) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b32 m, t;\n .reg .b64 a;\n"
      " setp.ne.s32 p, %2, %3;\n"
      " setp.lt.and.f32 p, %1, %4, p;\n"
      " vote.sync.ballot.b32 m, p, 0xffffffff;\n"
      " and.b32 t, m, %5;\n"
      " popc.b32 t, t;\n"
      " add.s32 t, t, %0;\n"
      " min.s32 t, t, %6;\n"
      " mad.wide.s32 a, t, 4, %7;\n"
      " @p st.global.b32 [a], %2;\n"
      " popc.b32 t, m;\n"
      " add.s32 %0, %0, t;\n}"
      : "+r"(count)
      : "f"(r2), "r"(j), "r"(centre), "f"(rl2), "r"(below), "r"(last), "l"(row)
      : "memory");
}

// The longest row so far, from one warp's rows: one atomic per warp, and none
// once the running maximum covers it (rather than one per centre on this one
// word).  Returns whether a row is wider than its allocation.
__device__ __forceinline__ bool neigh_count(const Dev& d, int mycount) {
  const int wmax = __reduce_max_sync(kFull, mycount);
  if ((threadIdx.x & 31) == 0 && wmax > *(volatile int*)&d.g->max_count) {
    atomicMax(&d.g->max_count, wmax);
    if (wmax > d.W) set_status(d.g, ST_OVERFLOW);
  }
  return wmax > d.W;
}

// The rows of one cell's centres, every axis of the box at least 4 cells long:
// each candidate then lies within two cell edges of o, the cell's first atom;
// offsets from o are exact fixed-point differences with no wrap, converted
// once per atom and staged as FP32, and a pair's displacement is their FP32
// difference.  The stencil is 9 runs of atoms (three cells along x lie next
// to one another; a cell at the box's x face splits each run in two): lane r
// holds run r, first its first atom, excl its place among the candidates.
// Each lane tests two neighbouring candidates at a time with packed FP32
// arithmetic, against kNeighCentres centres per staged record read.  Padding
// entries fail the test by their offset.  A count past the row width (an
// overflow: the status makes the caller grow the rows and build again) writes
// to the row's last slot, never past it.
// 2^20-atom slab, full build: 277 us, 253 M warp instructions (310 us and 289 M with one candidate a lane and every staging
// batch located by a binary search over the 27 cells; 3 centres at a time 290 us).
__device__ __forceinline__ bool neigh_rows_frame(const Dev& d, const uint4* qa, const uint4& o, float* stg, int a0, int ni, int first, int cnt,
                                                 int excl, int total, float L0, float L1, float L2, float rl2, int part,
                                                 int parts, bool slots) {
  static_assert(kNStage % 64 == 0, "whole groups of two candidates a lane");
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;  // lanes under this one
  float* const sx = stg;
  float* const sy = stg + kNStage;
  float* const sz = stg + 2 * kNStage;
  int* const sj = reinterpret_cast<int*>(stg + 3 * kNStage);
  unsigned* const marks = reinterpret_cast<unsigned*>(stg + 4 * kNStage);
  int* const delta = reinterpret_cast<int*>(marks + kNStage / 32);  // per run that is not empty: first atom - place
  bool over = false;
  {
    const unsigned full = __ballot_sync(kFull, cnt > 0);
    if (cnt > 0) delta[__popc(full & below)] = first - excl;
  }
  for (int ib = 0; ib < ni; ib += 32) {  // centre atoms of this cell, 32 at a time
    const int nb = min(32, ni - ib);
    const int ms = a0 + ib + min(lane, nb - 1);
    const uint4 qmine = qa[ms];  // lane k's centre
    const int me = slots ? ms : (int)qmine.w;  // and its index
    const float cx = fix_diff(qmine.x, o.x, L0), cy = fix_diff(qmine.y, o.y, L1), cz = fix_diff(qmine.z, o.z, L2);  // o - centre
    int mycount = 0;  // neighbours of lane k's centre so far
    for (int c0 = 0; c0 < total; c0 += kNStage) {  // chunks of the candidate list (warp-uniform)
      const int nch = min(kNStage, total - c0);
      const int nbat = (nch + 31) >> 5, ngrp = nbat >> 1;  // whole groups of 64; an odd batch of 32 is left over
      __syncwarp();  // the previous chunk's readers are done
      // the run that holds candidate t: as many marks (first candidates of
      // runs that are not empty) up to t, counted from the runs before c0
      if (lane < kNStage / 32) marks[lane] = 0u;
      __syncwarp();
      if (cnt > 0 && excl >= c0 && excl < c0 + kNStage) atomicOr(marks + ((excl - c0) >> 5), 1u << ((excl - c0) & 31));
      int seen = __popc(__ballot_sync(kFull, cnt > 0 && excl < c0)) - 1;
      __syncwarp();
      for (int t = lane; t - lane < nch; t += 32) {  // (warp-uniform)
        const unsigned mk = marks[t >> 5];
        const int r = seen + __popc(mk & (below | (1u << lane)));
        seen += __popc(mk);
        float x = 1e30f, y = 0.f, z = 0.f;  // past the last candidate: no hit
        int j = -1;
        if (t < nch) {
          j = c0 + t + delta[r];
          const uint4 qj = qa[j];
          if (!slots) j = (int)qj.w;
          x = fix_diff(o.x, qj.x, L0);
          y = fix_diff(o.y, qj.y, L1);
          z = fix_diff(o.z, qj.z, L2);
        }
        sx[t] = x;
        sy[t] = y;
        sz[t] = z;
        sj[t] = j;
      }
      __syncwarp();
      for (int k = kNeighCentres * part; k < nb; k += kNeighCentres * parts) {  // (warp-uniform)
        unsigned long long xc[kNeighCentres], yc[kNeighCentres], zc[kNeighCentres];
        int ic[kNeighCentres], cc[kNeighCentres];
        int* rc[kNeighCentres];
        bool on[kNeighCentres];  // (a last group may hold fewer centres)
        const int wl = d.W - 1;
#pragma unroll
        for (int c = 0; c < kNeighCentres; ++c) {
          on[c] = k + c < nb;
          const int kc = on[c] ? k + c : k;
          float x = __shfl_sync(kFull, cx, kc);
          const float y = __shfl_sync(kFull, cy, kc), z = __shfl_sync(kFull, cz, kc);
          if (!on[c]) x = 1e30f;  // no hits
          xc[c] = pk2(x, x);
          yc[c] = pk2(y, y);
          zc[c] = pk2(z, z);
          ic[c] = __shfl_sync(kFull, me, kc);
          cc[c] = __shfl_sync(kFull, mycount, kc);
          rc[c] = d.nbr + (size_t)ic[c] * d.W;
        }
        for (int gr = 0; gr < ngrp; ++gr) {
          const int at = (gr << 6) + 2 * lane;
          const unsigned long long ex = *reinterpret_cast<const unsigned long long*>(sx + at);
          const unsigned long long ey = *reinterpret_cast<const unsigned long long*>(sy + at);
          const unsigned long long ez = *reinterpret_cast<const unsigned long long*>(sz + at);
          const int2 j = *reinterpret_cast<const int2*>(sj + at);
#pragma unroll
          for (int c = 0; c < kNeighCentres; ++c) {
            const unsigned long long dx = add2(ex, xc[c]), dy = add2(ey, yc[c]), dz = add2(ez, zc[c]);
            float r0, r1;
            upk2(fma2(dx, dx, fma2(dy, dy, mul2(dz, dz))), r0, r1);
            neigh_hit(r0, rl2, j.x, ic[c], below, wl, rc[c], cc[c]);
            neigh_hit(r1, rl2, j.y, ic[c], below, wl, rc[c], cc[c]);
          }
        }
        if (nbat & 1) {  // one candidate a lane
          const int at = (ngrp << 6) + lane;
          const float ex = sx[at], ey = sy[at], ez = sz[at];
          const int j = sj[at];
#pragma unroll
          for (int c = 0; c < kNeighCentres; ++c) {
            float xx, yy, zz, u;
            upk2(xc[c], xx, u);
            upk2(yc[c], yy, u);
            upk2(zc[c], zz, u);
            const float dx = ex + xx, dy = ey + yy, dz = ez + zz;
            neigh_hit(fmaf(dx, dx, fmaf(dy, dy, dz * dz)), rl2, j, ic[c], below, wl, rc[c], cc[c]);
          }
        }
#pragma unroll
        for (int c = 0; c < kNeighCentres; ++c)
          if (on[c] && lane == k + c) mycount = cc[c];
      }
    }
    if (lane < nb && (lane / kNeighCentres) % parts == part) d.nbr_cnt[me] = mycount;
    over |= neigh_count(d, mycount);
  }
  return over;
}

// The same for grids of 1-3 cells on an axis.  Staging: lane t of a batch
// takes candidate t of the stencil's concatenated cells (located by a binary
// search over the warp's inclusive counts) and stores (x, y, z, j), x, y, z
// fixed-point; entries past the last candidate get j = -1.
__device__ __forceinline__ bool neigh_rows_wrap(const Dev& d, const uint4* qa, float4* stg, int a0, int ni, int incl, int start,
                                                int excl, int total, float L0, float L1, float L2, float rl2, int part,
                                                int parts, bool slots) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;  // lanes under this one
  bool over = false;
  for (int ib = 0; ib < ni; ib += 32) {  // centre atoms of this cell, 32 at a time
    const int nb = min(32, ni - ib);
    const int ms = a0 + ib + min(lane, nb - 1);
    const uint4 qmine = qa[ms];  // lane k's centre
    const int me = slots ? ms : (int)qmine.w;  // and its index
    int mycount = 0;  // neighbours of lane k's centre so far
    for (int c0 = 0; c0 < total; c0 += kNStage) {  // chunks of the candidate list (warp-uniform)
      const int nch = min(kNStage, total - c0);
      const int nbat = (nch + 31) >> 5;
      __syncwarp();  // the previous chunk's readers are done
      for (int bt = 0; bt < nbat; ++bt) {
        const int t = c0 + (bt << 5) + lane;
        int lo = 0, hi = 31;
#pragma unroll
        for (int it = 0; it < 5; ++it) {  // smallest lane k with incl_k > t
          const int mid = (lo + hi) >> 1;
          const int v = __shfl_sync(kFull, incl, mid);
          if (v > t) hi = mid; else lo = mid + 1;
        }
        const int sk = __shfl_sync(kFull, start, lo);
        const int ek = __shfl_sync(kFull, excl, lo);
        float4 e = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
        if (t < total) {
          const int j = sk + (t - ek);
          const uint4 qj = qa[j];
          e = make_float4(__uint_as_float(qj.x), __uint_as_float(qj.y), __uint_as_float(qj.z),
                          slots ? __int_as_float(j) : __uint_as_float(qj.w));
        }
        stg[(bt << 5) + lane] = e;
      }
      __syncwarp();
      for (int k = 0; k < nb; ++k) {  // one centre over the staged batch (warp-uniform)
        if ((k / kNeighCentres) % parts != part) continue;
        const uint32_t xc = __shfl_sync(kFull, qmine.x, k), yc = __shfl_sync(kFull, qmine.y, k), zc = __shfl_sync(kFull, qmine.z, k);
        int cc = __shfl_sync(kFull, mycount, k);
        const int ic = __shfl_sync(kFull, me, k);
        int* const rc = d.nbr + (size_t)ic * d.W;
        for (int bt = 0; bt < nbat; ++bt) {
          const float4 e = stg[(bt << 5) + lane];
          const int j = __float_as_int(e.w);
          const float dx = fix_diff(xc, __float_as_uint(e.x), L0), dy = fix_diff(yc, __float_as_uint(e.y), L1),
                      dz = fix_diff(zc, __float_as_uint(e.z), L2);
          const float r2 = j >= 0 ? fmaf(dx, dx, fmaf(dy, dy, dz * dz)) : 1e30f;
          neigh_hit(r2, rl2, j, ic, below, d.W - 1, rc, cc);
        }
        if (lane == k) mycount = cc;
      }
    }
    if (lane < nb && (lane / kNeighCentres) % parts == part) d.nbr_cnt[me] = mycount;
    over |= neigh_count(d, mycount);
  }
  return over;
}

// The rows of cell c of the box bx; stg: the warp's kNSlice float4 of shared
// memory.  A cell may be shared by `parts` warps, each staging the stencil
// for itself and taking every parts-th group of kNeighCentres centres (a
// build with fewer cells than warps is as long as one cell's chain of
// dependent batches).  Returns whether a row was wider than its allocation.
__device__ bool neigh_cell(const Dev& d, const Box& bx, float4* stg, int c, float rl2, int part = 0, int parts = 1,
                           bool slots = false) {
  const uint4* const qa = d.tq;  // cell-sorted positions; w: the atom's index (slots: its place)
  const int lane = threadIdx.x & 31;
  const int a0 = d.cell_start[c];
  const int ni = d.cell_start[c + 1] - a0;
  if (ni <= kNeighCentres * part) return false;  // warp-uniform
  // the cell's coordinates from its first atom, by the rule that binned it
  // (three high products instead of three integer divisions)
  const uint4 o = qa[a0];
  const int cx = (int)__umulhi(o.x, (unsigned)bx.nc[0]), cy = (int)__umulhi(o.y, (unsigned)bx.nc[1]),
            cz = (int)__umulhi(o.z, (unsigned)bx.nc[2]);
  const bool frame = bx.nc[0] >= 4 && bx.nc[1] >= 4 && bx.nc[2] >= 4;  // warp-uniform
  const float L0 = bx.Lq[0], L1 = bx.Lq[1], L2 = bx.Lq[2];
  int start = 0, cnt = 0;
  if (frame) {  // lanes 0-8: the runs of three x cells (two at an x face); lanes 9-17: the cell round the face
    const int r = lane < 9 ? lane : lane - 9;
    if (lane < 18) {
      int Y = cy + r % 3 - 1, Z = cz + r / 3 - 1;
      Y += Y < 0 ? bx.nc[1] : (Y >= bx.nc[1] ? -bx.nc[1] : 0);
      Z += Z < 0 ? bx.nc[2] : (Z >= bx.nc[2] ? -bx.nc[2] : 0);
      const int row = bx.cell_off + bx.nc[0] * (Y + bx.nc[1] * Z);
      int c0 = max(cx - 1, 0), c1 = min(cx + 2, bx.nc[0]);
      if (lane >= 9) {
        c0 = cx == 0 ? bx.nc[0] - 1 : 0;
        c1 = cx == 0 ? bx.nc[0] : (cx == bx.nc[0] - 1 ? 1 : 0);
      }
      start = d.cell_start[row + c0];
      cnt = d.cell_start[row + c1] - start;
    }
  } else {
    const int nx = stencil_n(bx.nc[0]), ny = stencil_n(bx.nc[1]), nz = stencil_n(bx.nc[2]);
    if (lane < nx * ny * nz) {
      const int ox = lane % nx, oy = (lane / nx) % ny, oz = lane / (nx * ny);
      const int X = (cx + stencil_off(bx.nc[0], ox) + bx.nc[0]) % bx.nc[0];
      const int Y = (cy + stencil_off(bx.nc[1], oy) + bx.nc[1]) % bx.nc[1];
      const int Z = (cz + stencil_off(bx.nc[2], oz) + bx.nc[2]) % bx.nc[2];
      const int cc = bx.cell_off + X + bx.nc[0] * (Y + bx.nc[1] * Z);
      start = d.cell_start[cc];
      cnt = d.cell_start[cc + 1] - start;
    }
  }
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += t;
  }
  const int excl = incl - cnt;
  const int total = __shfl_sync(kFull, incl, 31);
  if (frame) {
    return neigh_rows_frame(d, qa, o, reinterpret_cast<float*>(stg), a0, ni, start, cnt, excl, total, L0, L1, L2, rl2, part, parts, slots);
  }
  return neigh_rows_wrap(d, qa, stg, a0, ni, incl, start, excl, total, L0, L1, L2, rl2, part, parts, slots);
}

__device__ __forceinline__ void neigh_cell_warp(const Dev& d, float4* stg, int c, float rl2, bool slots = false) {
  const int b = d.cell_box[c];
  if (box_flagged(d, b)) neigh_cell(d, d.box[b], stg, c, rl2, 0, 1, slots);  // warp-uniform
}

// ---------------------------------------------------------------------------
// Fused two- + three-body force (k_force).  A block holds kFAtoms centre atoms.
//   leg phase A: kG lanes per centre walk its neighbour row; the pairs with
//     r^2 < (a sig)^2 are compacted (ballot + popc within the lane group) into
//     the centre's row of a padded shared-memory leg table;
//   leg phase B: the leg terms, spread over the group's lanes: the pair term
//     is taken by the owner (half energy, full force on the centre, half
//     virial), and the leg's three-body factors go into the table and into
//     the centre's moments (below);
//   leg phase C: each leg's three-body force from the moments, one
//     red.global.add.v4.f32 to the partner, the reaction kept for the centre;
//   per-box FP64 reduction of E2, E3 and the virial.
// Leg data: u (unit vector i->j), ee = sqrt(lam eps) exp(gam sig/(r - a sig)),
// -1/2 dphi2/dr, nde = gam sig/(r - a sig)^2, r, j (tr = 2/r from r).  With c_jk = u_j.u_k and
// D_jk = c_jk - cos th0 a centre's three-body energy (Sec. II.A) is
//   E3_i = sum_{j<k} ee_j ee_k D_jk^2 = 1/2 sum_j ee_j C_j,
// and the force on leg partner j is
//   F_j = ee_j [ nde_j C_j u_j - tr_j (A_j - B_j u_j) ],
//   A_j = sum_{k!=j} ee_k D_jk u_k,  B_j = sum_{k!=j} ee_k D_jk c_jk,
//   C_j = sum_{k!=j} ee_k D_jk^2.
// Because D_jk is affine in u_j.u_k, the three sums follow exactly from the
// centre's moments S0 = sum_k ee_k, s = sum_k ee_k u_k and the symmetric
// M = sum_k ee_k u_k u_k^T (all legs, k = j included):
//   A_j = M u_j - c0 s - self u_j,  B_j = u_j.M u_j - c0 u_j.s - self c_jj,
//   C_j = u_j.M u_j - 2 c0 u_j.s + c0^2 S0 - self D_jj,
// with c0 = cos th0, c_jj = u_j.u_j, D_jj = c_jj - c0 and self = ee_j D_jj
// (the k = j term taken back out).  This is the same sum reordered: O(n) per
// centre instead of O(n^2) leg pairs.
constexpr int kG = 4;                    // lanes per centre in the leg phase
constexpr int kFThreads = 128;
constexpr int kFAtoms = kFThreads / kG;  // centres per block
constexpr int kWAtoms = 32 / kG;         // centres per warp
constexpr int kPre = 4;                  // neighbour slots per lane fetched ahead in the leg phase (k_force at 2^20 atoms:
                                         // 206 us, 208 with 6, 219 with 8)

// The force kernel's shared-memory leg table: a row of kRow float4 records
// per centre (kRow a multiple of 8, i.e. of the 8 bank groups a quarter warp's
// 16-byte accesses spread over).  Leg l of centre a sits at a kRow +
// (l ^ ((a KG) & 7)): the XOR moves the centres that share a quarter warp
// onto disjoint bank groups when their lanes step through legs l = g, g + KG,
// ... together (KG = 2 or 4; with 8 lanes a quarter warp holds one centre).
template <int kRow, int kCent = kFAtoms>
struct LegTableT {
  static_assert(kRow % 8 == 0, "rows must cover whole sets of bank groups");
  // one species: dx, dy, dz, j (int bits); several: after phase B ux, uy, uz, ee
  float4 ue[kCent * kRow];
  // phase A: the rows' pieces; then, one species: ee, -1/2 dphi, nde, 1/r;
  // several: -1/2 dphi, nde, r, j
  float4 aux[kCent * kRow];
};
using LegTable = LegTableT<kLMax>;
// Several species: a solute's larger cutoff gives its centres more legs, so
// the species instantiation stages up to 48.
constexpr int kLMaxSp = 48;
using LegTableSp = LegTableT<kLMaxSp>;

// Whole owner contribution (pair terms and three-body terms) of a centre with
// more than kLMax legs (rare): legs in local memory, every unordered leg pair
// once, same arithmetic.  Called by the centre's group leader inside k_force,
// out of line so that its local arrays and registers stay off the common path.
template <bool kCount>
__device__ __noinline__ void force_overflow_item(const Dev& d, const FParams& P, int i, int par) {
  const uint4 qi = d.q[i];
  const int b = (int)qi.w;
  const Box& bx = d.box[b];
  int cnt = d.nbr_cnt[i];
  if (cnt > d.W) cnt = d.W;
  float ux[kMaxLegsOverflow], uy[kMaxLegsOverflow], uz[kMaxLegsOverflow], tr[kMaxLegsOverflow],
      nde[kMaxLegsOverflow], ee[kMaxLegsOverflow], rr[kMaxLegsOverflow];
  float ax[kMaxLegsOverflow], ay[kMaxLegsOverflow], az[kMaxLegsOverflow];
  int jj[kMaxLegsOverflow];
  int nl = 0;
  float e2acc = 0.f, px = 0.f, py = 0.f, pz = 0.f, w[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int s = 0; s < cnt; ++s) {
    const int j = d.nbr[(size_t)i * d.W + s];
    const uint4 qj = d.q[j];
    const float dx = fix_diff(qi.x, qj.x, bx.Lq[0]), dy = fix_diff(qi.y, qj.y, bx.Lq[1]),
                dz = fix_diff(qi.z, qj.z, bx.Lq[2]);
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    if (r2 >= P.rc2) continue;
    LegTerms lt;
    if (!leg_terms(r2, P, lt)) continue;
    if (nl >= kMaxLegsOverflow) {
      set_status(d.g, ST_LEGS);
      d.g->err_index = i;
      return;
    }
    const float invr = lt.invr, r = lt.r;
    ux[nl] = dx * invr;
    uy[nl] = dy * invr;
    uz[nl] = dz * invr;
    tr[nl] = 2.0f * invr;
    nde[nl] = lt.nde;
    ee[nl] = P.sle * lt.e3;
    rr[nl] = r;
    jj[nl] = j;
    ax[nl] = ay[nl] = az[nl] = 0.f;
    {  // pair term, owner computes (half energy, full force on the centre, half virial)
      const float dphi = lt.dphi;
      e2acc = fmaf(0.5f, lt.phi, e2acc);
      px = fmaf(dphi, ux[nl], px);
      py = fmaf(dphi, uy[nl], py);
      pz = fmaf(dphi, uz[nl], pz);
      const float wv = -0.5f * dphi * r;
      w[0] = fmaf(wv * ux[nl], ux[nl], w[0]);
      w[1] = fmaf(wv * uy[nl], uy[nl], w[1]);
      w[2] = fmaf(wv * uz[nl], uz[nl], w[2]);
      w[3] = fmaf(wv * ux[nl], uy[nl], w[3]);
      w[4] = fmaf(wv * ux[nl], uz[nl], w[4]);
      w[5] = fmaf(wv * uy[nl], uz[nl], w[5]);
    }
    ++nl;
  }
  if (kCount) atomicAdd((unsigned long long*)&d.g->ntrip, (unsigned long long)(nl * (nl - 1) / 2));
  float e3acc = 0.f;
  for (int j = 0; j < nl; ++j)
    for (int k = j + 1; k < nl; ++k) {
      const float c = fmaf(ux[j], ux[k], fmaf(uy[j], uy[k], uz[j] * uz[k]));
      const float D = c - P.c0;
      const float g = ee[j] * ee[k] * D;
      e3acc = fmaf(g, D, e3acc);
      const float aj = g * tr[j], bj = g * fmaf(c, tr[j], D * nde[j]);
      ax[j] = fmaf(-aj, ux[k], fmaf(bj, ux[j], ax[j]));
      ay[j] = fmaf(-aj, uy[k], fmaf(bj, uy[j], ay[j]));
      az[j] = fmaf(-aj, uz[k], fmaf(bj, uz[j], az[j]));
      const float ak = g * tr[k], bk = g * fmaf(c, tr[k], D * nde[k]);
      ax[k] = fmaf(-ak, ux[j], fmaf(bk, ux[k], ax[k]));
      ay[k] = fmaf(-ak, uy[j], fmaf(bk, uy[k], ay[k]));
      az[k] = fmaf(-ak, uz[j], fmaf(bk, uz[k], az[k]));
    }
  float fx = 0.f, fy = 0.f, fz = 0.f;
  for (int k = 0; k < nl; ++k) {
    red_add_v4(d.f + jj[k], ax[k], ay[k], az[k]);
    fx -= ax[k];
    fy -= ay[k];
    fz -= az[k];
    const float rx = rr[k] * ux[k], ry = rr[k] * uy[k], rz = rr[k] * uz[k];
    w[0] = fmaf(rx, ax[k], w[0]);
    w[1] = fmaf(ry, ay[k], w[1]);
    w[2] = fmaf(rz, az[k], w[2]);
    w[3] = fmaf(rx, ay[k], w[3]);
    w[4] = fmaf(rx, az[k], w[4]);
    w[5] = fmaf(ry, az[k], w[5]);
  }
  red_add_v4(d.f + i, fx + px, fy + py, fz + pz);
  double* p = &d.bst[b].ew[par][0];  // rare path: per-thread FP64 atomics
  atomicAdd(p + 0, (double)e2acc);
  atomicAdd(p + 1, (double)e3acc);
  for (int k = 0; k < 6; ++k) atomicAdd(p + 2 + k, (double)w[k]);
}

// Leg phase A of one species (k_force and the adjoint): the KG lanes of a
// centre walk its neighbour row and compact the pairs with r^2 < rc2 into the
// centre's leg records tab[at(l)] = (d, j), at most kLM of them; returns how
// many there are.  The row is copied to shared memory first (kRowBuf entries
// at a time, 16 bytes a lane, into warp_aux: the warp's own second records,
// which no other warp may touch), then candidate positions are fetched
// for kPre slots per lane before any is used; every slot's test comes first,
// then one compaction per batch (the lane's hits go to the group's running
// count plus the hits of the group's lower lanes in this batch, in slot
// order).  Every lane of the warp calls it.
// k_force is bound by the L1 data pipe (80 % busy): a row entry loaded by its
// own lane, 4 bytes from each of 8 rows per warp, takes 8 times the pipe
// slots of a 16-byte copy and a conflict-free shared-memory read.
constexpr int kRowBuf = 92;  // ints a centre (of the 96 that kLMax records hold): 28 mod 32, so the 8 centres of a
                             // warp (KG = 4) read their rows from disjoint banks, in whole 16-byte pieces
__device__ __forceinline__ void cp_async16(int* dst, const int* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int KG, int kLM, class At>
__device__ __forceinline__ int stage_legs(const Dev& d, float rc2, float4* tab, At at, float4* warp_aux, const uint4& qi,
                                          float L0, float L1, float L2, const int* row, int cnt) {
  static_assert(kRowBuf * 4 <= kLM * 16 && kRowBuf % 4 == 0, "the warp's row pieces fit its second records");
  const int lane = threadIdx.x & 31;
  int* const rowbuf = reinterpret_cast<int*>(warp_aux) + (lane / KG) * kRowBuf;  // this centre's piece
  const int g = threadIdx.x & (KG - 1);
  const int longest = __reduce_max_sync(kFull, cnt);
  int nl = 0;
  for (int r0 = 0; r0 < longest; r0 += kRowBuf) {  // pieces of the rows (warp-uniform; one but for very long rows)
    const int n = min(cnt - r0, kRowBuf);  // entries of this centre's piece (may be none)
    if (r0 > 0) __syncwarp();  // the last piece's readers are done
    if ((d.W & 3) == 0) {  // rows start on 16-byte boundaries (the last copy may read past cnt, inside the row)
      for (int t = 4 * g; t < n; t += 4 * KG) cp_async16(rowbuf + t, row + r0 + t);
      cp_async_wait();
    } else {
      for (int t = g; t < n; t += KG) rowbuf[t] = row[r0 + t];
    }
    __syncwarp();
    const int iters = (min(longest - r0, kRowBuf) + KG - 1) / KG;
    for (int t0 = 0; t0 < iters; t0 += kPre) {  // warp-uniform
      uint32_t qx[kPre], qy[kPre], qz[kPre];
#pragma unroll
      for (int t = 0; t < kPre; ++t) {
        const int s = g + KG * (t0 + t);
        uint4 qj = make_uint4(0u, 0u, 0u, 0u);
        if (s < n) qj = d.q[rowbuf[s]];
        qx[t] = qj.x;
        qy[t] = qj.y;
        qz[t] = qj.z;
      }
      float dx[kPre], dy[kPre], dz[kPre];
      unsigned hits = 0u;  // bit t: slot t is a leg
      int hc = 0;
#pragma unroll
      for (int t = 0; t < kPre; ++t) {
        const int s = g + KG * (t0 + t);
        dx[t] = fix_diff(qi.x, qx[t], L0);
        dy[t] = fix_diff(qi.y, qy[t], L1);
        dz[t] = fix_diff(qi.z, qz[t], L2);
        const bool hit = s < n && fmaf(dx[t], dx[t], fmaf(dy[t], dy[t], dz[t] * dz[t])) < rc2;
        hits |= hit ? 1u << t : 0u;
        hc += hit ? 1 : 0;
      }
      int incl = hc;  // inclusive prefix of the hit counts over the group's lanes
#pragma unroll
      for (int o = 1; o < KG; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o, KG);
        if (g >= o) incl += y;
      }
      int pos = nl + incl - hc;
#pragma unroll
      for (int t = 0; t < kPre; ++t)
        if ((hits >> t) & 1u) {
          if (pos < kLM) tab[at(pos)] = make_float4(dx[t], dy[t], dz[t], __int_as_float(rowbuf[g + KG * (t0 + t)]));
          ++pos;
        }
      nl += __shfl_sync(kFull, incl, lane | (KG - 1));  // the group's hits in this batch
    }
  }
  return nl;
}

template <bool kCount>
__device__ __noinline__ int species_item(const Dev& d, const SpPair* sp, const float2* st, int nsp, int i,
                                         float (&acc)[8]);

// One block of kFAtoms centres (atoms blk*kFAtoms ...); every thread of the
// block calls it.  kSp = 0: one species.  kSp = 1: several species whose
// three-body strengths factor into leg weights (SpPair::h) and whose
// cos theta0 is the centre's (SpPair::c0); every leg carries its own pair
// constants and weight and the moments stay exact.  kSp = 2: any table;
// phase C then walks the leg pairs, each lane its own legs j against every
// other leg k of the centre (each triplet seen from both legs, each visit
// giving the force on its own leg), with lambda epsilon and cos theta0 of
// (centre; j, k) from the shared triplet table stt.  sps is the nsp^2 pair
// table in shared memory; phase A tests each candidate against its own
// pair's cutoff.
// kOwn (one species only): 0 the scatter kernel; 1 and 2 the two passes of
// owner-computes.  Pass 1 takes the legs, the pair terms (energy, force on
// the centre, virial) and each centre's moments, and stores the moments and
// the staged legs per atom.  Pass 2 recomputes the leg terms from the stored
// legs and gives each centre the three-body reaction of its own terms and
// the forces its neighbours' terms put on it (from their stored moments,
// with the leg reversed), so no leg force is scattered; centres over the
// staged-leg limit keep the scatter path (pass 1), and their neighbours add
// their own terms' forces to them by scatter.
// force_group: the 32 / KG centres of one warp (centre i of this lane's
// group; valid: there is one), ue and aux the warp's rows of the leg table;
// adds to acc (E2, E3, W xx yy zz xy xz yz) and returns the centre's box.
// over: this lane leads a centre with more legs than the table holds, which
// has added nothing; the caller hands it to force_overflow_item when its own
// sums are done with (a call with them live would spill them).  Synchronises
// the warp only.
template <bool kCount, int kSp, int KG, int kOwn>
__device__ __forceinline__ int force_group(const Dev& d, const FParams& P, float4* ue, float4* aux, int i, bool valid,
                                           float (&acc)[8], bool& over, const SpPair* sps = nullptr, int nsp = 1,
                                           const float2* stt = nullptr) {
  constexpr int kLM = kSp ? kLMaxSp : kLMax;  // legs staged per centre
  const int lane = threadIdx.x & 31;
  const int g = threadIdx.x & (KG - 1);
  const int a = lane / KG;
  const int sw = (a * KG) & 7;                                  // the row's bank-group swizzle
  auto at = [&](int l) { return a * kLM + (l ^ sw); };          // leg l of this centre
  float fx = 0.f, fy = 0.f, fz = 0.f;  // force on the centre (pair part and three-body reaction)
  uint4 qi = make_uint4(0u, 0u, 0u, 0u);
  int cnt = 0, b = -1;
  float L0 = 0.f, L1 = 0.f, L2 = 0.f;
  const SpPair* spi = nullptr;  // the centre's row of the pair table (kSp)
  int ti = 0;                   // the centre's species (kSp)
  if (valid) {
    qi = d.q[i];
    b = (int)qi.w;
    cnt = min(d.nbr_cnt[i], d.W);
    const Box& bx = d.box[b];
    L0 = bx.Lq[0];
    L1 = bx.Lq[1];
    L2 = bx.Lq[2];
    if constexpr (kSp != 0) {
      ti = d.typ[i];
      spi = sps + ti * nsp;
    }
  }
  // ---- leg phase A (stage_legs).  Several species: each candidate is tested
  // against its own pair's cutoff, slot by slot (ballot + popc in the lane
  // group), and its record is (d, r^2) and (species, j).
  const int* row = d.nbr + (size_t)(valid ? i : 0) * d.W;
  int nl = 0;
  if constexpr (kOwn == 2) {  // the legs pass 1 staged, their vectors recomputed
    const int nlg = valid ? d.nleg[i] : 0;
    nl = nlg < 0 ? 0 : nlg;
    for (int l = g; l < nl; l += KG) {
      const int j = d.legs[(size_t)i * kLMax + l];
      const uint4 qj = d.q[j];
      const float dx = fix_diff(qi.x, qj.x, L0), dy = fix_diff(qi.y, qj.y, L1), dz = fix_diff(qi.z, qj.z, L2);
      ue[at(l)] = make_float4(dx, dy, dz, __int_as_float(j));
    }
  } else if constexpr (kSp == 0) {
    nl = stage_legs<KG, kLM>(d, P.rc2, ue, at, aux, qi, L0, L1, L2, row, cnt);
  } else {
    const int iters = __reduce_max_sync(kFull, (cnt + KG - 1) / KG);
    const unsigned gsh = lane & ~(KG - 1);
    for (int t0 = 0; t0 < iters; t0 += kPre) {  // warp-uniform
      int jr[kPre], tj[kPre];
      uint32_t qx[kPre], qy[kPre], qz[kPre];
#pragma unroll
      for (int t = 0; t < kPre; ++t) {
        const int s = g + KG * (t0 + t);
        jr[t] = (s < cnt) ? row[s] : -1;
      }
#pragma unroll
      for (int t = 0; t < kPre; ++t) {
        uint4 qj = make_uint4(0u, 0u, 0u, 0u);
        tj[t] = 0;
        if (jr[t] >= 0) {
          qj = d.q[jr[t]];
          tj[t] = d.typ[jr[t]];
        }
        qx[t] = qj.x;
        qy[t] = qj.y;
        qz[t] = qj.z;
      }
#pragma unroll
      for (int t = 0; t < kPre; ++t) {
        if (t0 + t >= iters) break;
        bool hit = false;
        float dx = 0.f, dy = 0.f, dz = 0.f, r2 = 0.f;
        if (jr[t] >= 0) {
          dx = fix_diff(qi.x, qx[t], L0);
          dy = fix_diff(qi.y, qy[t], L1);
          dz = fix_diff(qi.z, qz[t], L2);
          r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          hit = r2 < spi[tj[t]].rc2;
        }
        const unsigned m = (__ballot_sync(kFull, hit) >> gsh) & ((1u << KG) - 1u);
        const int pos = nl + __popc(m & ((1u << g) - 1u));
        if (hit && pos < kLM) {  // (the pair's cutoff test needs r^2 again in phase B: kept)
          ue[at(pos)] = make_float4(dx, dy, dz, r2);
          aux[at(pos)] = make_float4(__int_as_float(tj[t]), 0.f, 0.f, __int_as_float(jr[t]));
        }
        nl += __popc(m);
      }
    }
  }
  __syncwarp();
  if constexpr (kOwn == 1) {  // the staged legs for pass 2
    for (int l = g; l < min(nl, kLM); l += KG) d.legs[(size_t)i * kLMax + l] = __float_as_int(ue[at(l)].w);
    if (valid && g == 0) d.nleg[i] = nl <= kLM ? nl : -1;
  }
  // ---- leg phase B: leg terms for the compacted legs only, spread over the
  // group's lanes: pair term (owner computes), the leg's table entry and its
  // share of the centre's moments S0, s, M.
  const int nstage = (nl <= kLM) ? nl : 0;  // larger centres: force_overflow_item does everything
  float m0 = 0.f, msx = 0.f, msy = 0.f, msz = 0.f;                            // S0, s
  float mxx = 0.f, myy = 0.f, mzz = 0.f, mxy = 0.f, mxz = 0.f, myz = 0.f;     // M
  int nvalid = 0;  // legs inside their own pair's cutoff (kSp counting)
  for (int l = g; l < nstage; l += KG) {
    float4* ue_p = ue + at(l);
    float4* ax_p = aux + at(l);
    const float4 rec = *ue_p;
    // (one species: the record is d and j; r^2 as in phase A's test)
    const float r2 = kSp ? rec.w : fmaf(rec.x, rec.x, fmaf(rec.y, rec.y, rec.z * rec.z));
    // the leg's terms with the one species' constants, or its pair's (kSp)
    LegTerms lt;
    float p_h = P.sle;
    bool in;
    if constexpr (kSp) {
      const SpPair& pp = spi[__float_as_int(ax_p->x)];
      p_h = kSp == 2 ? 1.0f : pp.h;  // kSp = 2: the strengths come per leg pair in phase C
      in = leg_terms(r2, pp, lt);
    } else {
      in = leg_terms(r2, P, lt);
    }
    if (!in) {  // FP32 rounding put it on the cutoff (or past its pair's): contributes nothing (several
                // species: the second record's r is 0 from phase A)
      (kSp ? *ue_p : *ax_p) = make_float4(0.f, 0.f, 0.f, 0.f);
      continue;
    }
    if constexpr (kSp && kCount) ++nvalid;
    const float r = lt.r;
    const float ux = rec.x * lt.invr, uy = rec.y * lt.invr, uz = rec.z * lt.invr;
    const float ee = p_h * lt.e3;
    const float dphi = kOwn == 2 ? 0.f : lt.dphi;  // (pass 2: the pair terms were taken in pass 1)
    if constexpr (kOwn != 2) {
      acc[0] = fmaf(0.5f, lt.phi, acc[0]);
      fx = fmaf(dphi, ux, fx);
      fy = fmaf(dphi, uy, fy);
      fz = fmaf(dphi, uz, fz);
    }
    if constexpr (kOwn == 1) {  // pass 1 has no phase C: the pair virial here
      const float wv = -0.5f * dphi * r;
      acc[2] = fmaf(wv * ux, ux, acc[2]);
      acc[3] = fmaf(wv * uy, uy, acc[3]);
      acc[4] = fmaf(wv * uz, uz, acc[4]);
      acc[5] = fmaf(wv * ux, uy, acc[5]);
      acc[6] = fmaf(wv * ux, uz, acc[6]);
      acc[7] = fmaf(wv * uy, uz, acc[7]);
    }
    if constexpr (kSp == 1) {
      if (p_h == 0.f) {  // no three-body weight (a lambda = 0 pair): its pair virial here, no phase C
        const float wv = -0.5f * dphi * r;
        acc[2] = fmaf(wv * ux, ux, acc[2]);
        acc[3] = fmaf(wv * uy, uy, acc[3]);
        acc[4] = fmaf(wv * uz, uz, acc[4]);
        acc[5] = fmaf(wv * ux, uy, acc[5]);
        acc[6] = fmaf(wv * ux, uz, acc[6]);
        acc[7] = fmaf(wv * uy, uz, acc[7]);
        *ue_p = make_float4(0.f, 0.f, 0.f, 0.f);
        continue;
      }
    }
    // -1/2 dphi is the pair term's share of the virial, taken in phase C
    if constexpr (kSp == 0) {
      *ax_p = make_float4(ee, -0.5f * dphi, lt.nde, lt.invr);  // (the first record stays d and j)
    } else {
      *ue_p = make_float4(ux, uy, uz, ee);
      // (kSp = 2: j with the partner's species in bits 28-30)
      const float jw = kSp == 2 ? __int_as_float(__float_as_int(ax_p->w) | (__float_as_int(ax_p->x) << 28)) : ax_p->w;
      *ax_p = make_float4(-0.5f * dphi, lt.nde, r, jw);
    }
    if constexpr (kSp == 2) continue;  // no moments
    const float ex = ee * ux, ey = ee * uy, ez = ee * uz;
    m0 += ee;
    msx += ex;
    msy += ey;
    msz += ez;
    mxx = fmaf(ex, ux, mxx);
    myy = fmaf(ey, uy, myy);
    mzz = fmaf(ez, uz, mzz);
    mxy = fmaf(ex, uy, mxy);
    mxz = fmaf(ex, uz, mxz);
    myz = fmaf(ey, uz, myz);
  }
  // the centre's moments: sum over the lane group
#pragma unroll
  for (int o = 1; o < KG; o <<= 1) {
    m0 += __shfl_xor_sync(kFull, m0, o);
    msx += __shfl_xor_sync(kFull, msx, o);
    msy += __shfl_xor_sync(kFull, msy, o);
    msz += __shfl_xor_sync(kFull, msz, o);
    mxx += __shfl_xor_sync(kFull, mxx, o);
    myy += __shfl_xor_sync(kFull, myy, o);
    mzz += __shfl_xor_sync(kFull, mzz, o);
    mxy += __shfl_xor_sync(kFull, mxy, o);
    mxz += __shfl_xor_sync(kFull, mxz, o);
    myz += __shfl_xor_sync(kFull, myz, o);
  }
  __syncwarp();  // the group's table entries are complete
  if constexpr (kOwn == 1) {
    if (valid && g == 0) {
      d.mom[3 * (size_t)i] = make_float4(m0, msx, msy, msz);
      d.mom[3 * (size_t)i + 1] = make_float4(mxx, myy, mzz, mxy);
      d.mom[3 * (size_t)i + 2] = make_float4(mxz, myz, 0.f, 0.f);
    }
  } else if constexpr (kSp == 2) {
    // ---- leg phase C (any table): leg j against every other leg k
    const float2* stc = stt + ti * nsp * nsp;
    for (int l = g; l < nstage; l += KG) {
      const float4 uj = ue[at(l)];
      const float4 xj = aux[at(l)];
      if (xj.z == 0.f) continue;  // leg dropped in phase B
      const int wj = __float_as_int(xj.w);
      const float2* stj = stc + (wj >> 28) * nsp;
      const float r = xj.z;
      const float tr = 2.0f * rcp_approx(r);
      const float nde = xj.y;
      float gx = 0.f, gy = 0.f, gz = 0.f;  // three-body force on the partner of leg j
      for (int k = 0; k < nstage; ++k) {
        const float4 uk = ue[at(k)];
        if (k == l || uk.w == 0.f) continue;
        const float2 lc = stj[__float_as_int(aux[at(k)].w) >> 28];  // (lambda eps, cos theta0)
        const float c = fmaf(uj.x, uk.x, fmaf(uj.y, uk.y, uj.z * uk.z));
        const float D = c - lc.y;
        const float gg = lc.x * uj.w * uk.w * D;
        acc[1] = fmaf(0.5f * gg, D, acc[1]);  // each triplet is visited from both of its legs
        const float aj = gg * tr, bj = gg * fmaf(c, tr, D * nde);
        gx = fmaf(-aj, uk.x, fmaf(bj, uj.x, gx));
        gy = fmaf(-aj, uk.y, fmaf(bj, uj.y, gy));
        gz = fmaf(-aj, uk.z, fmaf(bj, uj.z, gz));
      }
      red_add_v4(d.f + (wj & 0x0FFFFFFF), gx, gy, gz);
      fx -= gx;
      fy -= gy;
      fz -= gz;
      const float hx = fmaf(xj.x, uj.x, gx), hy = fmaf(xj.x, uj.y, gy), hz = fmaf(xj.x, uj.z, gz);
      const float rx = r * uj.x, ry = r * uj.y, rz = r * uj.z;
      acc[2] = fmaf(rx, hx, acc[2]);
      acc[3] = fmaf(ry, hy, acc[3]);
      acc[4] = fmaf(rz, hz, acc[4]);
      acc[5] = fmaf(rx, hy, acc[5]);
      acc[6] = fmaf(rx, hz, acc[6]);
      acc[7] = fmaf(ry, hz, acc[7]);
    }
  } else {
  // ---- leg phase C: three-body force on each leg partner from the moments
  const float c0 = (kSp && valid) ? spi[0].c0 : P.c0;
  // a centre with one leg has no three-body term: its moments hold only that
  // leg, whose self term cancels up to rounding; the residue is not computed
  const bool three = nstage > 1;  // (uniform over the centre's lane group)
  // the three-body force on the partner of leg (u, ee, nde, tr = 2/r) of a centre
  // with moments (S0, s, M), and the leg's C; the k = j term is taken back
  // out with c_jj = |u|^2 as computed (not 1), so that it cancels the same
  // product inside the moments
  auto leg_force = [&](float ux, float uy, float uz, float ee, float nde, float tr, float S0, float sx, float sy,
                       float sz, float Mxx, float Myy, float Mzz, float Mxy, float Mxz, float Myz, float& gx,
                       float& gy, float& gz) {
    const float mx = fmaf(Mxx, ux, fmaf(Mxy, uy, Mxz * uz));  // M u
    const float my = fmaf(Mxy, ux, fmaf(Myy, uy, Myz * uz));
    const float mz = fmaf(Mxz, ux, fmaf(Myz, uy, Mzz * uz));
    const float qm = fmaf(ux, mx, fmaf(uy, my, uz * mz));     // u.M u
    const float ps = fmaf(ux, sx, fmaf(uy, sy, uz * sz));     // u.s
    const float cjj = fmaf(ux, ux, fmaf(uy, uy, uz * uz));
    const float djj = cjj - c0;
    const float self = ee * djj;
    const float Bj = fmaf(-c0, ps, qm) - self * cjj;
    const float Cj = fmaf(-2.0f * c0, ps, fmaf(c0 * c0, S0, qm)) - self * djj;
    const float Ax = fmaf(-c0, sx, mx) - self * ux;
    const float Ay = fmaf(-c0, sy, my) - self * uy;
    const float Az = fmaf(-c0, sz, mz) - self * uz;
    const float et = ee * tr;                       // ee_j tr_j
    const float cu = ee * fmaf(nde, Cj, tr * Bj);   // ee_j (nde_j C_j + tr_j B_j)
    gx = fmaf(cu, ux, -et * Ax);
    gy = fmaf(cu, uy, -et * Ay);
    gz = fmaf(cu, uz, -et * Az);
    return Cj;
  };
  for (int l = g; l < nstage; l += KG) {
    const float4 rec = ue[at(l)];
    const float4 xj = aux[at(l)];
    // the leg: its unit vector u, ee, -1/2 dphi, nde, 2 / r, its vector and partner
    // (not ee: it is 0 where lambda is, or where exp(gamma sigma / (r - a sigma))
    // underflows, and such a leg has its pair virial still)
    const float ee = kSp ? rec.w : xj.x;
    if ((kSp ? xj.z : xj.w) == 0.f) continue;  // leg dropped in phase B: r, or 1 / r, left 0
    const float hd = kSp ? xj.x : xj.y, nde = kSp ? xj.y : xj.z;
    const float tr = 2.0f * (kSp ? rcp_approx(xj.z) : xj.w);
    const float3 uj = kSp ? make_float3(rec.x, rec.y, rec.z) : make_float3(rec.x * xj.w, rec.y * xj.w, rec.z * xj.w);
    const int j = __float_as_int(kSp ? xj.w : rec.w);
    float gx = 0.f, gy = 0.f, gz = 0.f;
    if (three) {
      const float Cj = leg_force(uj.x, uj.y, uj.z, ee, nde, tr, m0, msx, msy, msz, mxx, myy, mzz, mxy, mxz, myz,
                                 gx, gy, gz);
      // the partner's share: scattered (pass 2: gathered by the partner, unless
      // it is a centre over the staged-leg limit)
      if (kOwn == 0 || d.nleg[j] < 0) red_add_v4(d.f + j, gx, gy, gz);
      fx -= gx;
      fy -= gy;
      fz -= gz;
      acc[1] = fmaf(0.5f * ee, Cj, acc[1]);
    }
    if constexpr (kOwn == 2) {  // the partner's terms on this centre, from its moments, leg reversed
      if (d.nleg[j] >= 0) {
        const float4 ma = d.mom[3 * (size_t)j], mb = d.mom[3 * (size_t)j + 1], mc = d.mom[3 * (size_t)j + 2];
        float hx, hy, hz;
        if (d.nleg[j] > 1) {
          leg_force(-uj.x, -uj.y, -uj.z, ee, nde, tr, ma.x, ma.y, ma.z, ma.w, mb.x, mb.y, mb.z, mb.w, mc.x, mc.y, hx,
                    hy, hz);
          fx += hx;
          fy += hy;
          fz += hz;
        }
      }
    }
    // virial: r u_a (g_b - 1/2 dphi u_b), the three-body and the pair part
    // (pass 2: hd = 0, the pair part was taken in pass 1)
    const float hx = fmaf(hd, uj.x, gx), hy = fmaf(hd, uj.y, gy), hz = fmaf(hd, uj.z, gz);
    const float rx = kSp ? xj.z * uj.x : rec.x, ry = kSp ? xj.z * uj.y : rec.y, rz = kSp ? xj.z * uj.z : rec.z;
    acc[2] = fmaf(rx, hx, acc[2]);
    acc[3] = fmaf(ry, hy, acc[3]);
    acc[4] = fmaf(rz, hz, acc[4]);
    acc[5] = fmaf(rx, hy, acc[5]);
    acc[6] = fmaf(rx, hz, acc[6]);
    acc[7] = fmaf(ry, hz, acc[7]);
  }
  }  // phase C
  // ---- force on the centre: pair part + three-body reaction, over the group
#pragma unroll
  for (int o = 1; o < KG; o <<= 1) {
    fx += __shfl_xor_sync(kFull, fx, o);
    fy += __shfl_xor_sync(kFull, fy, o);
    fz += __shfl_xor_sync(kFull, fz, o);
  }
  if (valid && g == 0) {
    red_add_v4(d.f + i, fx, fy, fz);
    if constexpr (kSp != 0)
      if (nl > kLM) species_item<kCount>(d, sps, d.sp_tri, nsp, i, acc);  // rare: more legs than the table holds
  }
  if constexpr (kSp == 0) over = valid && g == 0 && nl > kLM;
  if (kCount && kOwn != 2) {  // legs and table-path triplets, one atomic per warp (pass 2 counts nothing)
    int nleg = nl;
    if constexpr (kSp) {  // legs inside their own pair's cutoff, summed over the group
#pragma unroll
      for (int o = 1; o < KG; o <<= 1) nvalid += __shfl_xor_sync(kFull, nvalid, o);
      nleg = nvalid;
    }
    unsigned long long legs = (valid && g == 0 && (!kSp || nl <= kLM)) ? (unsigned long long)nleg : 0ull;
    unsigned long long tri =
        (valid && g == 0 && nl <= kLM) ? (unsigned long long)(nleg * (nleg - 1) / 2) : 0ull;
    for (int o = 16; o > 0; o >>= 1) {
      legs += __shfl_down_sync(kFull, legs, o);
      tri += __shfl_down_sync(kFull, tri, o);
    }
    if (lane == 0) {
      atomicAdd((unsigned long long*)&d.g->npairs, legs);
      atomicAdd((unsigned long long*)&d.g->ntrip, tri);
    }
  }
  return b;
}

// One block of kFThreads / KG centres; every thread of the block calls it.
template <bool kCount, int kSp = 0, int KG = kG, int kOwn = 0>
__device__ void force_block(const Dev& d, const FParams& P,
                            LegTableT<(kSp ? kLMaxSp : kLMax), kFThreads / KG>& T, int blk, int par,
                            const SpPair* sps = nullptr, int nsp = 1, const float2* stt = nullptr) {
  constexpr int kRows = (32 / KG) * (kSp ? kLMaxSp : kLMax);  // records of a warp's centres
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  bool over = false;
  const int w = (int)(threadIdx.x >> 5);
  const int i = blk * (kFThreads / KG) + (int)threadIdx.x / KG;
  const int b = force_group<kCount, kSp, KG, kOwn>(d, P, T.ue + w * kRows, T.aux + w * kRows, i, i < d.N, acc, over, sps, nsp, stt);
  box_accumulate<8>(acc, b, [&](int bb) { return &d.bst[bb].ew[par][0]; });
  if constexpr (kSp == 0)
    if (over) force_overflow_item<kCount>(d, P, i, par);  // rare
}

// k_force in several launch shapes, picked by the autotuner: KG lanes per
// centre (kFThreads / KG centres per block) and a register budget of MINB
// co-resident blocks per SM (65536 / (kFThreads MINB) registers a thread).
template <bool kCount, int KG = kG, int MINB = 8, int kOwn = 0>
__global__ void __launch_bounds__(kFThreads, MINB) k_force(const __grid_constant__ Dev d, const __grid_constant__ FParams P) {
  if (block_stop(d)) return;
  __shared__ LegTableT<kLMax, kFThreads / KG> T;
  const int par = (int)(d.g->step & 1ull);
  if (blockIdx.x == 0) {  // the rebuild (if any) is consumed
    for (int k = threadIdx.x; k < d.nbox; k += blockDim.x) d.bst[k].rebuild = 0;
    if (threadIdx.x == 0) {
      d.g->any_rebuild = 0;
      d.g->wpar = par;
    }
  }
  force_block<kCount, 0, KG, kOwn>(d, P, T, blockIdx.x, par);
}

// The shapes k_force is built in: {lanes per centre, blocks per SM}.  Shape 0
// is the default; the set spans what a sweep on 2^20 atoms measured within
// 20 % of the best (2 and 8 lanes give more or fewer, larger or smaller
// blocks for small systems).
// Shape 4 is owner-computes (two passes, 4 lanes, 8 blocks per SM) against
// the scatter of the others.
constexpr int kForceShapes = 5;
__host__ __device__ constexpr int force_shape_lanes(int s) { return s == 1 ? 2 : (s == 2 ? 8 : 4); }
__host__ __device__ constexpr int force_shape_blocks(int s) { return s == 3 ? 7 : 8; }
__host__ __device__ constexpr bool force_shape_owner(int s) { return s == 4; }


// ---------------------------------------------------------------------------
// Per-phase kernels (the graph engine and the standalone force call).

// kCond (the graph engine's instantiation): the last block to finish also
// sets the condition of the graph's IF node that holds the rebuild kernels
// (skipped when no box moved more than skin/2).  The other instantiation
// holds no conditional-node call, so profilers can capture it.
// kNpt: the isobaric instantiation (rebuild margin per box, and its last
// block makes the coming step's edges current).
// k_kick1: one atom per thread.  k_kick2: kK2Items atoms per thread, atom
// (blk kK2Items + j) blockDim + t for thread t of block blk (the block's
// threads on consecutive atoms at each j), all loads first; the kinetic
// energies are summed per warp (box by box) and once per block.
constexpr int kK2Items = 4;

// k_kick1 takes a 40-register budget (6 blocks per SM): more loads in flight
// per SM than at its natural 58 registers (26 against 28.5 us at 2^20 atoms).
template <bool kCond, bool kNpt = false>
__global__ void __launch_bounds__(kKThreads, 6) k_kick1(Dev d, cudaGraphConditionalHandle rebuild_cond) {
  if (block_stop(d)) return;
  const Integ I = *d.integ;
  const int par = (int)(d.g->step & 1ull);
  const int pend = d.g->pend;
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (i < d.N) kick1_atom<kNpt>(d, I, i, par, pend, d.box, d.bst, false);
  if constexpr (kCond || kNpt) {
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) last = (bar_arrive(&d.g->done1) == gridDim.x);
    __syncthreads();
    if (last) {
      if constexpr (kNpt)
        for (int b = threadIdx.x; b < d.nbox; b += blockDim.x) npt_commit_box(d, b);
      if (threadIdx.x == 0) {
        d.g->done1 = 0u;
        if constexpr (kCond) cudaGraphSetConditional(rebuild_cond, *(volatile int*)&d.g->any_rebuild ? 1u : 0u);
      }
    }
  }
}

// a2: cell of atom i and its rank among the atoms of that cell (counting sort).
__device__ __forceinline__ void bin_item(const Dev& d, int i) {
  const uint4 q = d.q[i];
  const int c = cell_of(q, d.box[q.w]);
  d.cell[i] = c;
  d.rank[i] = atomicAdd(d.cell_cnt + c, 1);
}

// a2: atom i to its sorted slot in the staging arrays: its position with its
// index (the list is built from these), and, when the box sorts its atoms,
// the rest of its state.  Otherwise the build position is recorded here.
// start: the cells' first slots (d.cell_start, or a shared copy).
__device__ __forceinline__ void scatter_item(const Dev& d, int i, const int* start) {
  uint4 q = d.q[i];
  const int b = (int)q.w;
  if (!box_flagged(d, b)) return;
  const int p = start[d.cell[i]] + d.rank[i];
  if ((unsigned)p >= (unsigned)d.N) {  // counts not cleared after an interrupted build: report, write nothing
    set_status(d.g, ST_CELLS);
    d.g->err_index = i;
    return;
  }
  if (box_sorts(d, b)) {
    d.tx[p] = d.x[i]; d.ty[p] = d.y[i]; d.tz[p] = d.z[i];
    d.tvx[p] = d.vx[i]; d.tvy[p] = d.vy[i]; d.tvz[p] = d.vz[i];
    d.tid[p] = d.id[i];
    d.timg[p] = d.img[i];
    if (d.typ) d.ttyp[p] = d.typ[i];
    q.w = (unsigned)p;
  } else {
    d.qb[i] = q;
    q.w = (unsigned)i;
  }
  d.tq[p] = q;
}

// a2: staging arrays back to the state arrays of a box that sorts; build
// positions recorded.
__device__ __forceinline__ void copyback_item(const Dev& d, int i) {
  const int b = (int)d.q[i].w;  // a box keeps its atom range
  if (!box_flagged(d, b) || !box_sorts(d, b)) return;
  d.x[i] = d.tx[i]; d.y[i] = d.ty[i]; d.z[i] = d.tz[i];
  d.vx[i] = d.tvx[i]; d.vy[i] = d.tvy[i]; d.vz[i] = d.tvz[i];
  d.id[i] = d.tid[i];
  d.img[i] = d.timg[i];
  if (d.typ) d.typ[i] = d.ttyp[i];
  uint4 q = d.tq[i];
  q.w = (unsigned)b;
  d.q[i] = q;
  d.qb[i] = q;
}

__global__ void k_bin(Dev d) {
  if (!d.g->any_rebuild || d.g->status) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) d.g->max_count = 0;
  if (i < d.N) bin_item(d, i);
}

// Exclusive scan of the per-cell counts into cell_start (one block of 1024
// threads, 8 cells per thread per tile), zeroing the counts for the next build.
constexpr int kScanThreads = 1024;
__global__ void __launch_bounds__(kScanThreads) k_scan(Dev d) {
  if (!d.g->any_rebuild || d.g->status) return;
  __shared__ int wsum[32];
  __shared__ int carry_s;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) carry_s = 0;
  __syncthreads();
  constexpr int PER = 8;
  for (int base = 0; base < d.ncell; base += kScanThreads * PER) {
    int v[PER];
    int sum = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int c = base + tid * PER + k;
      v[k] = (c < d.ncell) ? d.cell_cnt[c] : 0;
      sum += v[k];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      int w = wsum[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, w, o);
        if (lane >= o) w += t;
      }
      wsum[lane] = w;
    }
    __syncthreads();
    int run = carry_s + (wid > 0 ? wsum[wid - 1] : 0) + incl - sum;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int c = base + tid * PER + k;
      if (c < d.ncell) {
        d.cell_start[c] = run;
        d.cell_cnt[c] = 0;
      }
      run += v[k];
    }
    __syncthreads();
    if (tid == 0) carry_s += wsum[31];
    __syncthreads();
  }
  if (tid == 0) d.cell_start[d.ncell] = carry_s;
}

__global__ void k_scatter(Dev d) {
  if (!d.g->any_rebuild || d.g->status) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < d.N) scatter_item(d, i, d.cell_start);
}

__global__ void k_copyback(Dev d) {
  if (!d.g->any_rebuild || d.g->status) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) d.g->rebuild_steps += 1;
  if (i < d.N) copyback_item(d, i);
}

constexpr int kNeighThreads = 128;
// slots: the records of d.tq carry no indices, an atom's place is its index
// (the entry point that cannot allocate).
__global__ void __launch_bounds__(kNeighThreads) k_neigh(Dev d, float rl2, bool slots) {
  if (!d.g->any_rebuild || d.g->status) return;
  __shared__ float4 stg[kNeighThreads / 32][kNSlice];
  const int w = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5);
  if (w < d.ncell) neigh_cell_warp(d, stg[threadIdx.x >> 5], w, rl2, slots);
  const int b = (int)(blockIdx.x * blockDim.x + threadIdx.x);  // (there are at least as many threads as boxes)
  if (b < d.nbox && box_flagged(d, b)) box_built(d, b);
}


// a7 second half: kinetic energy of v + a per box; the last block to finish
// runs the thermostat halves of every box (FP32, a short serial tail) and
// advances the step.  The half-kick itself stays pending.
template <bool kNpt = false>
__global__ void __launch_bounds__(kKThreads) k_kick2(Dev d) {
  if (block_stop(d)) return;
  __shared__ float s_ke[kKThreads / 32];
  __shared__ int s_box[kKThreads / 32];
  const Integ I = *d.integ;
  const unsigned long long step = d.g->step;
  const int par = (int)(step & 1ull);
  const int nwb = (int)(blockDim.x >> 5), wib = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
  // per warp: a running FP32 sum for one box; a warp whose item changes box
  // adds its sum to the old box (FP64 atomic) and starts again; an item that
  // itself straddles two boxes is added atom by atom (rare)
  float acc = 0.f;
  int cur = -1;
  float ke[kK2Items];
  int bj[kK2Items];
  {  // every item's loads first, then the arithmetic
    float4 Fj[kK2Items];
    float2 vj[kK2Items][3];
#pragma unroll
    for (int j = 0; j < kK2Items; ++j) {
      const int i = ((int)blockIdx.x * kK2Items + j) * (int)blockDim.x + (int)threadIdx.x;
      const bool act = i < d.N;
      bj[j] = act ? (d.nbox == 1 ? 0 : (int)d.q[i].w) : -1;
      Fj[j] = act ? d.f[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      vj[j][0] = act ? d.vx[i] : make_float2(0.f, 0.f);
      vj[j][1] = act ? d.vy[i] : make_float2(0.f, 0.f);
      vj[j][2] = act ? d.vz[i] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < kK2Items; ++j) {
      const float Fc[3] = {Fj[j].x, Fj[j].y, Fj[j].z};
      ke[j] = 0.f;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float u = fmaf(I.cf_f, Fc[c], vj[j][c].x) + vj[j][c].y;
        ke[j] += (float)I.ke_fac * u * u;
      }
      if (bj[j] >= 0 && !(ke[j] < 1e30f)) {
        set_status(d.g, ST_NAN);
        d.g->err_index = ((int)blockIdx.x * kK2Items + j) * (int)blockDim.x + (int)threadIdx.x;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < kK2Items; ++j) {
    const int b0 = __shfl_sync(kFull, bj[j], 0);
    if (__all_sync(kFull, bj[j] == b0 || bj[j] < 0)) {
      if (b0 < 0) continue;  // an item past the last atom (warp-uniform)
      float v = ke[j];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
      if (b0 != cur) {
        if (cur >= 0 && lane == 0) atomicAdd(&d.bst[cur].ke_acc[par], (double)acc);
        acc = 0.f;
        cur = b0;
      }
      acc += v;
    } else if (bj[j] >= 0) {
      atomicAdd(&d.bst[bj[j]].ke_acc[par], (double)ke[j]);
    }
  }
  if (lane == 0) {
    s_ke[wib] = acc;
    s_box[wib] = cur;
  }
  __syncthreads();
  if (threadIdx.x == 0) {  // the warps' sums, one FP64 atomic per run of equal boxes
    float run = 0.f;
    int rb = -1;
    for (int w = 0; w < nwb; ++w) {
      if (s_box[w] < 0) continue;
      if (s_box[w] != rb) {
        if (rb >= 0) atomicAdd(&d.bst[rb].ke_acc[par], (double)run);
        run = 0.f;
        rb = s_box[w];
      }
      run += s_ke[w];
    }
    if (rb >= 0) atomicAdd(&d.bst[rb].ke_acc[par], (double)run);
  }
  __shared__ bool am_last;
  if (threadIdx.x == 0) am_last = (bar_arrive(&d.g->done) == gridDim.x);
  __syncthreads();
  if (am_last) {
    for (int bb = threadIdx.x; bb < d.nbox; bb += blockDim.x) end_of_step_box<kNpt>(d, I, bb, par);
    __syncthreads();
    if (threadIdx.x == 0) {
      d.g->done = 0u;
      d.g->pend = 1;
      d.g->step = step + 1ull;
    }
  }
}

__global__ void k_record(Dev d) {
  const Integ I = *d.integ;
  const unsigned long long step = d.g->step;
  const int pl = (int)((step - 1ull) & 1ull);
  for (int b = threadIdx.x; b < d.nbox; b += blockDim.x) write_record(d, I, b, pl, step);
}

// Thermo record from the energies in parity slot pp (a resumed checkpoint).
__global__ void k_record_at(Dev d, int pp) {
  const Integ I = *d.integ;
  const unsigned long long step = d.g->step;
  for (int b = threadIdx.x; b < d.nbox; b += blockDim.x) write_record(d, I, b, pp, step);
}

// ---------------------------------------------------------------------------
// Setup / IO kernels.

// Applies a pending second half-kick (v += dt/2 F/m) to atom i, before
// anything changes the forces or the atom order outside a step.
__device__ __forceinline__ void flush_atom(const Dev& d, double cf, int i) {
  const float4 F = d.f[i];
  d.vx[i] = split_df(join_df(d.vx[i]) + cf * F.x);
  d.vy[i] = split_df(join_df(d.vy[i]) + cf * F.y);
  d.vz[i] = split_df(join_df(d.vz[i]) + cf * F.z);
}
// Before a force call outside a step: the accumulators of this parity and the
// counters start from zero.
__device__ __forceinline__ void prep_box(const Dev& d, int i) {
  const int par = (int)(d.g->step & 1ull);
  if (i == 0) {
    d.g->npairs = 0;
    d.g->ntrip = 0;
  }
  if (i < d.nbox)
    for (int k = 0; k < 8; ++k) d.bst[i].ew[par][k] = 0.0;
}
// New positions for the current atom order (mw_energy_forces_dev): from a
// user-order AoS device array into the sorted arrays, x[i] = xin[id[i]],
// wrapped into [0, L); q recomputed.  Also flags every box for a rebuild and
// does what k_prep_force does (one launch instead of four: a small box's
// force call is as long as its launches).
__global__ void k_load_positions(Dev d, const double* __restrict__ xin, const int* __restrict__ boxid) {
  __shared__ BlockEdges S;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  prep_box(d, i);
  if (i < d.nbox) {  // every list is stale
    d.bst[i].rebuild = 1;
    d.bst[i].sorted = 0;
  }
  if (i == 0) d.g->any_rebuild = 1;
  const int u = i < d.N ? d.id[i] : 0;
  const int b = i < d.N ? boxid[u] : -1;
  block_edges(S, d.box, b);
  if (i >= d.N) return;
  if (d.g->pend) flush_atom(d, d.integ->cf, i);
  d.f[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  unsigned long long p[3];
  int im[3];
  for (int k = 0; k < 3; ++k) {
    double v = xin[3 * (size_t)u + k];
    if (!isfinite(v)) {  // reported to the host, which refuses the state; 0 keeps the arithmetic defined
      set_status(d.g, ST_INPUT);
      d.g->err_index = u;
      v = 0.0;
    }
    p[k] = edge_fraction(S, d.box, b, k, v, im[k]);
  }
  d.x[i] = p[0]; d.y[i] = p[1]; d.z[i] = p[2];
  if (d.img) d.img[i] = make_int4(im[0], im[1], im[2], 0);
  d.q[i] = make_uint4(q_of(p[0]), q_of(p[1]), q_of(p[2]), (unsigned)b);
}

// Fixed-point copies of restored positions (checkpoint resume): q and the
// build positions qb from the 64-bit fractions, the box from the atom's id.
__global__ void k_requantize(Dev d, const int* __restrict__ boxid) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= d.N) return;
  const uint4 q = make_uint4(q_of(d.x[i]), q_of(d.y[i]), q_of(d.z[i]), (unsigned)boxid[d.id[i]]);
  d.q[i] = q;
  d.qb[i] = q;
}

// A new state in one pass (mw_set_state): atom i takes the caller's atom i
// (identity order), its species, its velocity (zero when vin is null) and
// zero force, and adds its kinetic energy to its box's ke_last; the cell
// counts are cleared.  The host zeroes the box states and the status block
// before the launch; here each box is marked for a rebuild with no pending
// end scale, and the status block gets the rebuild flag and count_terms.  A
// non-finite value is replaced by 0 and reported (ST_INPUT, the atom in
// err_index); the host refuses the state.
__global__ void k_load_state(Dev d, const double* __restrict__ xin, const double* __restrict__ vin,
                             const int* __restrict__ boxid, int count_terms) {
  const Integ I = *d.integ;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < d.ncell) d.cell_cnt[i] = 0;
  if (i < d.nbox) {
    d.bst[i].s_endc = 1.0;
    d.bst[i].rebuild = 1;
  }
  if (i == 0) {
    d.g->any_rebuild = 1;
    d.g->count_terms = count_terms;
  }
  __shared__ BlockEdges S;
  float ke[1] = {0.f};
  const int b = i < d.N ? boxid[i] : -1;
  block_edges(S, d.box, b);
  if (i < d.N) {
    d.id[i] = i;
    unsigned long long p[3];
    int im[3];
    float vh[3];
    for (int k = 0; k < 3; ++k) {
      double x = xin[3 * (size_t)i + k];
      if (!isfinite(x)) {
        set_status(d.g, ST_INPUT);
        d.g->err_index = i;
        x = 0.0;
      }
      p[k] = edge_fraction(S, d.box, b, k, x, im[k]);
      double w = vin ? vin[3 * (size_t)i + k] : 0.0;
      if (!isfinite(w)) {
        set_status(d.g, ST_INPUT);
        d.g->err_index = i;
        w = 0.0;
      }
      const float2 sw = split_df(w);
      (k == 0 ? d.vx : (k == 1 ? d.vy : d.vz))[i] = sw;
      vh[k] = sw.x + sw.y;
    }
    d.x[i] = p[0];
    d.y[i] = p[1];
    d.z[i] = p[2];
    if (d.img) d.img[i] = make_int4(im[0], im[1], im[2], 0);
    d.q[i] = make_uint4(q_of(p[0]), q_of(p[1]), q_of(p[2]), (unsigned)b);
    if (d.typ) d.typ[i] = d.utyp[i];
    d.f[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    ke[0] = (float)I.ke_fac * fmaf(vh[0], vh[0], fmaf(vh[1], vh[1], vh[2] * vh[2]));
  }
  box_accumulate<1>(ke, b, [&](int bb) { return &d.bst[bb].ke_last; });
}

// A new state in the current atom order (mw_set_state while that order and
// the neighbour lists are current): sorted slot i takes the caller's atom
// id[i] with the same conversions as k_load_state (positions to 64-bit and
// fixed-point fractions, image counts, velocities as FP32 pairs, species,
// zero force, kinetic energy per box).  A box keeps its list when every one
// of its atoms lies within half the skin (hs2 = (skin/2)^2) of the position
// the list was built at, as between steps; any other box is flagged for a
// rebuild.  The host zeroes the box states and the status block (all but
// the widest-row record) before the launch.
// Per-atom parts of k_load_state_keep: slot i's position (fractions, image
// counts, fixed-point copy, species, zero force, the rebuild flag of its
// box) and its velocity (FP32 pair; returns its kinetic energy).
__device__ __forceinline__ void load_keep_position(const Dev& d, const BlockEdges& S, const double* __restrict__ xin, int i,
                                                   float hs2) {
  const int u = d.id[i];
  const int b = (int)d.q[i].w;
  const Box& bx = d.box[b];
  unsigned long long p[3];
  int im[3];
  for (int k = 0; k < 3; ++k) {
    double x = xin[3 * (size_t)u + k];
    if (!isfinite(x)) {
      set_status(d.g, ST_INPUT);
      d.g->err_index = u;
      x = 0.0;
    }
    p[k] = edge_fraction(S, d.box, b, k, x, im[k]);
  }
  d.x[i] = p[0];
  d.y[i] = p[1];
  d.z[i] = p[2];
  if (d.img) d.img[i] = make_int4(im[0], im[1], im[2], 0);
  const uint4 q = make_uint4(q_of(p[0]), q_of(p[1]), q_of(p[2]), (unsigned)b);
  d.q[i] = q;
  if (d.typ) d.typ[i] = d.utyp[u];
  d.f[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  const uint4 qb = d.qb[i];
  const float dx = fix_diff(qb.x, q.x, bx.Lq[0]), dy = fix_diff(qb.y, q.y, bx.Lq[1]), dz = fix_diff(qb.z, q.z, bx.Lq[2]);
  if (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) > hs2) {
    d.bst[b].rebuild = 1;
    d.g->any_rebuild = 1;
  }
}

__device__ __forceinline__ float load_keep_velocity(const Dev& d, const Integ& I, const double* __restrict__ vin,
                                                    int i) {
  const int u = d.id[i];
  float vh[3];
  for (int k = 0; k < 3; ++k) {
    double w = vin ? vin[3 * (size_t)u + k] : 0.0;
    if (!isfinite(w)) {
      set_status(d.g, ST_INPUT);
      d.g->err_index = u;
      w = 0.0;
    }
    const float2 sw = split_df(w);
    (k == 0 ? d.vx : (k == 1 ? d.vy : d.vz))[i] = sw;
    vh[k] = sw.x + sw.y;
  }
  return (float)I.ke_fac * fmaf(vh[0], vh[0], fmaf(vh[1], vh[1], vh[2] * vh[2]));
}

__global__ void k_load_state_keep(Dev d, const double* __restrict__ xin, const double* __restrict__ vin,
                                  int count_terms, float hs2) {
  const Integ I = *d.integ;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < d.ncell) d.cell_cnt[i] = 0;
  if (i < d.nbox) {
    d.bst[i].s_endc = 1.0;
    d.bst[i].Lb = d.box[i].L[0];  // the lists were built in these (unscaled) boxes
  }
  if (i == 0) d.g->count_terms = count_terms;
  __shared__ BlockEdges S;
  float ke[1] = {0.f};
  const int b = i < d.N ? (int)d.q[i].w : -1;
  block_edges(S, d.box, b);
  if (i < d.N) {
    load_keep_position(d, S, xin, i, hs2);
    ke[0] = load_keep_velocity(d, I, vin, i);
  }
  box_accumulate<1>(ke, b, [&](int bb) { return &d.bst[bb].ke_last; });
}

// The same in two launches, positions first (k_load_positions_keep: no
// velocity or kinetic energy is touched) and velocities later
// (k_load_velocities_keep: the kinetic energy into ke_last, which the host
// zeroed with the box states), so that a force call at the new positions can
// run between them while the velocities are still being copied in.
__global__ void k_load_positions_keep(Dev d, const double* __restrict__ xin, int count_terms, float hs2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < d.ncell) d.cell_cnt[i] = 0;
  if (i < d.nbox) {
    d.bst[i].s_endc = 1.0;
    d.bst[i].Lb = d.box[i].L[0];
  }
  if (i == 0) d.g->count_terms = count_terms;
  __shared__ BlockEdges S;
  block_edges(S, d.box, i < d.N ? (int)d.q[i].w : -1);
  if (i < d.N) load_keep_position(d, S, xin, i, hs2);
}

__global__ void k_load_velocities_keep(Dev d, const double* __restrict__ vin) {
  const Integ I = *d.integ;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  float ke[1] = {0.f};
  int b = -1;
  if (i < d.N) {
    b = (int)d.q[i].w;
    ke[0] = load_keep_velocity(d, I, vin, i);
  }
  box_accumulate<1>(ke, b, [&](int bb) { return &d.bst[bb].ke_last; });
}

__global__ void k_flush_pending(Dev d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (d.g->pend && i < d.N) flush_atom(d, d.integ->cf, i);
}

// Flags every box for a rebuild (new state, parameters, skin or list width).
__global__ void k_flag_all(Dev d) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < d.nbox) {
    d.bst[b].rebuild = 1;
    d.bst[b].sorted = 0;
  }
  if (b == 0) d.g->any_rebuild = 1;
}

// Blocks of the standalone kick kernels: `items` atoms per thread.
__host__ __device__ inline int kick_blocks(int n, int threads, int items = 1) {
  const int per = threads * items;
  return (n + per - 1) / per;
}

// The same with the forces (mode 1 to 3), a pending half-kick applied with the
// old ones first (mode 2: the host clears Global::pend after the launch).
// Mode 3 leaves everything as it is under a status, under which no force
// kernel runs either: the valid forces of an isobaric box that left its cell
// grid stay those of its last step.
__global__ void k_prep_force(Dev d, int mode) {
  if (mode == 3 && *(volatile int*)&d.g->status) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  prep_box(d, i);
  if (mode > 0 && i < d.N) {
    if (mode == 2 && d.g->pend) flush_atom(d, d.integ->cf, i);
    d.f[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// Thermo record from the current accumulators without advancing (forces just
// evaluated).
__device__ __forceinline__ void thermo_snapshot(const Dev& d, int b) {
  const Integ& I = *d.integ;
  const int par = (int)(d.g->step & 1ull);
  const BoxState* st = d.bst + b;
  const Box& bx = d.box[b];
  double* t = d.thermo + (size_t)b * TR_N;
  const double ke = st->ke_last;
  const double e2 = st->ew[par][0], e3 = st->ew[par][1];
  t[TR_STEP] = (double)d.g->step;
  t[TR_PE] = e2 + e3;
  t[TR_E2] = e2;
  t[TR_E3] = e3;
  t[TR_KE] = ke;
  t[TR_T] = 2.0 * ke * bx.inv_ndf_kb;
  double cons = ke + e2 + e3;
  const double xi = (double)st->th_e.x + (double)st->th_e.y, eta = (double)st->th_e.z + (double)st->th_e.w;
  if (I.kind == TH_NH || I.kind == TH_NPT) cons += 0.5 * bx.Q * xi * xi + bx.ndfkT0 * eta;
  if (I.kind == TH_NPT) cons += I.p_ext * bx.volume + 0.5 * st->pe_e * st->pe_e / bx.W;
  t[TR_CONS] = cons;
  t[TR_P] = (2.0 * ke + st->ew[par][2] + st->ew[par][3] + st->ew[par][4]) / (3.0 * bx.volume) * kATM;
  for (int k = 0; k < 6; ++k) t[TR_W0 + k] = st->ew[par][2 + k];
  t[TR_XI] = xi;
  t[TR_ETA] = eta;
  t[TR_REBUILDS] = (double)st->rebuilds;
  t[TR_VOL] = bx.volume;
  for (int k = 0; k < 3; ++k) t[TR_L0 + k] = bx.L[k];
}

// Sorted -> user order: x (wrapped) and (v + pending half-kick) * s_endc (the
// end scale of the last step, pending on the stored velocities).
__global__ void k_gather_state(Dev d, double* __restrict__ xo, double* __restrict__ vo, int unwrap) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= d.N) return;
  const int u = d.id[i];
  const Box& bx = d.box[d.q[i].w];
  if (xo) {
    constexpr double k2m64 = 5.421010862427522170037264e-20;  // 2^-64
    if (unwrap) {
      const int4 im = d.img[i];
      xo[3 * (size_t)u] = (__ull2double_rn(d.x[i]) * k2m64 + im.x) * bx.L[0];
      xo[3 * (size_t)u + 1] = (__ull2double_rn(d.y[i]) * k2m64 + im.y) * bx.L[1];
      xo[3 * (size_t)u + 2] = (__ull2double_rn(d.z[i]) * k2m64 + im.z) * bx.L[2];
    } else {
      xo[3 * (size_t)u] = fraction_times(d.x[i], bx.L[0]);
      xo[3 * (size_t)u + 1] = fraction_times(d.y[i], bx.L[1]);
      xo[3 * (size_t)u + 2] = fraction_times(d.z[i], bx.L[2]);
    }
  }
  if (vo) {  // pending half-kick and end-of-step thermostat scale applied
    const double s = d.bst[d.q[i].w].s_endc;
    const double cf = d.g->pend ? d.integ->cf : 0.0;
    const float4 F = d.f[i];
    vo[3 * (size_t)u] = (join_df(d.vx[i]) + cf * widen(F.x)) * s;
    vo[3 * (size_t)u + 1] = (join_df(d.vy[i]) + cf * widen(F.y)) * s;
    vo[3 * (size_t)u + 2] = (join_df(d.vz[i]) + cf * widen(F.z)) * s;
  }
}

// Forces to user order.
__device__ __forceinline__ void gather_force(const Dev& d, int i, double* __restrict__ fo64, float* __restrict__ fo32) {
  const int u = d.id[i];
  const float4 F = d.f[i];
  if (fo64) {
    fo64[3 * (size_t)u] = F.x;
    fo64[3 * (size_t)u + 1] = F.y;
    fo64[3 * (size_t)u + 2] = F.z;
  }
  if (fo32) {
    fo32[3 * (size_t)u] = F.x;
    fo32[3 * (size_t)u + 1] = F.y;
    fo32[3 * (size_t)u + 2] = F.z;
  }
}

// Neighbour sets to user order: out[u*width + s] = id[nbr[i][s]].
__global__ void k_gather_neighbors(Dev d, int* __restrict__ cnt_out, int* __restrict__ nbr_out, int width) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= d.N) return;
  const int u = d.id[i];
  const int c = d.nbr_cnt[i];
  cnt_out[u] = c;
  const int m = min(min(c, d.W), width);
  for (int s = 0; s < m; ++s) nbr_out[(size_t)u * width + s] = d.id[d.nbr[(size_t)i * d.W + s]];
}

// Energies and virial of the latest force evaluation: the parity slot that
// evaluation wrote (wpar).  After a step the step counter has moved on and
// its own parity names the slot the next step clears, not this one.
__device__ __forceinline__ void energy_out(const Dev& d, int b, double* e, double* w) {
  const int par = d.g->wpar;
  const BoxState* st = d.bst + b;
  if (e) {
    e[3 * b] = st->ew[par][0] + st->ew[par][1];
    e[3 * b + 1] = st->ew[par][0];
    e[3 * b + 2] = st->ew[par][1];
  }
  if (w)
    for (int k = 0; k < 6; ++k) w[6 * b + k] = st->ew[par][2 + k];
}

// What a force call returns, in one launch: the forces and the energies and
// virials, any of them null, and the thermo records of a force call just made
// (snapshot).  Nothing after a device error: a fresh call has evaluated
// nothing then, and of earlier forces the host reports the error.  An isobaric
// box that left its cell grid (ST_GRID) did so at a step boundary, whose
// forces are valid.
struct ForceOut {
  double* f64 = nullptr;
  float* f32 = nullptr;
  double* e = nullptr;
  double* w = nullptr;
};
__global__ void k_force_out(Dev d, ForceOut o, bool snapshot) {
  const int st = *(volatile int*)&d.g->status;
  if (st && (snapshot || st != ST_GRID)) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < d.nbox) {
    if (snapshot) thermo_snapshot(d, i);
    if (o.e || o.w) energy_out(d, i, o.e, o.w);
  }
  if ((o.f64 || o.f32) && i < d.N) gather_force(d, i, o.f64, o.f32);
}

}  // namespace mw

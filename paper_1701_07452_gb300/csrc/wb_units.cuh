// Device "units" of the CTU+CT MHDTVD step (Sec. "MHD in Three Dimensions",
// Steps 1-11 with the App. A flux): one function per stage, each working on
// one index (zone, face, edge or sweep tile) of one box.  The per-stage
// kernels of a grid (wb_stages.cu, wb_sweep.cu) and the persistent batch
// kernel (wb_batch.cu) call the same functions.
#pragma once
#include "wb_device.cuh"

// Field pointers of one box (or one patch slot).  F[d][F_BX + d] is unused.
struct WbView {
  WbGeo geo;
  double* q[8];
  double* b[3];
  double* Fp[3][8];
  double* Fc[3][8];
  double* Eref[3];
  double* Eedge[3];
  double* bh[3];
  double* qh[3][8];
  double* Erefh[3];
  double* Eedgeh[3];
  WbScalars* scal;
};

namespace wbu {

// ---------------------------------------------------------------- sweep ----
constexpr int kWarps = 4;             // warps of a sweep block
constexpr int kBlock = 32 * kWarps;
constexpr int kTile = kBlock - 3;     // faces a block emits from its kBlock zones
// resident blocks per SM the sweep kernels are compiled for: 128 registers a
// thread, 16 warps per SM (3 blocks, 168 registers and fewer spills: 17.8
// against 17.4 ms a launch of a 256^3 box, 2.21 against 2.07 of a 128^3)
constexpr int kSweepBlocks = 4;

// waves 2, 4, 6 (Alfven, entropy, Alfven) have eps = 0 (the default eps_k):
// the mask of the sweep specialisation that drops their Q-branch arithmetic
constexpr int kEpsZeroLD = (1 << 1) | (1 << 3) | (1 << 5);

struct Cell {
  double rho, ir, sr;             // rho, 1/rho, sqrt(rho)
  double vn, vt1, vt2;
  double bt1, bt2;
  double eref;                    // E - bn^2/2 (energy referred to the face field)
  double hr;                      // (gamma/(gamma-1) P + rho v^2/2 + |Bt|^2) / rho
  double F[7];                    // half the Sec. 3 flux (rho, Mn, Mt1, Mt2, Bt1, Bt2, E)
  double mn, mt1, mt2;
};

// Loads of fields a launch only reads may use the non-coherent read-only path
// (NC = true); the persistent batch kernel writes the same arrays in other
// stages of one launch and uses coherent loads (NC = false).
template <bool NC>
__device__ __forceinline__ double ld(const double* p) {
  if (NC) return __ldg(p);
  return *p;
}

// A product of the sweeps: on the integer pipes (SOFT) or the FP64 pipe, the
// same bits wherever the product is zero or of magnitude 2^-1021 and up (below,
// the integer form gives zero).  The integer form neither looks for infinities and
// NaN nor for overflow: a sweep takes it where every zone field and face field is zero
// or of magnitude between 2^-100 and 2^50, the density between 2^-50 and 2^50, dt/dx
// between 2^-100 and 2^50 (FieldRange) and the Roe state's a^2 above 2^-100
// (face_system).  No product then leaves the range upwards: with |v| < 2^100, a^2 <
// 2^204, every alpha_k < 2^356, |nu_k| < 2^155, g-tilde < 2^668, the sum of beta_k R_k
// below 2^920.  Downwards, a difference of two fields is zero or 2^-152 and up, and
// the longest product, w^2 in the band of beta_k, has dt/dx, a speed, a field and a
// difference twice each, 2^-904 for unit density: one below 2^-1021 takes rounding
// residues as factors several times over.
template <bool SOFT, int KNOWN = 0>
__device__ __forceinline__ double mul(double x, double y) {
  return SOFT ? wb_smul_finite<KNOWN>(x, y) : __dmul_rn(x, y);
}
// Reciprocals and roots of values those bounds keep normal (the FP64 form of a
// sweep, which meets everything else, looks at its inputs).
template <bool SOFT>
__device__ __forceinline__ double recip(double x) {
  return SOFT ? wb_rcp_sure(x) : wb_rcp(x);
}
template <bool SOFT>
__device__ __forceinline__ WbRoots roots(double x) {
  return SOFT ? wb_roots_sure(x) : wb_roots(x);
}

// The range of the fields a thread takes in (magnitudes, by twice their high words;
// zero counts as none; a bit below says that the low word is not zero, so that the
// smallest subnormals do not pass for it).
struct FieldRange {
  unsigned most = 0, least = 0xffffffffu;
  __device__ __forceinline__ void add(double x) {
    const unsigned u = (wb_hi32(x) << 1) + min(wb_lo32(x), 1u);
    most = max(most, u);
    least = min(least, u - 1u);
  }
  // Fields of other magnitudes go to the FP64 products (NaN and infinities too).
  // Nonzero fields below 2^-100 did not before; their products' flush to zero then
  // gave a grid of 32^3 zones with a tail of 2^-1000 other bits than its patches.
  __device__ __forceinline__ bool wild(double rho) const {
    return most >= ((1023u + 50u) << 21) || least < ((1023u - 100u) << 21) - 1u ||
           wb_hi32(rho) - ((1023u - 50u) << 20) >= (100u << 20);
  }
};

// Zone state of a sweep.  The arithmetic is written with explicit rounding
// (no contraction left to the compiler): several kernels and both forms of
// the products inline it, and all must round identically, or a face's flux would
// depend on how a box is split and launched.
// q: the fields in the sweep's frame (rho, Mn, Mt1, Mt2, E, Bn, Bt1, Bt2).
template <bool NC, bool SOFT>
__device__ __forceinline__ FieldRange load_cell(const double* const (&q)[8], long long off, const WbPhys& P, Cell& c) {
  c.rho = ld<NC>(q[0] + off);
  c.mn = ld<NC>(q[1] + off);
  c.mt1 = ld<NC>(q[2] + off);
  c.mt2 = ld<NC>(q[3] + off);
  const double e = ld<NC>(q[4] + off);
  const double bn = ld<NC>(q[5] + off);
  c.bt1 = ld<NC>(q[6] + off);
  c.bt2 = ld<NC>(q[7] + off);
  FieldRange range;
  range.add(c.mn);
  range.add(c.mt1);
  range.add(c.mt2);
  range.add(e);
  range.add(bn);
  range.add(c.bt1);
  range.add(c.bt2);
  const WbRoots rr = roots<SOFT>(c.rho);
  c.sr = rr.sq;
  c.ir = rr.rcp;
  c.vn = mul<SOFT, 2>(c.mn, c.ir);
  c.vt1 = mul<SOFT, 2>(c.mt1, c.ir);
  c.vt2 = mul<SOFT, 2>(c.mt2, c.ir);
  const double hbn = wb_half(bn), bn2 = mul<SOFT>(bn, bn);
  const double ke = wb_half(__fma_rn(c.mt2, c.vt2, __fma_rn(c.mt1, c.vt1, mul<SOFT>(c.mn, c.vn))));
  const double bt2 = __fma_rn(c.bt2, c.bt2, mul<SOFT>(c.bt1, c.bt1));
  const double me = wb_half(__dadd_rn(bn2, bt2));
  const double p = __dmul_rn(P.gm1, __dsub_rn(__dsub_rn(e, ke), me));
  const double pstar = __dadd_rn(p, me);
  const double ep = __dadd_rn(e, pstar);
  c.eref = __dsub_rn(e, wb_half(bn2));
  // rho h = gamma/(gamma-1) P + rho v^2/2 + |B_t|^2 = (E + P*) - B_n^2
  c.hr = __dmul_rn(__dsub_rn(ep, bn2), c.ir);
  // half fluxes: the face needs (F_L + F_R) / 2
  const double hmn = wb_half(c.mn), hvn = wb_half(c.vn);
  c.F[0] = hmn;
  c.F[1] = __fma_rn(hmn, c.vn, wb_half(__dsub_rn(pstar, bn2)));
  c.F[2] = __fma_rn(hmn, c.vt1, -mul<SOFT>(c.bt1, hbn));
  c.F[3] = __fma_rn(hmn, c.vt2, -mul<SOFT>(c.bt2, hbn));
  c.F[4] = __fma_rn(c.bt1, hvn, -mul<SOFT>(c.vt1, hbn));
  c.F[5] = __fma_rn(c.bt2, hvn, -mul<SOFT>(c.vt2, hbn));
  const double bv = __fma_rn(c.bt2, c.vt2, __fma_rn(c.bt1, c.vt1, mul<SOFT>(bn, c.vn)));
  c.F[6] = __fma_rn(ep, hvn, __dmul_rn(-hbn, bv));
  return range;
}

// Per-face record.
// R_PG = rho a^2 / (gamma-1); R_KX = (gamma-2)/(gamma-1) X - v^2/2 (= K - v^2 for the
// K = v^2/2 + (gamma-2)/(gamma-1) X of the energy row);
// R_AFCF = alpha_f c_f, R_ASCS = alpha_s c_s.
enum {
  R_AL = 0, R_NU = 7, R_RHO = 14, R_SRHO, R_A, R_PG, R_CF, R_ASCS, R_AFCF, R_AF, R_AS, R_B1, R_B2,
  R_VN, R_VT1, R_VT2, R_BTM, R_KX, R_FAVG, R_WORDS = R_FAVG + 7
};

// A face record in registers (every index a constant after unrolling).
struct RegRec {
  mutable double w[R_WORDS];
  __device__ __forceinline__ double& operator[](int i) const { return w[i]; }
};

// The flux arithmetic below is written with explicit rounding: every product
// that feeds a sum is one fused multiply-add (__fma_rn), every other operation
// is rounded on its own (__dmul_rn, __dadd_rn, __dsub_rn), and nothing is left
// to the compiler's contraction.  An interface then gives the same bits in
// every kernel this code is inlined into (the grid sweeps, both forms of the
// batch path), whatever else the kernel holds.  Shorthands:
#define WB_FMA __fma_rn
#define WB_MUL __dmul_rn
#define WB_ADD __dadd_rn
#define WB_SUB __dsub_rn

// Q_k(nu) - nu^2 for the g-tilde of App. A.  Waves in the compile-time mask
// EZ have eps_k = 0, where Q is |nu|; the branch test runs on the integer pipe.
template <int EZ, bool SOFT>
__device__ __forceinline__ double Qk_m_nu2(double nu, int k, const WbPhys& P) {
  if (EZ & (1 << k)) return WB_FMA(-nu, nu, wb_fabs(nu));
  // |nu| - nu^2, or for |nu| < 2 eps nu^2 / (4 eps) + eps - nu^2 = nu^2 (1/(4 eps) - 1) + eps:
  // one FMA of operands chosen on the integer pipe, FMA(x, nu, y) with (x, y) = (-nu, |nu|)
  // or (nu (1/(4 eps) - 1), eps), so that no warp issues both forms
  const bool band = wb_abs_less(nu, P.two_eps[k]);
  const double x = band ? mul<SOFT>(nu, P.inv4eps_m1[k]) : wb_flip(nu);
  return WB_FMA(x, nu, band ? P.eps[k] : wb_fabs(nu));
}

// Gas pressure of a zone from its sweep-frame fields (Sec. 3, Eq. totenergy)
__device__ __forceinline__ double zone_pressure(const Cell& c, const WbPhys& P) {
  const double mv = WB_FMA(c.mt2, c.vt2, WB_FMA(c.mt1, c.vt1, WB_MUL(c.mn, c.vn)));
  const double bb = WB_FMA(c.bt2, c.bt2, WB_MUL(c.bt1, c.bt1));
  return WB_MUL(P.gm1, WB_SUB(WB_SUB(c.eref, wb_half(mv)), wb_half(bb)));
}

// Protection floor of App. A: true when a zone state, or an intermediate
// state w_L + sum_{j<=k} alpha_j r_j of the linearised Riemann problem, has a
// density or pressure below the floors.  The density / pressure rows of r_k
// (k = 1..6) are rho_ af / rho_ a^2 af, 0 / 0, rho_ as / rho_ a^2 as, 1 / 0,
// rho_ as / rho_ a^2 as, 0 / 0.
__device__ __forceinline__ bool protection_hit(const Cell& L, const Cell& R, double rho, double ra2,
                                               double af, double as, const double al[7],
                                               const WbPhys& P) {
  const double pL = zone_pressure(L, P), pR = zone_pressure(R, P);
  if (L.rho < P.prot_rho || pL < P.prot_p || R.rho < P.prot_rho || pR < P.prot_p) return true;
  const double r1 = WB_FMA(al[0], WB_MUL(rho, af), L.rho), p1 = WB_FMA(al[0], WB_MUL(ra2, af), pL);
  if (r1 < P.prot_rho || p1 < P.prot_p) return true;
  const double r3 = WB_FMA(al[2], WB_MUL(rho, as), r1), p3 = WB_FMA(al[2], WB_MUL(ra2, as), p1);
  if (r3 < P.prot_rho || p3 < P.prot_p) return true;
  const double r4 = WB_ADD(r3, al[3]);
  if (r4 < P.prot_rho) return true;
  const double r5 = WB_FMA(al[4], WB_MUL(rho, as), r4), p5 = WB_FMA(al[4], WB_MUL(ra2, as), p3);
  return r5 < P.prot_rho || p5 < P.prot_p;
}

// Fast speed of one zone along the sweep axis with its own zone field (Sec. 3)
__device__ __forceinline__ double zone_fast_speed(const Cell& c, double bn, const WbPhys& P) {
  const double a2 = WB_MUL(P.gamma, zone_pressure(c, P)) / c.rho;
  const double bn2 = WB_MUL(bn, bn);
  const double b2 = WB_FMA(c.bt2, c.bt2, WB_FMA(c.bt1, c.bt1, bn2)) / c.rho;
  const double s = WB_ADD(a2, b2);
  double disc = WB_FMA(s, s, -(WB_MUL(WB_MUL(4.0, a2), bn2) / c.rho));
  if (disc < 0.0) disc = 0.0;
  return sqrt(wb_half(WB_ADD(s, sqrt(disc))));
}

// HLL flux of App. A of one face:
//   b+ = max(a_max, vR + cfR, 0), b- = min(a_min, vL - cfL, 0),
//   u = (b+ F_L - b- F_R + b+ b- (q_R - q_L)) / (b+ - b-),
// with a_max, a_min = vn_ +- cf_ of the Roe state when it exists (roe), the
// Einfeldt sign of the F_R term (the printed +b- F_R is not consistent), and
// bounds +-max(|v| + c_f) if both speeds vanish.  Rare path.
//
// The zones are loaded again: this path is rare, and its use of both zone states
// would keep 40 doubles of every thread in registers through face_system.  vn,
// cf: of the Roe state (roe).  The interface's flux in out.
template <bool NC>
__device__ __noinline__ void hll_face(const double* const (&q)[8], long long offL, long long offR, bool roe, double vn,
                                      double cf, const WbPhys& P, double* out) {
  Cell L, R;
  load_cell<NC, false>(q, offL, P, L);
  load_cell<NC, false>(q, offR, P, R);
  const double cfL = zone_fast_speed(L, ld<NC>(q[5] + offL), P), cfR = zone_fast_speed(R, ld<NC>(q[5] + offR), P);
  double bp = fmax(WB_ADD(R.vn, cfR), 0.0);
  double bm = fmin(WB_SUB(L.vn, cfL), 0.0);
  if (roe) {
    bp = fmax(bp, WB_ADD(vn, cf));
    bm = fmin(bm, WB_SUB(vn, cf));
  }
  if (!(WB_SUB(bp, bm) > 0.0)) {
    const double sp = fmax(WB_ADD(fabs(L.vn), cfL), WB_ADD(fabs(R.vn), cfR));
    bp = sp;
    bm = -sp;
  }
  const double dq[7] = {WB_SUB(R.rho, L.rho), WB_SUB(R.mn, L.mn), WB_SUB(R.mt1, L.mt1), WB_SUB(R.mt2, L.mt2),
                        WB_SUB(R.bt1, L.bt1), WB_SUB(R.bt2, L.bt2), WB_SUB(R.eref, L.eref)};
  const double inv = 1.0 / WB_SUB(bp, bm);
  const double bpm = WB_MUL(bp, bm);
#pragma unroll
  for (int m = 0; m < 7; ++m) {
    // the zone fluxes hold F/2
    const double FL = WB_MUL(2.0, L.F[m]), FR = WB_MUL(2.0, R.F[m]);
    out[m] = WB_MUL(WB_FMA(bpm, dq[m], WB_FMA(bp, FL, -WB_MUL(bm, FR))), inv);
  }
}

// Bit of face_system's result: the interface's numbers may be beyond the range of
// the integer products, its flux takes FP64 ones too.
constexpr int kFp64Face = 4;

template <int EZ, bool PROT>
__device__ __noinline__ int face_system_fp64(const Cell& L, const Cell& R, double b, double dtdx, const WbPhys& P, const RegRec& f,
                                double gt[7]);

// Roe average of one interface's zones (reading of the Cargo-Gallice type
// average, App. A).
struct RoeState {
  double rho, irho, isrho, srho, vn, vt1, vt2, bt1, bt2, b2, dbt1, dbt2, gX, hv2, bt2s, a2;  // gX: (gamma-2) X
};
template <bool SOFT>
__device__ __forceinline__ void roe_state(const Cell& L, const Cell& R, double b, const WbPhys& P, RoeState& o) {
  const double iD = recip<SOFT>(WB_ADD(L.sr, R.sr));
  const double wL = mul<SOFT, 7>(L.sr, iD), wR = mul<SOFT, 7>(R.sr, iD);
  o.rho = mul<SOFT, 7>(L.sr, R.sr);
  const WbRoots rroe = roots<SOFT>(o.rho);
  o.irho = rroe.rcp;
  o.isrho = rroe.rsq;
  o.srho = rroe.sq;
  o.vn = WB_FMA(wL, L.vn, mul<SOFT, 2>(R.vn, wR));
  o.vt1 = WB_FMA(wL, L.vt1, mul<SOFT, 2>(R.vt1, wR));
  o.vt2 = WB_FMA(wL, L.vt2, mul<SOFT, 2>(R.vt2, wR));
  o.bt1 = WB_FMA(wR, L.bt1, mul<SOFT, 2>(R.bt1, wL));
  o.bt2 = WB_FMA(wR, L.bt2, mul<SOFT, 2>(R.bt2, wL));
  o.b2 = mul<SOFT>(b, b);
  // H = wL (h_L + b^2)/rho_L + wR (h_R + b^2)/rho_R, with wL/rho_L + wR/rho_R = 1/rho_
  const double H = WB_FMA(o.b2, o.irho, WB_FMA(wL, L.hr, mul<SOFT, 2>(R.hr, wR)));
  o.dbt1 = WB_SUB(R.bt1, L.bt1);
  o.dbt2 = WB_SUB(R.bt2, L.bt2);
  o.gX = WB_MUL(P.hgm2, WB_MUL(WB_FMA(o.dbt1, o.dbt1, mul<SOFT>(o.dbt2, o.dbt2)), mul<SOFT, 7>(iD, iD)));
  o.hv2 = wb_half(WB_FMA(o.vn, o.vn, WB_FMA(o.vt1, o.vt1, mul<SOFT>(o.vt2, o.vt2))));
  o.bt2s = WB_FMA(o.bt1, o.bt1, mul<SOFT>(o.bt2, o.bt2));
  o.a2 = WB_FMA(P.gm1, WB_FMA(-WB_ADD(o.b2, o.bt2s), o.irho, WB_SUB(H, o.hv2)), -o.gX);
}

// Roe state, eigen-system, alpha_k, nu_k and g-tilde_k (doubled) of one interface.
// Returns 0 for an MHDTVD face, 1 when the protection floor asks for the HLL
// flux (the record holds the Roe state), 2 when the Roe state has no real
// sound speed (HLL without Roe speeds).  The protection test is compiled in
// only when PROT is set.
template <int EZ, bool PROT, bool SOFT, class Rc>
__device__ __forceinline__ int face_system(const Cell& L, const Cell& R, double b, double dtdx,
                                           const WbPhys& P, const Rc& f, double gt[7]) {
  RoeState o;
  roe_state<SOFT>(L, R, b, P, o);
  const double rho = o.rho, irho = o.irho, isrho = o.isrho, srho = o.srho, vn = o.vn, vt1 = o.vt1, vt2 = o.vt2;
  const double bt1 = o.bt1, bt2 = o.bt2, b2 = o.b2, dbt1 = o.dbt1, dbt2 = o.dbt2, gX = o.gX, hv2 = o.hv2;
  const double bt2s = o.bt2s, a2 = o.a2;
  if (!wb_normal_pos(a2)) return 2;
  if (SOFT && wb_hi32(a2) < ((1023u - 100u) << 20)) {  // 1/a^2 may carry products out of the range
    Cell l = L, r = R;
    RegRec f2;
    double g2[7];
    const int code = face_system_fp64<EZ, PROT>(l, r, b, dtdx, P, f2, g2);
#pragma unroll
    for (int i = 0; i < R_WORDS; ++i) f[i] = f2[i];
#pragma unroll
    for (int k = 0; k < 7; ++k) gt[k] = g2[k];
    return code | kFp64Face;
  }
  const double ca2 = mul<SOFT, 2>(b2, irho), ct2 = mul<SOFT, 2>(bt2s, irho);
  const double dac = WB_SUB(a2, ca2);
  const double disc = WB_FMA(dac, dac, WB_MUL(ct2, WB_FMA(2.0, WB_ADD(a2, ca2), ct2)));
  const double sum = WB_ADD(WB_ADD(a2, ca2), ct2);
  // a subnormal discriminant is degenerate (sd ~ 0)
  const double sd = wb_normal_pos(disc) ? roots<SOFT>(disc).sq : 0.0;
  const double cf2 = wb_half(WB_ADD(sum, sd));
  const WbRoots rcf = roots<SOFT>(cf2), ra_ = roots<SOFT>(a2);
  const double icf = rcf.rsq, ia = ra_.rsq, ia2 = ra_.rcp;
  const double cf = rcf.sq, a = ra_.sq;
  const double ca = mul<SOFT, 2>(wb_fabs(b), isrho);
  const double cs = mul<SOFT, 2>(mul<SOFT, 1>(a, ca), icf);  // c_f c_s = a c_a
  // 1/|B_t| and c_t = |B_t| / sqrt(rho_); a transverse field whose square is
  // not a normal double (underflowing noise ahead of a front) counts as 0
  double ib = 0.0, btm = 0.0;  // btm = |B_t|
  if (wb_normal_pos(bt2s)) {
    const WbRoots rb = roots<SOFT>(bt2s);
    ib = rb.rsq;
    btm = rb.sq;
  }
  // With t1 = ca^2 + ct^2 - a^2: alpha_f^2 = (sd - t1) / (2 sd) and
  // alpha_s^2 = (sd + t1) / (2 sd) (cf^2 + cs^2 = a^2 + ca^2 + ct^2,
  // cf^2 - cs^2 = sd), and (sd - t1)(sd + t1) = disc - t1^2 = 4 a^2 ct^2,
  // so alpha_f alpha_s = a ct / sd.  The larger of the two is sqrt(m / (2 sd))
  // with m = sd + |t1| (no cancellation), = m r for r = 1/sqrt(2 sd m), and
  // the smaller a ct / (sd m r) = 2 a ct r: one reciprocal square root.
  // t1 takes the difference ca^2 - a^2 first: it is exact where the two
  // nearly cancel (the degenerate neighbourhood, where sd is small).
  const double t1 = WB_ADD(WB_SUB(ca2, a2), ct2);
  const bool slow_major = !wb_neg(t1);
  const double m = WB_ADD(sd, slow_major ? t1 : wb_flip(t1));
  const double r = roots<SOFT>(wb_twice(mul<SOFT>(sd, m))).rsq;
  const double major = mul<SOFT>(m, r);
  const double minor = WB_MUL(mul<SOFT, 1>(a, mul<SOFT, 2>(btm, isrho)), wb_twice(r));
  double af = slow_major ? minor : major;
  double as = slow_major ? major : minor;
  if (wb_maybe_below(sd, 39, wb_hi32(sum)) && wb_at_most(sd, 1e-12, sum)) {
    const bool fast = wb_le_nonneg(ca2, a2);
    af = fast ? 1.0 : 0.0;
    as = fast ? 0.0 : 1.0;
  }
  const double ra2 = mul<SOFT, 7>(rho, a2);
  double b1n = mul<SOFT>(bt1, ib), b2n = mul<SOFT>(bt2, ib);
  if (wb_maybe_small(bt2s, ra2, b2) && wb_at_most(bt2s, 1e-24, WB_ADD(WB_ADD(ra2, b2), bt2s)))
    b1n = b2n = 0.70710678118654752440;
  const double S = wb_sgn(b);
  // primitive differences of the 7-variable system; the velocity differences
  // are kept times rho_ (dv' = rho_ dv), the 1/rho_ goes into the coefficients
  const double drho = WB_SUB(R.rho, L.rho);
  const double dmn = WB_SUB(R.mn, L.mn), dmt1 = WB_SUB(R.mt1, L.mt1), dmt2 = WB_SUB(R.mt2, L.mt2);
  const double de = WB_SUB(R.eref, L.eref);
  const double dvn = WB_FMA(-vn, drho, dmn);
  const double dvt1 = WB_FMA(-vt1, drho, dmt1);
  const double dvt2 = WB_FMA(-vt2, drho, dmt2);
  const double vdm = WB_FMA(vn, dmn, WB_FMA(vt1, dmt1, mul<SOFT>(vt2, dmt2)));
  const double bdb = WB_FMA(bt1, dbt1, mul<SOFT>(bt2, dbt2));
  const double dp = WB_FMA(-gX, drho, WB_MUL(P.gm1, WB_SUB(WB_FMA(hv2, drho, WB_SUB(de, vdm)), bdb)));
  // projections on the transverse field direction beta and its normal; S = sign(b)
  const double dvbS = wb_xsgn(WB_FMA(b1n, dvt1, mul<SOFT>(dvt2, b2n)), S);
  const double dvp = WB_FMA(-b2n, dvt1, mul<SOFT>(dvt2, b1n));
  const double dbb = WB_FMA(b1n, dbt1, mul<SOFT>(dbt2, b2n));
  const double dbpS = wb_xsgn(WB_FMA(-b2n, dbt1, mul<SOFT>(dbt2, b1n)), S);
  const double hir = wb_half(irho), hisr = wb_half(isrho);
  const double i2ra = mul<SOFT, 7>(hisr, ia);   // 1 / (2 sqrt(rho) a)
  const double ri2a2 = mul<SOFT, 7>(hir, ia2);  // 1 / (2 rho a^2)
  const double dpr = mul<SOFT, 2>(dp, ri2a2);
  const double afcf = mul<SOFT, 2>(af, cf), ascs = mul<SOFT>(as, cs);
  const double dbbi = mul<SOFT, 2>(dbb, i2ra);
  // alpha_{1,7} = Cf -+ Xf / (2 rho a^2), alpha_{3,5} = Cs -+ Xs / (2 rho a^2): the factor
  // goes into the FMAs that form them
  const double Xf = WB_FMA(afcf, dvn, -mul<SOFT>(dvbS, ascs));
  const double Cf = WB_FMA(as, dbbi, mul<SOFT>(af, dpr));
  const double Xs = WB_FMA(ascs, dvn, mul<SOFT>(dvbS, afcf));
  const double Cs = WB_FMA(-af, dbbi, mul<SOFT>(as, dpr));
  const double hAa = mul<SOFT, 1>(hisr, dbpS);
  double al[7];
  al[0] = WB_FMA(-ri2a2, Xf, Cf);
  al[6] = WB_FMA(ri2a2, Xf, Cf);
  al[2] = WB_FMA(-ri2a2, Xs, Cs);
  al[4] = WB_FMA(ri2a2, Xs, Cs);
  al[1] = WB_FMA(hir, dvp, hAa);
  al[5] = WB_FMA(hir, dvp, -hAa);
  al[3] = WB_FMA(-dp, ia2, drho);
  // nu_k = (dt/dx) a_k for the eigenvalues a_1..a_7 (Sec. 3)
  const double tvn = mul<SOFT, 2>(vn, dtdx);
  const double nuk[7] = {WB_FMA(-dtdx, cf, tvn), WB_FMA(-dtdx, ca, tvn), WB_FMA(-dtdx, cs, tvn), tvn,
                         WB_FMA(dtdx, cs, tvn),  WB_FMA(dtdx, ca, tvn),  WB_FMA(dtdx, cf, tvn)};
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    const double nu = nuk[k];
    f[R_AL + k] = al[k];
    f[R_NU + k] = nu;
    gt[k] = mul<SOFT>(Qk_m_nu2<EZ, SOFT>(nu, k, P), al[k]);  // 2 g-tilde
  }
  f[R_RHO] = rho; f[R_SRHO] = wb_xsgn(srho, S); f[R_A] = a; f[R_PG] = mul<SOFT, 7>(ra2, P.inv_gm1); f[R_CF] = cf;
  f[R_ASCS] = ascs; f[R_AFCF] = afcf; f[R_AF] = af; f[R_AS] = as; f[R_B1] = b1n; f[R_B2] = b2n;
  f[R_VN] = vn; f[R_VT1] = vt1; f[R_VT2] = vt2; f[R_BTM] = btm;
  f[R_KX] = WB_FMA(gX, P.inv_gm1, -hv2);  // K - v^2 (the energy row of face_flux)
#pragma unroll
  for (int m = 0; m < 7; ++m) f[R_FAVG + m] = WB_ADD(L.F[m], R.F[m]);
  if (PROT && P.prot && protection_hit(L, R, rho, ra2, af, as, al, P)) return 1;
  return 0;
}

// The same with FP64 products, for the rare interface (not inlined).
template <int EZ, bool PROT>
__device__ int face_system_fp64(const Cell& L, const Cell& R, double b, double dtdx, const WbPhys& P,
                                             const RegRec& f, double gt[7]) {
  return face_system<EZ, PROT, false>(L, R, b, dtdx, P, f, gt);
}

// beta_k of App. A from the limited slopes carried doubled, G = 2 g (the
// limiter commutes with the factor 2), without forming gamma_k.  With
// w = nu alpha + g_{i+1} - g_i, Q(nu + gamma) alpha = Q(w / alpha) alpha.  Where
// Q(x) = |x| (eps_k = 0, or |w| >= 2 eps |alpha|) that is |w| sign(alpha), and
// beta = |w| sign(alpha) - (g_i + g_{i+1}) is nu alpha - G_i when w has the sign
// of alpha, else -nu alpha - G_{i+1}: the larger of the two for alpha > 0, the
// smaller for alpha < 0, one FMA after an integer-pipe choice of operands.
// Inside the band, Q(x) alpha = w^2 / (4 eps alpha) + eps alpha, with
// 2 w = 2 nu alpha + G_{i+1} - G_i.  alpha = 0 needs no case of its own: this
// face's g-tilde is then 0, the limiter makes G_i = G_{i+1} = 0 and either form
// gives 0.
template <int EZ, bool SOFT>
__device__ __forceinline__ double beta_k(double al, double nu, double Gi, double Gi1, int k,
                                         const WbPhys& P) {
  if (EZ & (1 << k)) {
    const double b1 = WB_FMA(nu, al, -Gi), b2 = WB_FMA(-nu, al, -Gi1);
    return (wb_order_less(b1, b2) != wb_neg(al)) ? b2 : b1;
  }
  const double d = WB_FMA(wb_twice(nu), al, WB_SUB(Gi1, Gi));  // 2 w
  if (!wb_abs_less(d, mul<SOFT>(al, P.four_eps[k]))) {
    const bool same = (__double_as_longlong(d) ^ __double_as_longlong(al)) >= 0;
    return WB_FMA(same ? nu : wb_flip(nu), al, -(same ? Gi : Gi1));
  }
  // |nu + gamma| < 2 eps: beta = (2 w)^2 / (16 eps alpha) + eps alpha - (g_i + g_{i+1})
  const double t = WB_FMA(P.eps[k], al, -wb_half(WB_ADD(Gi, Gi1)));
  if (wb_abs_less(al, 1e-290)) return t;  // (2 w)^2 / (16 eps alpha) < eps |alpha|
  return WB_FMA(mul<SOFT>(mul<SOFT>(d, d), P.inv16eps[k]), recip<SOFT>(al), t);
}

// u-bar = (F_L + F_R)/2 - (dx/(2 dt)) sum_k beta_k R_k  (App. A)
template <int EZ, bool SOFT, class Rc>
__device__ __forceinline__ void face_flux(const Rc& f, const double gi[7], const double gi1[7],
                                          double dx_2dt, const WbPhys& P, double out[7]) {
  double be[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) be[k] = beta_k<EZ, SOFT>(f[R_AL + k], f[R_NU + k], gi[k], gi1[k], k, P);
  const double rho = f[R_RHO], af = f[R_AF], as = f[R_AS];
  const double S = f[R_SRHO], b1 = f[R_B1], b2 = f[R_B2];  // S: sign(b) sqrt(rho_)
  // sum_k beta_k r_k in w = (rho, vn, vt, Bt, p)
  const double sf = WB_ADD(be[0], be[6]), df = WB_SUB(be[6], be[0]);
  const double ss = WB_ADD(be[2], be[4]), ds = WB_SUB(be[4], be[2]);
  const double afcf = f[R_AFCF], ascs = f[R_ASCS], srho = wb_fabs(S);
  const double vp = WB_ADD(be[1], be[5]);                             // along beta-perp
  const double tfs = WB_FMA(af, sf, mul<SOFT>(ss, as));
  const double wr = WB_FMA(rho, tfs, be[3]);
  const double wvn = WB_FMA(afcf, df, mul<SOFT>(ds, ascs));
  const double vb = wb_xsgn(WB_FMA(afcf, ds, -mul<SOFT>(df, ascs)), S);  // along beta
  const double bb = mul<SOFT>(WB_FMA(as, sf, -mul<SOFT>(ss, af)), mul<SOFT, 7>(f[R_A], srho));
  const double bp = wb_xsgn(mul<SOFT, 2>(WB_SUB(be[1], be[5]), srho), S);
  const double wvt1 = WB_FMA(b1, vb, -mul<SOFT>(vp, b2)), wvt2 = WB_FMA(b2, vb, mul<SOFT>(vp, b1));
  const double wbt1 = WB_FMA(b1, bb, -mul<SOFT>(bp, b2)), wbt2 = WB_FMA(b2, bb, mul<SOFT>(bp, b1));
  // to conserved variables (the pressure row enters the energy as p/(gamma-1))
  const double vn = f[R_VN], vt1 = f[R_VT1], vt2 = f[R_VT2];
  const double u1 = WB_FMA(vn, wr, mul<SOFT, 2>(wvn, rho));
  const double u2 = WB_FMA(vt1, wr, mul<SOFT, 2>(wvt1, rho));
  const double u3 = WB_FMA(vt2, wr, mul<SOFT, 2>(wvt2, rho));
  // energy: B_t . w_Bt + p/(gamma-1) row + K w_rho + rho v . w_v, with
  // rho v . w_v = v . u - v^2 w_rho and the record holding K - v^2, and
  // B_t . w_Bt = |B_t| w_beta: beta is B_t / |B_t|, so the beta-perpendicular
  // part has no component along B_t (where |B_t|^2 is below 1e-24 of the
  // energy scale and beta is set to (1, 1)/sqrt 2 instead, the term is of that
  // size either way)
  const double u6 = WB_FMA(f[R_BTM], bb, WB_FMA(f[R_PG], tfs,
                    WB_FMA(f[R_KX], wr, WB_FMA(vn, u1, WB_FMA(vt1, u2, WB_MUL(vt2, u3))))));
  out[0] = WB_FMA(-dx_2dt, wr, f[R_FAVG + 0]);
  out[1] = WB_FMA(-dx_2dt, u1, f[R_FAVG + 1]);
  out[2] = WB_FMA(-dx_2dt, u2, f[R_FAVG + 2]);
  out[3] = WB_FMA(-dx_2dt, u3, f[R_FAVG + 3]);
  out[4] = WB_FMA(-dx_2dt, wbt1, f[R_FAVG + 4]);
  out[5] = WB_FMA(-dx_2dt, wbt2, f[R_FAVG + 5]);
  out[6] = WB_FMA(-dx_2dt, u6, f[R_FAVG + 6]);
}

// The same with FP64 products, for the rare interface (not inlined).
template <int EZ>
__device__ __noinline__ void face_flux_fp64(const RegRec& f, const double gi[7], const double gi1[7], double dx_2dt,
                                            const WbPhys& P, double out[7]) {
  face_flux<EZ, false>(f, gi, gi1, dx_2dt, P, out);
}

// What a face needs of its left zone, word by word.
constexpr int kCellWords = 19;
__device__ __forceinline__ double& cell_word(Cell& c, int i) {
  switch (i) {
    case 0: return c.rho;
    case 1: return c.sr;
    case 2: return c.vn;
    case 3: return c.vt1;
    case 4: return c.vt2;
    case 5: return c.bt1;
    case 6: return c.bt2;
    case 7: return c.eref;
    case 8: return c.hr;
    case 9: return c.mn;
    case 10: return c.mt1;
    case 11: return c.mt2;
    default: return c.F[i - 12];
  }
}

// The words that cross from one warp of a block to another.  Of a warp's
// threads at most two have a right neighbour in another warp, lane 31 (slot 0)
// and the end of a ring that began in an earlier warp (slot 1), and two a left
// one, lane 0 and the start of a ring that ends in a later warp.
struct LaneEdge {
  double cell[kWarps][2][kCellWords];             // zone, to the right neighbour
  double gt[kWarps][2][7], gz[kWarps][2][7];      // g-tilde to the left, limited slope to the right neighbour
};

// A sweep along one axis: fields in the sweep's frame (q: rho, Mn, Mt1, Mt2,
// E, Bn, Bt1, Bt2; F: rho, Mn, Mt1, Mt2, Bt1, Bt2, E), faces of `box` along
// axis d, zones of it across.
struct SweepFrame {
  const double* q[8];
  const double* bn;
  double* F[7];
};
template <int D>
__host__ __device__ __forceinline__ void sweep_frame(const double* const* q, const double* bn, double* const* F,
                                                     SweepFrame& f) {
  constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
  f.q[0] = q[F_RHO];
  f.q[1] = q[F_MX + D];
  f.q[2] = q[F_MX + T1];
  f.q[3] = q[F_MX + T2];
  f.q[4] = q[F_EN];
  f.q[5] = q[F_BX + D];
  f.q[6] = q[F_BX + T1];
  f.q[7] = q[F_BX + T2];
  f.bn = bn;
  f.F[0] = F[F_RHO];
  f.F[1] = F[F_MX + D];
  f.F[2] = F[F_MX + T1];
  f.F[3] = F[F_MX + T2];
  f.F[4] = F[F_BX + T1];
  f.F[5] = F[F_BX + T2];
  f.F[6] = F[F_EN];
}

// How the faces of a sweep are laid out over threads.  In the open layout
// every pencil of len faces is a run of len + 3 zones (two before its first
// face's right zone, one after its last), the runs follow one another, and a
// block takes kBlock zones of them, emits the faces that find both neighbours'
// slopes in the block and advances by kTile: kTile / kBlock x len / (len + 3)
// of the threads emit a face.  A closed pencil (periodic, its first and last
// zone neighbours) of at most kBlock zones can sit in a block as a ring
// instead: floor(kBlock / len) len of its threads emit.  The better of the two
// is taken: a ring at 16, 32, 64, 128 zones (all threads against 82, 89, 93,
// 95 %), at 40 (94 against 91), not at 48 or 96 (75 against 92 and 95).
__host__ __device__ __forceinline__ bool sweep_ring(int len, bool closed) {
  return closed && len <= kBlock && (kBlock / len) * (len + 3) >= kTile;
}
// Kernels compiled for one layout, for either at run time (2 % slower), or for
// either with the flux of one-zone pencils apart (0.5 to 1 % slower on others).
enum { kOpen = 0, kRing = 1, kAnyLayout = 2, kThin = 3 };
// tiles (blocks' worth of work) of npen pencils
__host__ __device__ __forceinline__ long long sweep_tiles(long long npen, int len, bool ring) {
  const long long per = ring ? kBlock / len : kTile;
  const long long n = ring ? npen : npen * (len + 3) - 3;
  return (n + per - 1) / per;
}

template <int EZ, bool PROT, bool NC>
__device__ __noinline__ int sweep_tile_fp64(const WbGeo& g, const WbBox& box, int d, const SweepFrame& s, long long tile, bool closed,
                               bool ring, int nslots, long long slot_in, long long slot_out, const WbScalars* scal,
                               const WbPhys& P, LaneEdge& X);

// One tile of a sweep, one face per thread: the thread holds a zone and its low
// face; its neighbours along the pencil hand over zone state, g-tilde and
// limited slopes by shuffles and, at the ends of a warp, through shared memory
// (X).  Every thread of the block calls this.  Faces without a Roe state or
// below the protection floor take the HLL flux and give g-tilde = 0 to the
// limiters of their neighbours.  Returns 1 when the thread's stored flux is an
// HLL flux of an interior face of the box (ghost rings, which depend on how a
// box is split, are not counted).
//
// What bounds it: the FP64 pipe (one warp instruction per 19 cycles and SM) and
// beside it the latency of the integer work that takes FP64 work over (wb_soft).
// A thread that marched along a pencil kept two zones, two slopes and a face
// record in 226 to 255 registers and 40 KB of shared memory a block, which left
// 2 warps per scheduler; one face per thread runs with 128 registers, 4 warps
// (some 200 bytes of spills).  (F_L + F_R)/2 in shared memory rather than in the
// spills was no faster (17.5 against 17.4 ms a 256^3 launch).
template <int EZ, bool PROT, bool SOFT, bool NC, int LAYOUT>
__device__ __forceinline__ int sweep_tile(const WbGeo& g, const WbBox& box, int d, const SweepFrame& s, long long tile,
                                          bool closed, bool ring_, int nslots, long long slot_in, long long slot_out,
                                          const WbScalars* scal, const WbPhys& P, LaneEdge& X) {
  const bool ring = LAYOUT >= kAnyLayout ? ring_ : LAYOUT == kRing;
  const int U = d == 0 ? 1 : 0, W = d == 2 ? 1 : 2;
  const int nu = box.hi[U] - box.lo[U] + 1, nw = box.hi[W] - box.lo[W] + 1;
  const int len = box.hi[d] - box.lo[d] + 1;
  // pencils and zones of a launch fit 32 bits (64-bit divisions cost hundreds of instructions)
  const unsigned npen = (unsigned)(nu * nw) * (unsigned)nslots;
  const int t = threadIdx.x, lane = t % 32, wp = t / 32;
  unsigned pen;
  int idx, lt, rt;  // zone along the pencil; threads of the neighbours
  bool has_left, emit;
  if (ring) {
    const int per = kBlock / len, seg = t / len;
    idx = t - seg * len;
    pen = (unsigned)tile * per + seg;
    emit = seg < per && pen < npen;
    if (pen >= npen) pen = npen - 1;
    has_left = true;
    lt = idx > 0 ? t - 1 : t + len - 1;
    rt = idx < len - 1 ? t + 1 : t - len + 1;
    if (seg >= per) lt = rt = t;
  } else {
    const unsigned total = npen * (unsigned)(len + 3);
    unsigned z = (unsigned)tile * kTile + t;
    emit = z < total;
    if (z >= total) z = total - 1;
    pen = z / (unsigned)(len + 3);
    idx = (int)(z - pen * (unsigned)(len + 3)) - 2;
    has_left = idx > -2 && t > 0;
    emit = emit && idx >= 0 && idx < len && t >= 2 && t <= kBlock - 2;
    lt = t > 0 ? t - 1 : t;
    rt = t < kBlock - 1 ? t + 1 : t;
    // the zones past the ends of a closed pencil are those of its other end
    // (an open layout is only taken for 3 zones or more, see sweep_ring)
    if (closed) idx = idx < 0 ? idx + len : (idx >= len ? idx - len : idx);
  }
  // The pencils of a closed axis of one zone: every face lies between a zone and
  // itself, the jump and with it every alpha_k is exactly zero, and the flux is
  // the zone's own.  Only the test for a real Roe sound speed is left.  (A third of
  // the faces of a plane: ten steps of 192^2 zones 1377 us before, 1185 so.)
  const bool self = LAYOUT == kThin && !PROT && ring && len == 1;
  const long long slot = pen / (unsigned)(nu * nw);
  const int r = (int)(pen - (unsigned)slot * (unsigned)(nu * nw));
  int pos[3];
  pos[U] = box.lo[U] + r % nu;
  pos[W] = box.lo[W] + r / nu;
  pos[d] = box.lo[d] + idx;
  const long long at = wb_at(g, pos[0], pos[1], pos[2]);
  const long long off = slot * slot_in + at;
  const long long o = slot * slot_out + at;
  Cell R;
  if (self) {
    RoeState w;
    load_cell<NC, false>(s.q, off, P, R);
    roe_state<false>(R, R, ld<NC>(s.bn + off), P, w);
    if (!emit) return 0;
    const bool hll = !wb_normal_pos(w.a2);
    double out[7];
#pragma unroll
    for (int m = 0; m < 7; ++m) out[m] = WB_ADD(R.F[m], R.F[m]);
    if (hll) hll_face<NC>(s.q, off, off, false, 0.0, 0.0, P, out);
#pragma unroll
    for (int m = 0; m < 7; ++m) s.F[m][o] = out[m];
    return hll && pos[0] >= 0 && pos[0] < g.n[0] && pos[1] >= 0 && pos[1] < g.n[1] && pos[2] >= 0 && pos[2] < g.n[2];
  }
  FieldRange range = load_cell<NC, SOFT>(s.q, off, P, R);
  const double b = ld<NC>(s.bn + off), dtdx = scal->dtdx[d];
  range.add(b);
  range.add(dtdx);
  const bool wild = SOFT && range.wild(R.rho);
  Cell L;
  L.ir = 0.0;  // not used across a face
  // neighbours in other warps go through X, unless every ring sits in a warp
  const bool cross = !(ring && 32 % len == 0);
  const int wl = lt / 32, wr = rt / 32, sl = lt % 32 == 31 ? 0 : 1, sr = rt % 32 == 0 ? 0 : 1;
  const int mine_r = lane == 31 ? 0 : 1, mine_l = lane == 0 ? 0 : 1;
  if (cross) {
    if (wr != wp) {
#pragma unroll
      for (int i = 0; i < kCellWords; ++i) X.cell[wp][mine_r][i] = cell_word(R, i);
    }
  }
  // a block (a warp of its own rings) that meets a field beyond the integer
  // products' range starts over with FP64 products
  if (SOFT) {
    if (cross ? __syncthreads_or(wild) : __any_sync(0xffffffffu, wild))
      return sweep_tile_fp64<EZ, PROT, NC>(g, box, d, s, tile, closed, ring, nslots, slot_in, slot_out, scal, P, X);
  } else if (cross) {
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < kCellWords; ++i) cell_word(L, i) = __shfl_sync(0xffffffffu, cell_word(R, i), lt % 32);
  if (cross && wl != wp) {
#pragma unroll
    for (int i = 0; i < kCellWords; ++i) cell_word(L, i) = X.cell[wl][sl][i];
  }
  RegRec f;
  double gt[7];
  int code = face_system<EZ, PROT, SOFT>(L, R, b, dtdx, P, f, gt);
  const bool fp64 = SOFT && (code & kFp64Face);
  code &= ~kFp64Face;
  bool hll = false;
  if (code) {
    if (has_left) {
      long long st = d == 0 ? 1LL : (d == 1 ? g.sy : g.sz);
      if (closed && idx == 0) st *= 1 - len;
      double h[7];
      hll_face<NC>(s.q, off - st, off, code == 1, code == 1 ? f[R_VN] : 0.0, code == 1 ? f[R_CF] : 0.0, P, h);
#pragma unroll
      for (int m = 0; m < 7; ++m) f[R_FAVG + m] = h[m];
      hll = true;
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) gt[k] = 0.0;
  }
  __syncwarp();
  if (cross) {
    if (wl != wp) {
#pragma unroll
      for (int k = 0; k < 7; ++k) X.gt[wp][mine_l][k] = gt[k];
    }
    __syncthreads();
  }
  double gz[7], gl[7];  // 2 g of this zone, of the left zone
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    double gr = __shfl_sync(0xffffffffu, gt[k], rt % 32);
    if (cross && wr != wp) gr = X.gt[wr][sr][k];
    gz[k] = wb_sweby(gr, gt[k], P.sweby, P.minmod);
  }
  if (cross) {
    if (wr != wp) {
#pragma unroll
      for (int k = 0; k < 7; ++k) X.gz[wp][mine_r][k] = gz[k];
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    gl[k] = __shfl_sync(0xffffffffu, gz[k], lt % 32);
    if (cross && wl != wp) gl[k] = X.gz[wl][sl][k];
  }
  if (!emit) return 0;
  double out[7];
  if (hll) {
#pragma unroll
    for (int m = 0; m < 7; ++m) out[m] = f[R_FAVG + m];
  } else if (fp64) {
    RegRec f2 = f;
    double a[7], c[7], o2[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) {
      a[k] = gl[k];
      c[k] = gz[k];
    }
    face_flux_fp64<EZ>(f2, a, c, scal->dx_2dt[d], P, o2);
#pragma unroll
    for (int m = 0; m < 7; ++m) out[m] = o2[m];
  } else {
    face_flux<EZ, SOFT>(f, gl, gz, scal->dx_2dt[d], P, out);
  }
#pragma unroll
  for (int m = 0; m < 7; ++m) s.F[m][o] = out[m];
  return hll && pos[0] >= 0 && pos[0] < g.n[0] && pos[1] >= 0 && pos[1] < g.n[1] && pos[2] >= 0 && pos[2] < g.n[2];
}

template <int EZ, bool PROT, bool NC>
__device__ int sweep_tile_fp64(const WbGeo& g, const WbBox& box, int d, const SweepFrame& s, long long tile,
                                            bool closed, bool ring, int nslots, long long slot_in, long long slot_out,
                                            const WbScalars* scal, const WbPhys& P, LaneEdge& X) {
  return sweep_tile<EZ, PROT, false, NC, kAnyLayout>(g, box, d, s, tile, closed, ring, nslots, slot_in, slot_out, scal, P,
                                                     X);
}

// ---------------------------------------------------------------- stages ---

__device__ __forceinline__ bool in_box(const WbBox& b, int i, int j, int k) {
  return i >= b.lo[0] && i <= b.hi[0] && j >= b.lo[1] && j <= b.hi[1] && k >= b.lo[2] && k <= b.hi[2];
}

// The cheap stages are split into a load of their inputs and a finish that
// computes and stores, so that the batch kernel can load a second item before
// storing the first (two memory requests in flight per thread).  Their
// arithmetic is written with explicit rounding: an item gives the same bits
// whichever inlined copy (first or second of a pair, or alone) handles it.

// Offsets to the high and low neighbours of a zone along each axis.  closed:
// bit d set when axis d is periodic and whole in this patch; the neighbour of
// its last zone is then its first one, so no stage of such a box reads a ghost.
struct Nbr {
  long long up[3], dn[3];
};
__device__ __forceinline__ Nbr neighbours(const WbGeo& g, int i, int j, int k, int closed) {
  const int x[3] = {i, j, k};
  const long long s[3] = {1, g.sy, g.sz};
  Nbr b;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const bool c = (closed >> d) & 1;
    b.up[d] = c && x[d] == g.n[d] - 1 ? -(g.n[d] - 1) * s[d] : s[d];
    b.dn[d] = c && x[d] == 0 ? (g.n[d] - 1) * s[d] : -s[d];
  }
  return b;
}

// Step 2: zone-centred reference EMF E = -v x B from q^n.
struct ErefIn {
  long long w;
  double rho, m[3], B[3];
};

__device__ __forceinline__ void eref_load(const WbView& v, long long qo, long long wo, int i, int j, int k,
                                          ErefIn& in) {
  const long long o = qo + wb_at(v.geo, i, j, k);
  in.w = wo + wb_at(v.geo, i, j, k);
  in.rho = v.q[F_RHO][o];
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    in.m[e] = v.q[F_MX + e][o];
    in.B[e] = v.q[F_BX + e][o];
  }
}

__device__ __forceinline__ void eref_finish(double* const* E, const ErefIn& in) {
  const double ir = wb_rcp(in.rho);
  const double vx = __dmul_rn(in.m[0], ir), vy = __dmul_rn(in.m[1], ir), vz = __dmul_rn(in.m[2], ir);
  const double bx = in.B[0], by = in.B[1], bz = in.B[2];
  E[0][in.w] = __fma_rn(vz, by, __dmul_rn(-vy, bz));
  E[1][in.w] = __fma_rn(vx, bz, __dmul_rn(-vz, bx));
  E[2][in.w] = __fma_rn(vy, bx, __dmul_rn(-vx, by));
}

__device__ __forceinline__ void eref(const WbView& v, long long qo, long long wo, int i, int j, int k) {
  ErefIn in;
  eref_load(v, qo, wo, i, j, k, in);
  eref_finish(v.Eref, in);
}

// The mean of the two one-sided differences, for a zero mass flux.  Not
// inlined: inlined, the compiler if-converts it and every warp issues its
// instructions with every lane predicated off (the FP64 pipe's warp-level
// count exceeded its thread-level count by a third in the corner-EMF kernel).
static __device__ __noinline__ double mean_diff(double xm, double ym, double x0, double y0) {
  return __dmul_rn(0.5, __dadd_rn(__dsub_rn(xm, ym), __dsub_rn(x0, y0)));
}

// Difference x - y upwind of the mass flux m: (xm - ym) from the minus-side
// zone if m > 0, (x0 - y0) from the plus-side zone if m < 0, the mean of both
// if m = 0.  The operands are selected first (integer pipe), so one FP64
// subtraction is spent; the mean is taken only by warps in which some lane
// has a zero mass flux, so the common case carries none of its arithmetic.
__device__ __forceinline__ double upwind_diff(double m, double xm, double ym, double x0, double y0) {
  const bool minus = wb_neg(m);
  double d = __dsub_rn(minus ? x0 : xm, minus ? y0 : ym);
  const bool zero = wb_zero(m);
  if (__any_sync(__activemask(), zero)) {
    const double mean = mean_diff(xm, ym, x0, y0);
    if (zero) d = mean;
  }
  return d;
}

// Steps 3 and 9: upwinded corner EMF (GS05 "CT-contact" form).  Edge along
// axis C at the low faces of axes a = C+1 and b = C+2 (cyclic).  Face EMFs
// E^a = -F_a[B_b], E^b = +F_b[B_a]; the corner value is their average plus
// one quarter of [(dE/db) at -3/4 minus (dE/db) at -1/4] and the same along
// a, each derivative taken from the zone upwind of the mass flux through the
// face it sits on (the mean of both zones when that flux is zero).
struct EdgeIn {
  long long o;
  double Ea_0, Ea_m, Eb_0, Eb_m, ma_0, ma_m, mb_0, mb_m, R00, Rm0, R0m, Rmm;
};

template <int C>
__device__ __forceinline__ void edge_load(const WbView& v, long long wo, bool corr, int i, int j, int k, const Nbr& nb,
                                          EdgeIn& in) {
  constexpr int a = (C + 1) % 3, b = (C + 2) % 3;
  const WbGeo& g = v.geo;
  const long long o = wo + wb_at(g, i, j, k);
  const long long sa = -nb.dn[a], sb = -nb.dn[b];
  WB_CHECK_ZONE(g, i - (a == 0) - (b == 0), j - (a == 1) - (b == 1), k - (a == 2) - (b == 2));
  double* const* Fa = corr ? v.Fc[a] : v.Fp[a];
  double* const* Fb = corr ? v.Fc[b] : v.Fp[b];
  const double* Er = corr ? v.Erefh[C] : v.Eref[C];
  in.o = o;
  in.Ea_0 = wb_flip(Fa[F_BX + b][o]);
  in.Ea_m = wb_flip(Fa[F_BX + b][o - sb]);
  in.Eb_0 = Fb[F_BX + a][o];
  in.Eb_m = Fb[F_BX + a][o - sa];
  in.ma_0 = Fa[F_RHO][o];
  in.ma_m = Fa[F_RHO][o - sb];
  in.mb_0 = Fb[F_RHO][o];
  in.mb_m = Fb[F_RHO][o - sa];
  in.R00 = Er[o];
  in.Rm0 = Er[o - sa];
  in.R0m = Er[o - sb];
  in.Rmm = Er[o - sa - sb];
}

template <int C>
__device__ __forceinline__ void edge_finish(const WbView& v, bool corr, const EdgeIn& in) {
  const double db_hi = upwind_diff(in.ma_0, in.Rm0, in.Eb_m, in.R00, in.Eb_0);
  const double db_lo = upwind_diff(in.ma_m, in.Eb_m, in.Rmm, in.Eb_0, in.R0m);
  const double da_hi = upwind_diff(in.mb_0, in.R0m, in.Ea_m, in.R00, in.Ea_0);
  const double da_lo = upwind_diff(in.mb_m, in.Ea_m, in.Rmm, in.Ea_0, in.Rm0);
  double* out = corr ? v.Eedgeh[C] : v.Eedge[C];
  out[in.o] = wb_quarter((in.Ea_0 + in.Ea_m) + (in.Eb_0 + in.Eb_m) + (db_lo - db_hi) + (da_lo - da_hi));
}

template <int C>
__device__ __forceinline__ void edge(const WbView& v, long long wo, bool corr, int i, int j, int k, const Nbr& nb) {
  EdgeIn in;
  edge_load<C>(v, wo, corr, i, j, k, nb, in);
  edge_finish<C>(v, corr, in);
}

// Steps 4 and 11: b_out = b_in - tau curl E on the faces normal to D.
// Step 4 writes b^{n+1/2} to the workspace, Step 11 updates b in place.
struct CtIn {
  long long w, q;
  double Eb0, Eb1, Ea0, Ea1, b;
};

template <int D>
__device__ __forceinline__ void ct_load(const WbView& v, long long qo, long long wo, bool fin, int i, int j,
                                        int k, const Nbr& nb, CtIn& in) {
  constexpr int a = (D + 1) % 3, b = (D + 2) % 3;
  const WbGeo& g = v.geo;
  in.w = wo + wb_at(g, i, j, k);
  in.q = qo + wb_at(g, i, j, k);
  const long long sa = nb.up[a], sb = nb.up[b];
  WB_CHECK_ZONE(g, i + (a == 0), j + (a == 1), k + (a == 2));
  WB_CHECK_ZONE(g, i + (b == 0), j + (b == 1), k + (b == 2));
  const double* Eb = fin ? v.Eedgeh[b] : v.Eedge[b];
  const double* Ea = fin ? v.Eedgeh[a] : v.Eedge[a];
  in.Eb0 = Eb[in.w];
  in.Eb1 = Eb[in.w + sa];
  in.Ea0 = Ea[in.w];
  in.Ea1 = Ea[in.w + sb];
  in.b = v.b[D][in.q];
}

template <int D>
__device__ __forceinline__ void ct_finish(const WbView& v, bool fin, double dt, const CtIn& in) {
  constexpr int a = (D + 1) % 3, b = (D + 2) % 3;
  const double tau = fin ? dt : wb_half(dt);
  const double curl = __fma_rn(in.Eb1 - in.Eb0, v.geo.idx[a], __dmul_rn(in.Ea0 - in.Ea1, v.geo.idx[b]));
  const double bn = __fma_rn(-tau, curl, in.b);
  if (fin) v.b[D][in.q] = bn;
  else v.bh[D][in.w] = bn;
}

template <int D>
__device__ __forceinline__ void ct(const WbView& v, long long qo, long long wo, bool fin, double dt,
                                   int i, int j, int k, const Nbr& nb) {
  CtIn in;
  ct_load<D>(v, qo, wo, fin, i, j, k, nb, in);
  ct_finish<D>(v, fin, dt, in);
}

// Steps 5 and 7: q^{n+1/2}_D = q^n - dt/2 (transverse flux divergence)
// + dt/2 S_D, zone B_D := mean of b_D^{n+1/2}, with the GS08-type div B
// source S_D built from face differences of b^n and minmod pairings.
//
// Zone quantities shared by the directions: velocity v, zone field B, B_e v_e,
// the face-field differences scaled by dt/2 (h db_e = dt/2 (b_e+ - b_e)/dx_e;
// minmod commutes with the positive factor dt/2), the flux-difference factors
// c_e = dt/2 / dx_e and the transverse flux differences dF_e = F_e+ - F_e.
// The arithmetic is written with explicit rounding: the same bits in every
// kernel it is inlined into (the grid path, both forms of the batch path).
struct TransZone {
  double qn[8];
  double vv[3], B[3], Bv[3], hdb[3], c[3];
  double dF[3][8];
};

__device__ __forceinline__ void trans_zone(const WbView& v, long long q, long long w, int need,
                                           const Nbr& nb, TransZone& z) {
  const long long (&s)[3] = nb.up;
#pragma unroll
  for (int cc = 0; cc < 8; ++cc) z.qn[cc] = v.q[cc][q];
  const double ir = wb_rcp(z.qn[F_RHO]);
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    z.vv[e] = __dmul_rn(z.qn[F_MX + e], ir);
    z.B[e] = z.qn[F_BX + e];
    z.Bv[e] = __dmul_rn(z.B[e], z.vv[e]);
    z.c[e] = v.scal->hdtdx[e];
    z.hdb[e] = __dmul_rn(__dsub_rn(v.b[e][q + s[e]], v.b[e][q]), z.c[e]);
  }
#pragma unroll
  for (int e = 0; e < 3; ++e) {
#pragma unroll
    for (int cc = 0; cc < 8; ++cc) {
      if (cc == F_BX + e || !(need & (1 << e))) { z.dF[e][cc] = 0.0; continue; }
      z.dF[e][cc] = __dsub_rn(v.Fp[e][cc][w + s[e]], v.Fp[e][cc][w]);
    }
  }
}

// q^{n+1/2}_D of one zone from its shared quantities.  The t1 (t2) field
// component is carried only by the t2 (t1) sweep; density has no source.
template <int D>
__device__ __forceinline__ void trans_dir(const WbView& v, long long w, const Nbr& nb, const TransZone& z) {
  constexpr int t1 = (D + 1) % 3, t2 = (D + 2) % 3;
  const long long sD = nb.up[D];
  const double hm2 = wb_minmod(z.hdb[D], wb_flip(z.hdb[t1]));  // for the t2 field component
  const double hm1 = wb_minmod(z.hdb[D], wb_flip(z.hdb[t2]));  // for the t1 field component
  const double hSe = __fma_rn(z.Bv[t1], hm1, __dmul_rn(z.Bv[t2], hm2));
  const double c1 = z.c[t1], c2 = z.c[t2];
  double u[8];
#pragma unroll
  for (int cc = F_RHO; cc <= F_EN; ++cc)
    u[cc] = __fma_rn(-c2, z.dF[t2][cc], __fma_rn(-c1, z.dF[t1][cc], z.qn[cc]));
  v.qh[D][F_RHO][w] = u[F_RHO];
#pragma unroll
  for (int e = 0; e < 3; ++e) v.qh[D][F_MX + e][w] = __fma_rn(z.B[e], z.hdb[D], u[F_MX + e]);
  v.qh[D][F_EN][w] = __dadd_rn(u[F_EN], hSe);
  v.qh[D][F_BX + t1][w] = __fma_rn(z.vv[t1], hm1, __fma_rn(-c2, z.dF[t2][F_BX + t1], z.qn[F_BX + t1]));
  v.qh[D][F_BX + t2][w] = __fma_rn(z.vv[t2], hm2, __fma_rn(-c1, z.dF[t1][F_BX + t2], z.qn[F_BX + t2]));
  v.qh[D][F_BX + D][w] = wb_half(__dadd_rn(v.bh[D][w], v.bh[D][w + sD]));
}

// The directions in mask (bit d) at one zone, sharing the zone quantities and
// each transverse flux difference between the two states that use it.
__device__ __forceinline__ void transverse_set(const WbView& v, long long qo, long long wo, int mask,
                                               int i, int j, int k, const Nbr& nb) {
  const long long q = qo + wb_at(v.geo, i, j, k);
  const long long w = wo + wb_at(v.geo, i, j, k);
  WB_CHECK_ZONE(v.geo, i + 1, j + 1, k + 1);  // the high neighbours of every axis
  // flux differences of every direction some state needs
  int need = 0;
#pragma unroll
  for (int e = 0; e < 3; ++e)
    if (mask & ~(1 << e)) need |= 1 << e;
  TransZone z;
  trans_zone(v, q, w, need, nb, z);
  if (mask & 1) trans_dir<0>(v, w, nb, z);
  if (mask & 2) trans_dir<1>(v, w, nb, z);
  if (mask & 4) trans_dir<2>(v, w, nb, z);
}

// Step 8: reference EMF at n+1/2 from v of q^n - dt/2 div F* and B = mean of
// b^{n+1/2}.
struct ErefHalfIn {
  long long w;
  double q[4];        // rho, M of q^n
  double dF[4][3];    // F*_e+ - F*_e for rho, M
  double bh[3][2];    // b^{n+1/2} on the low and high faces
};

__device__ __forceinline__ void eref_half_load(const WbView& v, long long qo, long long wo, int i, int j,
                                               int k, const Nbr& nb, ErefHalfIn& in) {
  const WbGeo& g = v.geo;
  const long long q = qo + wb_at(g, i, j, k);
  const long long w = wo + wb_at(g, i, j, k);
  const long long (&s)[3] = nb.up;
  WB_CHECK_ZONE(g, i + 1, j + 1, k + 1);
  in.w = w;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    in.q[c] = v.q[c][q];
#pragma unroll
    for (int e = 0; e < 3; ++e) in.dF[c][e] = v.Fc[e][c][w + s[e]] - v.Fc[e][c][w];
  }
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    in.bh[e][0] = v.bh[e][w];
    in.bh[e][1] = v.bh[e][w + s[e]];
  }
}

__device__ __forceinline__ void eref_half_finish(const WbView& v, double dt, const ErefHalfIn& in) {
  const WbGeo& g = v.geo;
  const double hdt = wb_half(dt);
  double u[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    double div = __dmul_rn(in.dF[c][0], g.idx[0]);
    div = __fma_rn(in.dF[c][1], g.idx[1], div);
    div = __fma_rn(in.dF[c][2], g.idx[2], div);
    u[c] = __fma_rn(-hdt, div, in.q[c]);
  }
  const double ir = wb_rcp(u[0]);
  const double vx = __dmul_rn(u[1], ir), vy = __dmul_rn(u[2], ir), vz = __dmul_rn(u[3], ir);
  double B[3];
#pragma unroll
  for (int e = 0; e < 3; ++e) B[e] = wb_half(in.bh[e][0] + in.bh[e][1]);
  v.Erefh[0][in.w] = __fma_rn(vz, B[1], __dmul_rn(-vy, B[2]));
  v.Erefh[1][in.w] = __fma_rn(vx, B[2], __dmul_rn(-vz, B[0]));
  v.Erefh[2][in.w] = __fma_rn(vy, B[0], __dmul_rn(-vx, B[1]));
}

__device__ __forceinline__ void eref_half(const WbView& v, long long qo, long long wo, double dt,
                                          int i, int j, int k, const Nbr& nb) {
  ErefHalfIn in;
  eref_half_load(v, qo, wo, i, j, k, nb, in);
  eref_half_finish(v, dt, in);
}

// sqrt for the CFL rate; inputs below the normal range (or not > 0) give 0
__device__ __forceinline__ double wb_sqrt_fast(double x) {
  return wb_normal_pos(x) ? wb_sqrt(x) : 0.0;
}

// CFL signal rate sum_d (|v_d| + c_f,d)/dx_d of one zone (Sec. 3 fast speed)
// from 1/rho, the velocity, the gas pressure and the zone field.  The fast
// speed along d: c_f^2 = (S + sqrt(disc_d))/2 with S = a^2 + |B|^2/rho and
// disc_d = (a^2 - c_n^2)^2 + c_t^2 (c_t^2 + 2 (a^2 + c_n^2)) (the sum of
// non-negative terms), c_n^2 = B_d^2/rho, c_t^2 = |B|^2/rho - c_n^2.
//
// Written with explicit rounding: the final update (for the next step) and
// the rate of a freshly loaded state are inlined in different kernels and
// must give the same bits, or a resumed run would take a different dt.
__device__ __forceinline__ double signal_rate_core(double ir, const double vv[3], double p,
                                                   const double B[3], const WbPhys& P,
                                                   const WbGeo& g) {
  const double a2 = __dmul_rn(__dmul_rn(P.gamma, p), ir);
  double cn2[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) cn2[d] = __dmul_rn(__dmul_rn(B[d], B[d]), ir);
  const double bbi = __dadd_rn(__dadd_rn(cn2[0], cn2[1]), cn2[2]);
  const double S = __dadd_rn(a2, bbi);
  double w = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double ct2 = __dsub_rn(bbi, cn2[d]);
    const double dd = __dsub_rn(a2, cn2[d]);
    const double disc = __fma_rn(dd, dd, __dmul_rn(ct2, __fma_rn(2.0, __dadd_rn(a2, cn2[d]), ct2)));
    const double cf = wb_sqrt_fast(wb_half(__dadd_rn(S, wb_sqrt_fast(disc))));
    w = __fma_rn(__dadd_rn(wb_fabs(vv[d]), cf), g.idx[d], w);
  }
  return w;
}

// FP32 copy of a double by exponent re-biasing and mantissa truncation on the
// integer pipe (relative error below 2^-23).  Zero maps to zero; magnitudes
// outside [2^-60, 2^61), subnormals, inf and NaN clear *ok.
__device__ __forceinline__ float wb_f32_of(double x, bool* ok) {
  const long long b = __double_as_longlong(x);
  if (wb_zero(x)) return 0.0f;
  const int hi = (int)(b >> 32);
  const int ex = (hi >> 20) & 0x7ff;
  if (ex < 1023 - 60 || ex > 1023 + 60) {
    *ok = false;
    return 0.0f;
  }
  const unsigned sign = (unsigned)hi & 0x80000000u;
  const unsigned mant = (unsigned)((b >> 29) & 0x7fffff);
  return __uint_as_float(sign | ((unsigned)(ex - 1023 + 127) << 23) | mant);
}

// The CFL signal rate in FP32 (same formula as signal_rate_core, relative
// error well below 1e-5 for inputs the conversion accepts; *ok cleared when it
// cannot vouch for one).  p enters already computed in FP64, so the rate has
// no cancellation left: every term of the sum and of the discriminant is
// non-negative except a^2 - c_n^2, which only enters squared.
__device__ __forceinline__ float signal_rate_f32(double ir, const double vv[3], double p, const double B[3],
                                                 const WbPhys& P, const WbGeo& g, bool* ok) {
  const float fir = wb_f32_of(ir, ok), fp = wb_f32_of(p, ok);
  float fv[3], sq[3], fidx[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    fv[d] = fabsf(wb_f32_of(vv[d], ok));
    const float b = wb_f32_of(B[d], ok);
    sq[d] = b * b;
    fidx[d] = wb_f32_of(g.idx[d], ok);
  }
  const float a2 = P.gamma_f * fp * fir;
  float w = 0.0f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float cn2 = sq[d] * fir;
    const float ct2 = (sq[(d + 1) % 3] + sq[(d + 2) % 3]) * fir;
    const float dd = a2 - cn2;
    const float disc = dd * dd + ct2 * (ct2 + 2.0f * (a2 + cn2));
    const float cf = sqrtf(0.5f * (a2 + cn2 + ct2 + sqrtf(disc)));
    w += (fv[d] + cf) * fidx[d];
  }
  return w;
}

// The zone's exact (FP64) signal rate when it could be the largest of the
// box, else 0.  The max over zones is all the time step needs: a zone whose
// FP32 screen r32 lies below 0.9999 of the running maximum of the screens
// already seen cannot hold the largest exact rate (with screen errors e < 1e-5,
// the largest exact rate R* has r32 >= R*(1 - e) while the running maximum
// is <= R*(1 + e)), so it skips the FP64 evaluation.  The maximum of the
// returned values is bit-identical to the maximum of signal_rate_core over
// all zones.
__device__ __forceinline__ double screened_rate(double ir, const double vv[3], double p, const double B[3],
                                                const WbPhys& P, const WbGeo& g, WbScalars* scal) {
  bool ok = true;
  const float r32 = signal_rate_f32(ir, vv, p, B, P, g, &ok);
  const float G = __uint_as_float(*(volatile unsigned*)&scal->rate_screen);
  if (ok && r32 < 0.9999f * G) return 0.0;
  if (ok && r32 > G) atomicMax(&scal->rate_screen, __float_as_uint(r32));
  return signal_rate_core(ir, vv, p, B, P, g);
}

// kinetic energy density rho v^2 / 2 from the momentum and the velocity
__device__ __forceinline__ double kinetic(const double m[3], const double vv[3]) {
  return wb_half(__fma_rn(m[2], vv[2], __fma_rn(m[1], vv[1], __dmul_rn(m[0], vv[0]))));
}

// The signal rate of one stored zone (conserved state and zone field), or 0
// when the screen shows it cannot be the box's largest (screened_rate).
__device__ __forceinline__ double signal_rate(double rho, double mx, double my, double mz, double e,
                                              double bx, double by, double bz, const WbPhys& P,
                                              const WbGeo& g, WbScalars* scal) {
  const double ir = wb_rcp(rho);
  const double m[3] = {mx, my, mz};
  const double vv[3] = {mx * ir, my * ir, mz * ir};
  const double B[3] = {bx, by, bz};
  const double me = wb_half(fma(bz, bz, fma(by, by, bx * bx)));
  const double p = P.gm1 * (e - kinetic(m, vv) - me);
  if (!(rho > 0.0)) return __longlong_as_double(0x7ff8000000000000LL);
  return screened_rate(ir, vv, p, B, P, g, scal);
}

// Step 10 (+ the zone field of Step 11, floors and the next step's signal
// rate): U^{n+1} = ((U^n - dt/dx dF*) - dt/dy dG*) - dt/dz dH* at one interior
// zone, zone B = mean of b^{n+1}.  Returns the zone's signal rate (NaN if the
// state is unphysical); floor hits are added to *hits.  The rate is the one
// signal_rate gives for the stored result.  ohi: bit d set when the zone
// row's high end along d is the domain boundary of an outflow axis, whose
// boundary face the ghost fill makes a copy of the last owned face (the
// zero-gradient rule); the last zone's field then averages that copy, so the
// stored state is the one a load of the same faces gives.
__device__ __forceinline__ double final_update(const WbView& v, long long qo, long long wo,
                                               const WbPhys& P, int i, int j, int k, const Nbr& nb,
                                               int ohi, int* hits, int* bad) {
  const WbGeo& g = v.geo;
  const long long q = qo + wb_at(g, i, j, k);
  const long long wi = wo + wb_at(g, i, j, k);
  WB_CHECK_ZONE(g, i + 1, j + 1, k + 1);
  const long long (&s)[3] = nb.up;
  // explicit rounding: the same bits in every kernel this is inlined into
  const double cx = v.scal->dtdx[0], cy = v.scal->dtdx[1], cz = v.scal->dtdx[2];
  double u[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    double x = v.q[c][q];
    x = __fma_rn(-cx, __dsub_rn(v.Fc[0][c][wi + s[0]], v.Fc[0][c][wi]), x);
    x = __fma_rn(-cy, __dsub_rn(v.Fc[1][c][wi + s[1]], v.Fc[1][c][wi]), x);
    x = __fma_rn(-cz, __dsub_rn(v.Fc[2][c][wi + s[2]], v.Fc[2][c][wi]), x);
    u[c] = x;
  }
  double B[3];
  const int idx[3] = {i, j, k};
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const bool last = ((ohi >> e) & 1) && idx[e] == g.n[e] - 1;
    const double lo = v.b[e][q];
    const double hi = last ? lo : v.b[e][q + s[e]];
    B[e] = wb_half(__dadd_rn(lo, hi));
    v.q[F_BX + e][q] = B[e];
  }
  // the tests below run on the integer pipe (FP64 compares take FP64 issue)
  if (wb_below_floor(u[0], P.rho_floor)) { u[0] = P.rho_floor; ++*hits; }
  const double ir = wb_rcp(u[0]);
  const double m[3] = {u[1], u[2], u[3]};
  const double vv[3] = {__dmul_rn(u[1], ir), __dmul_rn(u[2], ir), __dmul_rn(u[3], ir)};
  const double ke = kinetic(m, vv);
  const double me = wb_half(__fma_rn(B[2], B[2], __fma_rn(B[1], B[1], __dmul_rn(B[0], B[0]))));
  double p = __dmul_rn(P.gm1, __dsub_rn(__dsub_rn(u[4], ke), me));
  if (wb_below_floor(p, P.p_floor)) {
    u[4] = __dadd_rn(__fma_rn(P.p_floor, P.inv_gm1, ke), me);
    p = __dmul_rn(P.gm1, __dsub_rn(__dsub_rn(u[4], ke), me));
    ++*hits;
  }
  const bool fin = wb_pos(u[0]) && wb_finite(u[1]) && wb_finite(u[2]) && wb_finite(u[3]) &&
                   wb_finite(u[4]) && wb_finite(p);
#pragma unroll
  for (int c = 0; c < 5; ++c) v.q[c][q] = u[c];
  if (!fin) {
    ++*bad;
    return __longlong_as_double(0x7ff8000000000000LL);
  }
  return screened_rate(ir, vv, p, B, P, g, v.scal);
}

// The shell of points outside a block of n[] zones from off[] on, dep[] zones
// deep along each axis: enumerated as the two z slabs of the padded block, then
// the two y slabs and the two x slabs of its own z (and y) range.
struct Shell {
  int off[3], n[3], dep[3];
};
__host__ __device__ __forceinline__ Shell shell_of(const WbGeo& g, int depth) {
  return {{0, 0, 0}, {g.n[0], g.n[1], g.n[2]}, {depth, depth, depth}};
}
__host__ __device__ __forceinline__ long long shell_count(const Shell& s) {
  const long long e0 = s.n[0] + 2 * s.dep[0], e1 = s.n[1] + 2 * s.dep[1];
  return e0 * e1 * (2 * s.dep[2]) + e0 * (2 * s.dep[1]) * s.n[2] + (long long)(2 * s.dep[0]) * s.n[1] * s.n[2];
}
__host__ __device__ __forceinline__ long long shell_count(const WbGeo& g, int depth) {
  return shell_count(shell_of(g, depth));
}

// Shell point t (0 <= t < shell_count) -> its zone index.
__device__ __forceinline__ void shell_point(const Shell& s, long long t, int x[3]) {
  const unsigned e0 = s.n[0] + 2 * s.dep[0], e1 = s.n[1] + 2 * s.dep[1];
  const unsigned wx = 2 * s.dep[0], wy = 2 * s.dep[1], wz = 2 * s.dep[2];
  const unsigned long long zs = (unsigned long long)e0 * e1 * wz, ys = (unsigned long long)e0 * wy * s.n[2];
  unsigned long long u = (unsigned long long)t;
  if (u < zs) {
    const unsigned r = (unsigned)(u % ((unsigned long long)e0 * e1));
    const int dz = (int)(u / ((unsigned long long)e0 * e1));
    x[0] = (int)(r % e0) - s.dep[0];
    x[1] = (int)(r / e0) - s.dep[1];
    x[2] = dz < s.dep[2] ? dz - s.dep[2] : s.n[2] + dz - s.dep[2];
  } else if ((u -= zs) < ys) {
    const unsigned per = e0 * wy;
    x[2] = (int)(u / per);
    const unsigned r = (unsigned)(u % per);
    const int dy = (int)(r / e0);
    x[0] = (int)(r % e0) - s.dep[0];
    x[1] = dy < s.dep[1] ? dy - s.dep[1] : s.n[1] + dy - s.dep[1];
  } else {
    u -= ys;
    const unsigned r = (unsigned)(u / wx);
    const int dx = (int)(u % wx);
    x[1] = (int)(r % (unsigned)s.n[1]);
    x[2] = (int)(r / (unsigned)s.n[1]);
    x[0] = dx < s.dep[0] ? dx - s.dep[0] : s.n[0] + dx - s.dep[0];
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) x[d] += s.off[d];
}

// Ghost fill of a box that is its own periodic/outflow domain (no patches):
// ghost point t of the 5-zone shell (shell_point order) copies the wrapped
// (periodic) or clamped (outflow) interior zone of the same box, all 11
// fields; face arrays use the same rule on their face index.
__device__ __forceinline__ void halo_self_offsets(const WbGeo& g, const int bc[3], long long t, long long* dst,
                                                  long long* src_off) {
  int loc[3];
  shell_point(shell_of(g, WB_NG), t, loc);
  int src[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    int x = loc[d];
    const int n = g.n[d];
    if (x < 0 || x >= n) {
      if (bc[d] == 0) x = ((x % n) + n) % n;
      else x = x < 0 ? 0 : n - 1;
    }
    src[d] = x;
  }
  *dst = wb_at(g, loc[0], loc[1], loc[2]);
  *src_off = wb_at(g, src[0], src[1], src[2]);
}

}  // namespace wbu

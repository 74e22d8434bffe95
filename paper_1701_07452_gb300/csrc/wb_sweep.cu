// MHDTVD sweep kernel: the modified flux of App. A (Eq. mhdtvd_flux2 and the
// definitions of f, beta, alpha, gamma, g, g-tilde and Q) along one axis, used
// for the predictor fluxes of Step 1 and the corrector fluxes of Steps 6-7 of
// the 3D CTU+CT integrator (Sec. "MHD in Three Dimensions").
//
// One launch takes the three axes (and the predictor's the reference EMF of
// Step 2, whose short blocks fill the tail), one thread one face: it builds the
// Roe-averaged interface state (a Cargo-Gallice type average, App. A), the
// characteristic amplitudes alpha_k, nu_k = (dt/dx) a_k and g-tilde_k, trades
// g-tilde and limited slopes with its neighbours along the pencil and emits the
// flux (wbu::sweep_tile).
//
// Eigen-structure (derived for this implementation): the linearisation
// dF = A dU with rho_ = sL sR, s-weighted v and H, opposite-weighted B_t and
// the face normal field b is the ideal-MHD Jacobian at that state with sound
// speed a_^2 = (gamma-1)(H_ - v_^2/2 - (b^2+B_t^2)/rho_) - (gamma-2) X,
// X = |dB_t|^2 / (2 (sL+sR)^2).  The waves are projected in primitive
// variables w = (rho, vn, vt, Bt, p) and sum_k beta_k R_k is accumulated in w
// and mapped to conserved variables once (the map is linear).
//
// The default entropy-fix widths vanish on the linearly degenerate waves
// (Alfven and entropy); a specialisation with those eps_k = 0 known at compile
// time drops their Q-branch arithmetic.
//
// FP64 is the scarce unit on this GPU, so the arithmetic avoids the library
// divide and square-root sequences (wb_rcp / wb_roots run on the integer pipes), and gamma_k = dg/alpha
// is never formed: Q(nu + gamma) alpha = |nu alpha + dg| sign(alpha) when
// |nu alpha + dg| >= 2 eps |alpha|, else (nu alpha + dg)^2 / (4 eps alpha) +
// eps alpha, which is the same quantity with one reciprocal, needed only for
// waves with eps > 0.
#include "wb_device.cuh"
#include "wb_internal.h"

namespace {

using wbu::kEpsZeroLD;

template <int EZ, bool PROT, bool SOFT, int LAYOUT>
__global__ void __launch_bounds__(wbu::kBlock, wbu::kSweepBlocks) k_sweep(SweepArgs A) {
  __shared__ wbu::LaneEdge X;
  wb_pdl_begin();
  if (!wb_pos(A.scal->dt)) return;
  const long long t = blockIdx.x;
  if (t >= A.tile0[3]) {  // Step 2: zone-centred reference EMF from q^n, one zone a thread
    const WbBox& e = A.ebox;
    const unsigned nx = e.hi[0] - e.lo[0] + 1, ny = e.hi[1] - e.lo[1] + 1, nz = e.hi[2] - e.lo[2] + 1;
    const unsigned z = (unsigned)(t - A.tile0[3]) * wbu::kBlock + threadIdx.x, per = nx * ny * nz;
    if (z >= per * (unsigned)A.nslots) return;
    const unsigned slot = z / per, r = z - slot * per, row = r / nx, k = row / ny;
    const long long at = wb_at(A.geo, e.lo[0] + (int)(r - row * nx), e.lo[1] + (int)(row - k * ny), e.lo[2] + (int)k);
    const double* const* q = A.s[0].q;  // the x frame: rho, Mx, My, Mz, E, Bx, By, Bz
    const long long o = slot * A.slot_in + at;
    wbu::ErefIn in;
    in.w = slot * A.slot_out + at;
    in.rho = __ldg(q[0] + o);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      in.m[c] = __ldg(q[1 + c] + o);
      in.B[c] = __ldg(q[5 + c] + o);
    }
    wbu::eref_finish(A.Eref, in);
    return;
  }
  const int d = t >= A.tile0[2] ? 2 : (t >= A.tile0[1] ? 1 : 0);
  const int hll = wbu::sweep_tile<EZ, PROT, SOFT, true, LAYOUT>(A.geo, A.box[d], d, A.s[d], t - A.tile0[d], (A.closed >> d) & 1, A.ring[d] != 0,
                                                  A.nslots, A.slot_in, A.slot_out, A.scal, A.phys, X);
  if (hll) atomicAdd((unsigned long long*)&A.scal->hll_faces, 1ULL);
}

}  // namespace

// Kernel variants: eps_k = 0 on the linearly degenerate waves (the default)
// or general eps; protection floors off (the default) or on.
void wb_launch_sweeps(SweepArgs a, cudaStream_t s) {
  const bool ez = (a.phys.eps_zero & kEpsZeroLD) == kEpsZeroLD;
  auto axis = [&](int d) {  // faces of a pencil
    return a.box[d].hi[d] - a.box[d].lo[d] + 1;
  };
  int rings = 0;
  for (int d = 0; d < 3; ++d) rings += a.ring[d] = wbu::sweep_ring(axis(d), (a.closed >> d) & 1);
  auto tiles_of = [&](int d) {
    const int U = d == 0 ? 1 : 0, W = d == 2 ? 1 : 2;
    const WbBox& b = a.box[d];
    return wbu::sweep_tiles((long long)(b.hi[U] - b.lo[U] + 1) * (b.hi[W] - b.lo[W] + 1) * a.nslots, axis(d), a.ring[d] != 0);
  };
  long long e = 0;  // tiles of the reference EMF
  if (a.Eref[0]) {
    e = a.nslots;
    for (int d = 0; d < 3; ++d) e *= a.ebox.hi[d] - a.ebox.lo[d] + 1;
    e = (e + wbu::kBlock - 1) / wbu::kBlock;
  }
  // With a block or less for each SM a scheduler has one warp: nothing hides the
  // integer products' latency, and the FP64 pipe has room for them (16^3: 18.7
  // against 22.4 us a launch; 24^3, 500 blocks: 35.1 against 28.9)
  const bool soft = tiles_of(0) + tiles_of(1) + tiles_of(2) + e > kSMs;
  // The default variant's large launches are compiled for each layout; when the
  // axes differ, all take the open one (a thin axis only as a ring)
  const bool fixed = ez && !a.phys.prot && soft && !(rings > 0 && rings < 3 && (axis(0) < 3 || axis(1) < 3 || axis(2) < 3));
  if (fixed && rings < 3)
    for (int d = 0; d < 3; ++d) a.ring[d] = 0;
  a.tile0[0] = 0;
  for (int d = 0; d < 3; ++d) a.tile0[d + 1] = a.tile0[d] + tiles_of(d);
  const dim3 grid((unsigned)(a.tile0[3] + e));
#define WB_SWEEP(...) wb_launch_dependent(k_sweep<__VA_ARGS__>, grid, wbu::kBlock, s, a)
  if (a.phys.prot) {
    if (ez) WB_SWEEP(kEpsZeroLD, true, true, wbu::kAnyLayout);
    else WB_SWEEP(0, true, true, wbu::kAnyLayout);
  } else if (!ez) {
    WB_SWEEP(0, false, true, wbu::kAnyLayout);
  } else if (!soft) {
    WB_SWEEP(kEpsZeroLD, false, false, wbu::kAnyLayout);
  } else if (!fixed || (rings == 3 && (axis(0) == 1 || axis(1) == 1 || axis(2) == 1))) {
    WB_SWEEP(kEpsZeroLD, false, true, wbu::kThin);
  } else if (rings == 3) {
    WB_SWEEP(kEpsZeroLD, false, true, wbu::kRing);
  } else {
    WB_SWEEP(kEpsZeroLD, false, true, wbu::kOpen);
  }
#undef WB_SWEEP
}

// Self-test of the FP64 reciprocal helpers against the library division and
// reciprocal square root on n inputs spread over [1e-300, 1e300].
namespace {
__global__ void k_math_selftest(int n, unsigned long long seed, unsigned long long* worst) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  double e_rcp = 0.0, e_rsq = 0.0;
  if (i < n) {
    unsigned long long z = seed + 0x9e3779b97f4a7c15ULL * (unsigned long long)(i + 1);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    z ^= z >> 31;
    double u = (double)(z >> 11) * (1.0 / 9007199254740992.0);
    double x = exp((u - 0.5) * 1381.55);
    e_rcp = fabs(wb_rcp(x) * x - 1.0);
    e_rsq = fabs(wb_rsqrt(x) / rsqrt(x) - 1.0);
  }
  atomicMax(&worst[0], (unsigned long long)__double_as_longlong(e_rcp));
  atomicMax(&worst[1], (unsigned long long)__double_as_longlong(e_rsq));
}
}  // namespace

void wb_launch_math_selftest(int n, unsigned long long* worst, cudaStream_t s) {
  k_math_selftest<<<(n + 255) / 256, 256, 0, s>>>(n, 0x1234567ULL, worst);
}

WB_CHECK_ACCESSOR(wb_check_take_sweep)

// Host-side declarations of the kernel launchers (internal to the library).
#pragma once
#include <cuda_runtime.h>

#include "wb_device.cuh"
#include "wb_pages.h"
#include "wb_units.cuh"

constexpr int kSMs = 152;  // streaming multiprocessors of the GPU this is written for

// Launch of a kernel that begins with wb_pdl_begin().  Dependent: it may be set up
// before the kernel ahead of it on the stream has finished.  Under stream capture
// that becomes a programmatic edge, whose source has to be a kernel; a launch that
// may follow anything else (a memset or copy, whatever the caller captured before
// the call) is a plain one.
template <class... P, class... A>
inline cudaError_t wb_launch(bool dependent, void (*kernel)(P...), dim3 grid, int threads, cudaStream_t s,
                             const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <class... P, class... A>
inline cudaError_t wb_launch_dependent(void (*kernel)(P...), dim3 grid, int threads, cudaStream_t s, const A&... args) {
  return wb_launch(true, kernel, grid, threads, s, args...);
}

struct wb_desc;
// Physics constants of a descriptor (gamma, CFL, eps_k, limiter, floors).
WbPhys wb_phys_of(const struct wb_desc* d);

// The sweeps along the three axes of one pass.
struct SweepArgs {
  wbu::SweepFrame s[3];    // fields (slot 0)
  long long slot_in, slot_out;
  WbGeo geo;
  WbBox box[3];            // faces along the sweep axis, zones across it
  WbPhys phys;
  WbScalars* scal;
  int nslots;
  int closed;              // bit d: the pencils along axis d are periodic and whole
  int ring[3];             // thread layout (wbu::sweep_ring; set at launch)
  long long tile0[4];      // first tile of each axis (set at launch)
  double* Eref[3];         // predictor: the reference EMF of the zones of ebox too
  WbBox ebox;              // (Eref[0] null: none)
};

// Pointers of one pipeline pass over a batch of patches: the view holds the
// slot-0 pointers; slot s of the state is at +s*slot_q, of the workspace at
// +s*slot_w.
struct StageArgs {
  WbView v;
  long long slot_q, slot_w;
  WbPhys phys;
  int nslots;
  int closed;  // axes whose neighbours wrap inside the patch (wbu::neighbours)
  // the final update's view of the domain boundary: slot s holds patch
  // p0 + s of a grid with np[] patches per axis; bit a of ohi_bc is set when
  // axis a is outflow (its high boundary face is a copy of the last owned one)
  long long p0;
  int np[3];
  int ohi_bc;
};

// Global description needed by the halo fill and by load/read scatter.
struct GridMap {
  int N[3];        // global zones
  int np[3];       // patches per axis
  int bc[3];
  long long npatch;
};

void wb_launch_sweeps(SweepArgs a, cudaStream_t s);

void wb_launch_edges(const StageArgs& a, bool corrector, const WbBox box[3], cudaStream_t s);
void wb_launch_ct(const StageArgs& a, bool final_step, const WbBox box[3], cudaStream_t s);
void wb_launch_transverse(const StageArgs& a, const WbBox box[3], cudaStream_t s);
void wb_launch_eref_half(const StageArgs& a, const WbBox& box, cudaStream_t s);
// The time-step control of a grid (wb_launch_dt_step); chain: another step
// follows, and the final update's last block prepares its dt.
struct StepControl {
  double cfl, t_end;
  int lag, chain;
  double dx[3], idx[3];
};
void wb_launch_final(const StageArgs& a, const StepControl& c, cudaStream_t s);

void wb_launch_halo(double* const q[8], double* const b[3], const WbGeo& geo, const GridMap& m,
                    cudaStream_t s);

// Arrays whose ghost points a periodic wrap fills, and the sides of the patch on
// which a later stage reads them: bit 2 d the low side of axis d, 2 d + 1 the high one.
struct WrapList {
  double* a[24];
  unsigned char sides[24];
  int n;
};
// Periodic images of the shell sh of the patches p0 .. p0 + nslots (slot = patch
// - p0); along the axes that sh has a depth for, every patch of a row is among them.
void wb_launch_wrap(const WrapList& L, const WbGeo& geo, const GridMap& m, const wbu::Shell& sh, long long p0,
                    int nslots, cudaStream_t s);
// The zone field, conserved state (from a primitive one) and first signal rate
// of a loaded state.
void wb_launch_init(double* const q[8], double* const b[3], const WbGeo& geo, long long npatch, int closed,
                    const WbPhys& ph, bool primitive, WbScalars* scal, cudaStream_t s);
// Ghost points sh of the predictor's arrays (fluxes and reference EMF) of a grid
// of one patch: a ghost row of an outflow axis holds the data of the boundary
// row, so the values there are those of the interior, copied.  face[a]: the axis
// along which array a lives on faces (computed up to the high boundary face of an
// outflow axis), or -1.
struct ImageList {
  double* a[24];
  int face[24];
  int n;
};
void wb_launch_images(const ImageList& L, const WbGeo& geo, const wbu::Shell& sh, cudaStream_t s);
// (dependent: right behind a kernel of the same call, not the first of an advance)
void wb_launch_dt_step(WbScalars* scal, const StepControl& c, cudaStream_t s, bool dependent = false);
// global <-> patch copies of up to 11 arrays; comp: 0..4 zone field, 5..7 face
// field of axis comp-5
struct MoveList {
  const double* src[11];
  double* dst[11];
  int comp[11];
  int n;
};
inline void wb_add_move(MoveList& L, const double* src, double* dst, int comp) {
  L.src[L.n] = src;
  L.dst[L.n] = dst;
  L.comp[L.n++] = comp;
}
// (plain launches, but for a gather right behind a kernel of the same call; fresh:
// the scalars of the loaded state, set to zero by the scatter)
void wb_launch_scatter(const MoveList& L, const WbGeo& geo, const GridMap& m, cudaStream_t s,
                       WbScalars* fresh = nullptr);
void wb_launch_gather(const MoveList& L, const WbGeo& geo, const GridMap& m, cudaStream_t s, bool dependent = false);
// Conserved totals: nblocks partial pairs in part (16 doubles each), the 8
// totals x vol in out (device memory).
void wb_launch_totals(double* const q[8], double* const b[3], const WbGeo& geo, long long npatch, double vol,
                      double* part, int nblocks, double* out, cudaStream_t s);
void wb_launch_divb(double* const b[3], const WbGeo& geo, long long npatch, int closed,
                    unsigned long long* out_bits, cudaStream_t s);
void wb_launch_copy_box(const double* src, long long slot, const WbGeo& geo, const WbBox& box,
                        double* dst, cudaStream_t s);
void wb_launch_fp64_probe(double* out, int blocks, int iters, cudaStream_t s);
void wb_launch_math_selftest(int n, unsigned long long* worst, cudaStream_t s);
void wb_launch_bits_selftest(int n, unsigned long long* counts, cudaStream_t s);

// check words of the translation units (checked build; 0 otherwise)
unsigned wb_check_take_sweep();
unsigned wb_check_take_stages();
unsigned wb_check_take_capi();
unsigned wb_check_take_batch();

// Internal interface between the C-ABI host code and the kernel translation
// units. Not part of the public boundary (include/sphmesh.h).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "sph_device.cuh"

namespace sph {

// Raw device pointers of one relaxation instance. The particle state (integer
// positions, colours, ids) is double-buffered: ctl->buf names the buffer that
// holds it in the current (cell-sorted at the last list build) order; the list
// rebuild gathers it into the other buffer. Views are double-buffered by
// ctl->vp (pass B writes the next step's views while pass A/B read the current).
struct DevState {
  int n = 0, dim = 2, fp64 = 0, cap = 0;
  int pass_threads = 0;  // threads per block of the pair passes (128 or 256; 0: the rules of pass_a_shape, pass_b_shape)
  void* X[2] = {nullptr, nullptr};       // int64 x, y, z (+ pad) per particle
  uint32_t* meta[2] = {nullptr, nullptr};  // colour
  uint32_t* pid[2] = {nullptr, nullptr};   // particle id
  void* view[2] = {nullptr, nullptr};    // int4 (FP32) or double4 (FP64)
  void* vbuild = nullptr;                // view at the list build with the particle's reach (FP32: build_reach, FP64: coded_reach)
  void* view32 = nullptr;                // FP64 path: FP32 view (list build; pass A's screen)
  uint32_t* key = nullptr;               // cell key (old order, rebuild only)
  uint32_t* tmp = nullptr;               // scatter slots
  uint32_t* cnt = nullptr;               // per-cell counters (all zero between rebuilds)
  uint32_t* cstart = nullptr;            // exclusive prefix of cell counts, total+1 entries
  uint32_t* scan_part = nullptr;         // per-tile counters (all zero between rebuilds)
  uint32_t total_cells = 0;
  uint32_t* list = nullptr;              // skin lists, entries (j << 8 | colour_j), see list_at
  uint32_t* lcount = nullptr;            // entries per particle; bit 31: FP32 coarse test exact
  void* plist = nullptr;                 // the force pairs of the current step (PairRec, pass A -> B), see pair_at
  uint32_t* words = nullptr;             // tape slot: the list words of its step's force pairs, see pair_at
  // staged pass A (FP32, 256-thread pair passes): per 256-target block its
  // distinct neighbours sj (kStageCap per block), their count scount (-1: not
  // staged) and the list again with ranks in that set (llist, as list)
  int stage = 0;
  uint32_t* llist = nullptr;
  int* scount = nullptr;
  int* sj = nullptr;
  uint32_t* pcount = nullptr;
  void* acc4 = nullptr;   // V4<T>: a_n and g = 0.05 rho_t r_c |a|
  void* rho = nullptr;    // T
  void* visc = nullptr;   // V4<T>: a~ (recorded steps only)
  void* pc = nullptr;     // T: p/rho^2 (general EOS only)
  Partial* partials = nullptr;
  Scalars* scal = nullptr;
  StepCtl* ctl = nullptr;
  unsigned* tickets = nullptr;
  int* err = nullptr;
  int* dbg_count = nullptr;        // 2n: density / force set sizes by particle id
  long long* dbg_sum = nullptr;    // 2n: sums of member ids
};

// Lists in tiles of one warp's 32 particles, so that everything a warp walks
// lies together and consecutive steps are constant offsets (rows across all
// particles put a warp's list words 4 n bytes apart, a page each).
// The skin list: four consecutive entries of a particle side by side, the 32
// particles' quads after one another: one 16-byte load per lane and quad, 512
// contiguous bytes per warp.
__host__ __device__ inline int list_rows(int cap) { return (cap + 3) & ~3; }
__host__ __device__ inline size_t list_at(int i, int row, int cap) {
  return ((size_t)(i >> 5) * (list_rows(cap) >> 2) + (row >> 2)) * 128 + (i & 31) * 4 + (row & 3);
}
inline size_t list_words(size_t n, int cap) { return (n + 31) / 32 * 32 * (size_t)list_rows(cap); }
// The force pairs: row k holds the k-th pair of the 32 particles (the warp
// writes them together, one pair of each lane at a time).
__host__ __device__ inline size_t pair_at(int i, int k, int cap) {
  return ((size_t)(i >> 5) * cap + k) * 32 + (i & 31);
}
// A force pair as pass A leaves it to pass B: the list word and what the viscous
// force needs of the pair's geometry, f = (1/rho_t,i^2 + 1/rho_t,j^2) (1 - q)^3
// / H^(D+2) (FP32: over a factor common to all pairs, pair_scale).
template <class T> struct PairRec;
template <> struct alignas(8) PairRec<float> { uint32_t e; float f; };
template <> struct alignas(16) PairRec<double> { double f; uint32_t e, pad; };
inline size_t pair_bytes(size_t n, int cap, bool fp64) {
  return (n + 31) / 32 * 32 * (size_t)cap * (fp64 ? sizeof(PairRec<double>) : sizeof(PairRec<float>));
}

// cells per tile of the counting sort's scan, and the tiles of a grid
constexpr int kScanTile = 4096;
constexpr size_t scan_tiles(size_t cells) { return (cells + kScanTile - 1) / kScanTile; }

// the next step rebuilds the list (after set-up or a diagnostic evaluation)
cudaError_t launch_request_rebuild(const DevState& S, cudaStream_t st);
// overwrite the control block (a kernel: no host synchronisation)
cudaError_t launch_write_ctl(const DevState& S, const StepCtl& v, cudaStream_t st);
// cell starts and scatter slots from the counts of k_rekey (predicated on ctl->rebuild)
cudaError_t build_cells(const DevState& S, cudaStream_t st);
// colours by particle id
cudaError_t launch_set_surface(const DevState& S, const uint8_t* flags, cudaStream_t st);
cudaError_t launch_get_colors(const DevState& S, uint8_t* out, cudaStream_t st);

// streaming multiprocessors of the current device (cached once per process)
inline int device_sms() {
  static const int sms = [] {
    int d = 0, v = 0;
    if (cudaGetDevice(&d) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, d) != cudaSuccess)
      return 152;
    return v > 0 ? v : 152;
  }();
  return sms;
}
// Launch of a rebuild kernel, which follows another of the same rebuild: it may
// be set up while its predecessor still runs (programmatic dependent launch) and
// waits for it on the device, by after_predecessor(), before it touches memory.
// On most steps these kernels exit at once and are mostly launch latency, which
// this hides (circle of 4,289 particles 36 -> 33 us per step). Not for kernels
// with work on every step: blocks that start early crowd onto the SMs that the
// predecessor leaves first (the reverse pass of 20,011 FP64 particles in 3D took
// 13.6 ms so, 11.5 without).
template <class... K, class... A>
inline cudaError_t launch_after(void (*kernel)(K...), int grid, int block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &attr;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, (K)args...);
}
// the successor may be set up from here on
__device__ __forceinline__ void let_successor() {
#if defined(__CUDA_ARCH__)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
}
// First statement of a kernel launched by launch_after: the predecessor is
// complete and its writes are visible; then the successor may be set up.
// (Waiting first keeps the chain: a kernel that exits at once has still waited.)
__device__ __forceinline__ void after_predecessor() {
#if defined(__CUDA_ARCH__)
  asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
  let_successor();
}

// Grid of a predicated list-rebuild kernel: grid-stride over n with at most
// per_sm blocks per SM. Most steps do not rebuild, and such a kernel then
// exits at once: with one block per 256 particles an 8M-particle grid took
// about 19 us to launch and retire its 32,768 blocks, a capped grid a few.
inline int rebuild_grid(int n, int tb, int per_sm) {
  const int g = (n + tb - 1) / tb, cap = device_sms() * per_sm;
  return g < 1 ? 1 : (g < cap ? g : cap);
}

// Small particle counts, where one thread per particle leaves most of the chip
// idle and a thread's own chain of loads (FP64: of arithmetic) is the whole
// time: several lanes share a particle. One step, us, without and with groups:
//   list build (8 lanes): 6 / 2 less for the circle (2D, FP32) of 4,289 / 16,001
//     particles, 8 / 6 for a ball (3D) of 10,001 / 16,001; at 24,001 both lose
//   FP32 pass B (8 lanes), graded hole (2D) and inclusion (3D): 4,096 29.2 / 27.2
//     and 92.3 / 90.1, 16,384 29.4 / 29.3 and 77.8 / 76.4, 20,480 31.2 / 30.6 and
//     71.8 / 73.6, 24,576 31.3 / 33.3 and 76.1 / 78.2
//   FP64 passes (4 lanes), the same: 4,096 72 / 46 and 206 / 129, 8,192 72 / 54 and
//     202 / 148, 12,288 74 / 67 and 195 / 166, 16,384 80 / 83 and 195 / 191, 24,576
//     93 / 113 and 229 / 272: the gain ends past 12,288, the line is well inside it
// (Pass A in FP32 gained nothing at any size.)
constexpr int kListLanes = 8, kListGroupMax = 20480;
constexpr int kPassLanes = 8, kPassGroupMax = 16384;
constexpr int kLanes64 = 4, kGroupMax64 = 8192;
// Threads per block of the FP64 pair passes where the caller has not chosen: one
// warp of FP64 work keeps an SM's FP64 pipe busy, so small blocks spread the
// particles evenly over the SMs. 200,003 particles in 2D, one step: 674 -> 561 us
// (256 -> 64 threads), 300,007 in 3D: 2,264 -> 2,077; the 4,096-particle square,
// 16 blocks of 256 on 152 SMs: 106 -> 74 us (32). Between 32 and 64 it matters
// little: 32,768 in 2D / 3D 107 / 246 against 115 / 267 us, 131,072 325 / 792
// against 329 / 795, 200,000 483 / 1,166 against 487 / 1,169; past the line 64
// halves the partials that the end of pass A merges.
inline int fp64_threads(int n) { return n <= (1 << 17) ? 32 : 64; }
// Launch of a pair pass: threads per block and lanes per particle. The rules
// choose where the caller has not (DevState::pass_threads); groups of lanes make
// blocks of 32 particles whatever the caller chose.
struct PassShape {
  int threads, lanes;
};
inline PassShape pass_a_shape(const DevState& S, bool groups) {
  if (!S.fp64) return {S.pass_threads == 128 ? 128 : 256, 1};
  if (groups && S.n <= kGroupMax64) return {32 * kLanes64, kLanes64};
  return {S.pass_threads ? S.pass_threads : fp64_threads(S.n), 1};
}
inline PassShape pass_b_shape(const DevState& S) {
  if (S.fp64) return pass_a_shape(S, true);
  if (S.n <= kPassGroupMax) return {32 * kPassLanes, kPassLanes};
  // large runs in small blocks, whose warps wait for no one else's tail: with 128
  // threads for 256, 8,388,608 particles in 3D 873 -> 805 us, 1,048,576 in 3D 112 ->
  // 105 and in 2D 66 -> 64, 524,288 62 -> 54 and 32 -> 31; 393,216 and 262,144 the
  // same to the event clock's 2 us, 240,370 in 3D 31 -> 33
  return {S.pass_threads ? S.pass_threads : S.n >= (1 << 19) ? 128 : 256, 1};
}

struct PassFlags {
  int general_eos = 0;  // gamma != 2: density pass first, pressure p/rho^2
  int record = 0;       // keep rho and a~ for output
  int nbr_debug = 0;    // write neighbour-set sizes and id sums by particle id
  int advance = 1;      // count this pass as a step (sigma schedule, counter)
  int move = 1;         // pass B: integrate (0: only a~, for the reverse pass)
  uint32_t* words = nullptr;  // pass B: a taped step's list words of the force pairs (DevState::words)
  const double* dt_fix = nullptr;  // pass A: prescribed {dt1, dt2} (device)
  double* dt_rec = nullptr;        // pass A: record {dt1, dt2} (device)
  const void* geo = nullptr;       // pass A: the Geom<T> of the handle (feature-surface normals)
  int surface = 0;                 // pass A: feature-surface particles may be flagged
  const Frame<float>* f32 = nullptr;  // FP64 path: frame of its FP32 views (view32), kept current
                                      // by pass B and screened on by pass A
};

// Start of a step: flip the view buffer; rebuild the list (and flip the state
// buffer) when pass B asked for it or `force` is set.
template <int D, class T>
cudaError_t launch_rebuild(const DevState& S, int force, const Grid<T>& G, const Frame<T>& F, const Geom<T>& g, T kappa,
                           cudaStream_t st, const Grid<float>* G32 = nullptr, const Frame<float>* F32 = nullptr);
template <int D, class T>
cudaError_t launch_pass_a(const DevState& S, const Frame<T>& F, const Phys<T>& P, PassFlags f, cudaStream_t st);
// the staged pass A wants the largest shared-memory carveout (5 blocks of
// 256 threads with 40 KB of staged views each); once per process
template <int D>
cudaError_t prepare_staged_pass();
// whether pass A runs staged for these flags (the variant exists for FP32,
// gamma = 2, no feature-surface particles, no neighbour diagnostics, 256 threads)
inline bool staged_pass(const DevState& S, const PassFlags& f) {
  return S.stage && !S.fp64 && S.pass_threads != 128 && !f.general_eos && !f.nbr_debug && !f.surface;
}
template <int D, class T>
cudaError_t launch_pass_b(const DevState& S, const Frame<T>& F, const Phys<T>& P, const Geom<T>& g, PassFlags f,
                          cudaStream_t st);
template <int D, class T>
cudaError_t launch_set_state(const DevState& S, const Frame<T>& F, const double* xyz, const uint8_t* col,
                             cudaStream_t st);
template <int D, class T>
cudaError_t launch_get_positions(const DevState& S, const Frame<T>& F, double* out, cudaStream_t st);
template <int D, class T>
cudaError_t launch_get_fields(const DevState& S, int which, double* out, cudaStream_t st);

// accumulated results (double slots of AdjBufs::acc)
enum AdjSlot : int {
  kAdjL = 0,       // objective value
  kAdjSigma0 = 1,  // dL/dsigma0
  kAdjGamma = 2,
  kAdjP0 = 3,
  kAdjPoly = 4,    // 8 slots: dL/dpoly[m]
  kAdjDt1b = 12,   // per step: adjoint of dt1 (reset by k_bwd_out)
  kAdjDt2b = 13,   // per step: adjoint of dt2
  kAdjMbar = 14,   // per step: adjoint of m = min r_c/|a|
  kAdjSlots = 16
};
constexpr int kAdjPartials = 12;  // doubles per block partial
constexpr int kAdjGroup = 64;     // blocks whose partials are added together first

template <class T>
struct AdjBufs {
  const double* gin = nullptr;  // n x D by id: adjoint of the state the step produced (or the seed)
  double* gout = nullptr;       // n x D by id: adjoint of the state it started from
  V4<double>* xb = nullptr;     // current order: adjoint of x (accumulating)
  V4<T>* atb = nullptr;         // adjoint of a~
  V4<T>* ab = nullptr;          // adjoint of a
  T* hb = nullptr;              // adjoint of h
  T* Tb = nullptr;              // adjoint of T = 1/rho_t^2
  T* rtb = nullptr;             // adjoint of rho_t
  T* rhob = nullptr;            // adjoint of rho
  double* part = nullptr;       // kAdjPartials per block
  double* acc = nullptr;        // kAdjSlots
  unsigned* ticket = nullptr;
};

// reverse pass of one step whose state, lists and forward quantities (a tape
// slot) are in S; B.gin -> B.gout
template <int D, class T>
cudaError_t launch_bwd_step(const DevState& S, const Frame<T>& F, const Phys<T>& P, const Geom<T>& geo,
                            const AdjBufs<T>& B, int recomputed_dt, int general_eos, cudaStream_t st);
// objective at the current state (list in place) and its gradient -> B.gout;
// B.gin (may be null) is an extra seed added to dL/dx
template <int D, class T>
cudaError_t launch_objective(const DevState& S, const Frame<T>& F, const Phys<T>& P, const Geom<T>& geo,
                             const AdjBufs<T>& B, double wd, double lambda, cudaStream_t st);

// copy the state pass A used (current order: X, meta, pid, view), ctl and
// scal into tape.X[0], meta[0], pid[0], view[0], ctl, scal
template <int D, class T>
cudaError_t launch_tape_snapshot(const DevState& S, const DevState& tape, cudaStream_t st);

// per-colour volume sum m/rho and particle count over the current order (rho
// of the last pass A); vpart/cpart hold color_volume_blocks(n) x 256 partials,
// vol/cnt 256 results (device)
int color_volume_blocks(int n);
template <class T>
cudaError_t launch_color_volumes(const DevState& S, double* vpart, unsigned long long* cpart, double* vol,
                                 long long* cnt, cudaStream_t st);

// initial sampling (create)
struct FieldBounds {
  double sum_w, min_seff, max_seff, max_w;
};
template <int D>
cudaError_t field_bounds(const Geom<double>& g, int res, FieldBounds* host_out, double* scratch,
                         cudaStream_t st);
int field_bounds_scratch_doubles();
template <int D>
cudaError_t sample_positions(const Geom<double>& g, int n, int n_colors, uint64_t seed, double wmax,
                             double* xyz, uint8_t* col, double* gens, int* err, cudaStream_t st);

}  // namespace sph

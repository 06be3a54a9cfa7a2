// C ABI of the coupled lattice-Boltzmann ice-crystal step (include/lbmice.h): parameter
// derivation, device state, kernel launches and CUDA-graph replay of step chunks.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <type_traits>
#include <utility>
#include <vector>

#include "../../include/lbmice.h"
#include "lbmice_adjoint.cuh"
#include "lbmice_aux.cuh"
#include "lbmice_step.cuh"
#include "lbmice_row.cuh"
#include "lbmice_step2.cuh"

using namespace lbmice;

namespace {

constexpr double kA2 = 0.6267;   // Sec. 2.1: a2 of the sharp-interface mapping
constexpr double kHdrag = 2.757; // Sec. 2.2.1: drag constant h
// Steps per captured graph: a multiple of 12, so the population double buffer and the phi
// planes (3 or 4 of them) are back in their slots after each replay, whether its launches take
// one step or two.
constexpr int kGraphSteps = 60;
// A graph is captured once a grid has taken this many steps by single launches: capture and
// instantiation cost about as much as they save over 300 steps.
constexpr int kGraphAfter = 4 * kGraphSteps;
constexpr int kMaxGridY = 65535; // blocks a launch may have in y
constexpr int kStatBlocks = 608; // 4 x 152 SMs
constexpr int kMaxPhi = 4;       // phi planes: 3, or 4 where launches take two steps
// two steps by tiles up to here (two_tile_warps has the times of both forms)
constexpr long long two_tile_max(bool flow) { return flow ? 11LL << 16 : 1LL << 21; }
// stencils that reach two nodes: pairs up to the first and from the second on (two_possible), the
// latter by tiles up to the third where a grid has no flow (two_tile_warps)
constexpr long long kTwoFarSmall = 1LL << 16, kTwoFarLarge = 9LL << 16, kTwoFarTileNodes = 3LL << 19;
// 16-bit storage in pairs up to here: bound by issue, the redundant collisions of the tiles cost it
// more than what they save in launches beyond (F16 with flow, us per step, pairs / single: 256^2
// 3.4 / 5.2, 512^2 10.1 / 11.6, 1024^2 36.1 / 34.6)
constexpr long long kTwoDevMaxNodes = 1LL << 18;
constexpr int kBatchTwoRows = 64;        // segment height of a batch's two-step march
// warps of the largest two-step tile (two CTAs per SM), with and without flow
template <bool FLOW>
constexpr int kTileWide = FLOW ? 16 : 20;
// nodes of a batched launch up to which it takes two-step tiles
constexpr long long kBatchTileMaxNodes = 1LL << 20;
// nodes up to which members of the march shape that otherwise step in pairs take a single step in
// 32 x 8 tiles: a march's few CTAs leave most of the GPU idle. us per step, march / tiles, without
// flow: four of 64^2 18.8 / 4.0, 32 of 128^2 26.8 / 19.0, 12 of 256^2 29.7 / 29.3, 24 of 256^2 58.0 /
// 55.0, eight of 512^2 67.7 / 70.9; with flow: four of 64^2 21.6 / 4.9, 32 of 128^2 35.2 / 29.0, 12 of
// 256^2 39.2 / 41.9, 17 of 256^2 57.6 / 56.9, 24 of 256^2 75.5 / 77.2
constexpr long long batch_single_tile_nodes(bool flow) { return flow ? 11LL << 16 : 3LL << 19; }
constexpr int kBatchTileWarps = 16;      // warps of a batch's two-step tiles
constexpr int kMaxPhases = 2 * kMaxPhi;  // population slot x phi plane
constexpr long long kTapePairsMaxNodes = 1LL << 19;  // segment states recomputed in pairs up to here
constexpr int kTapeGraphSegments = 6;  // full segments from which the reverse sweep uses graphs
constexpr int kMapsPerPhase = 6; // tensor maps of one step's inputs (StepPtrs::tm)

}  // namespace

namespace {

// Several device buffers in one allocation: place() each, allocate(), and the pointers given to
// place() are set. cudaMalloc and cudaFree cost about 40 us each whatever the size (a 512^2
// gradient's work space of 100 states: 4.5 ms + 4.3 ms in pieces, 0.14 + 1.1 ms as one).
class Slab {
 public:
  template <class T>
  void place(T** p, size_t bytes) {
    items_.push_back({reinterpret_cast<void**>(p), size_});
    size_ += (bytes + 1023) / 1024 * 1024;
  }
  cudaError_t allocate(void** base) {
    const cudaError_t e = cudaMalloc(base, size_);
    if (e != cudaSuccess) {
      *base = nullptr;
      return e;
    }
    for (const Item& i : items_) *i.p = static_cast<char*>(*base) + i.offset;
    return e;
  }
  size_t bytes() const { return size_; }

 private:
  struct Item {
    void** p;
    size_t offset;
  };
  std::vector<Item> items_;
  size_t size_ = 0;
};

}  // namespace

struct lbmice_ctx {
  lbmice_params p;
  Consts C;
  double Dphi3, lambda;
  int device = 0;
  cudaStream_t stream = nullptr;   // caller's stream: every launch goes here
  cudaStream_t capture = nullptr;  // private stream used only to record graphs
  int nplanes = 0;
  size_t elem = 4;                 // bytes per stored population
  void* slab = nullptr;            // the device allocation holding every buffer below
  void* pops[2] = {nullptr, nullptr};
  float* phi[kMaxPhi] = {};        // phi^n is plane ring mod nphi, phi^{n-1} the one before
  int nphi = 3;                    // phi planes in use; 4: steps are taken in pairs (two_kernel)
  bool pad_used = false;           // host exports wrote over the padding columns of a phi plane
  int cur = 0;                     // population buffer (Um, rhom) holding the current state
  float* Um[2] = {nullptr, nullptr};   // 16-bit storage: U (zeroth moment of g), ping-pong
  float* rhom[2] = {nullptr, nullptr}; // 16-bit storage with flow: rho, ping-pong
  double* stat_partial = nullptr;
  double* stat_host = nullptr;     // pinned, in one block with tip_host
  double* tip_host = nullptr;      // pinned: (cos, sin) of up to LBMICE_MAX_RAYS rays, then their radii
                                   //   (8 doubles after stat_host)
  cudaGraphExec_t graph[kMaxPhases] = {};  // kGraphSteps steps from each buffer phase
  bool tile_step = false;          // single steps of the other stencils and folds: tile_kernel
  int tile_warps = 0;              // two-step launches: warps of a tile CTA, 0: the march
  int64_t step = 0;                // steps since the last init
  int64_t ring = 0;                // the same, but for steps that left the planes where they were
                                   //   (Phase::turn)
  int64_t taken = 0;               // steps launched one by one since create (kGraphAfter)
  // tensor maps of the march, kMapsPerPhase per buffer phase, in device memory
  CUtensorMap* tmaps = nullptr;
};

namespace {

inline dim3 node_grid(const Consts& C, dim3 blk) {
  return dim3((C.nx + blk.x - 1) / blk.x, (C.ny + blk.y - 1) / blk.y);
}

// name of the last CUDA error this thread turned into an error code (lbmice_last_error)
thread_local const char* g_last_cuda_error = "none";

int cuda_err(cudaError_t e) {
  if (e == cudaSuccess) return LBMICE_OK;
  g_last_cuda_error = cudaGetErrorName(e);
  return e == cudaErrorMemoryAllocation ? LBMICE_ENOMEM : LBMICE_ECUDA;
}

#define LB_TRY(expr)                          \
  do {                                        \
    int rc_ = cuda_err(expr);                 \
    if (rc_ != LBMICE_OK) return rc_;         \
  } while (0)

int validate(const lbmice_params& p) {
  if (p.nx < 4 || p.ny < 4) return LBMICE_EINVAL;
  const long long pitch = ((long long)p.nx + 31) / 32 * 32;
  if (pitch * p.ny >= (1LL << 31)) return LBMICE_EINVAL;
  if (!(p.dx > 0) || !(p.dt > 0) || !(p.W0 > 0) || !(p.tau0 > 0)) return LBMICE_EINVAL;
  if (!(p.D >= 0) || !(p.eps >= 0 && p.eps < 1) || !(p.kappa_N >= 0)) return LBMICE_EINVAL;
  if (!std::isfinite(p.L_sat) || !std::isfinite(p.U_in) || !std::isfinite(p.lambda))
    return LBMICE_EINVAL;
  for (int f = 0; f < 4; ++f)
    if (p.bc[f] < LBMICE_BC_PERIODIC || p.bc[f] > LBMICE_BC_FREESLIP) return LBMICE_EINVAL;
  if ((p.bc[0] == LBMICE_BC_PERIODIC) != (p.bc[1] == LBMICE_BC_PERIODIC)) return LBMICE_EINVAL;
  if ((p.bc[2] == LBMICE_BC_PERIODIC) != (p.bc[3] == LBMICE_BC_PERIODIC)) return LBMICE_EINVAL;
  if (p.flow != 0 && p.flow != 1) return LBMICE_EINVAL;
  if (p.check_every < 0) return LBMICE_EINVAL;
  if (p.storage < LBMICE_STORAGE_F32 || p.storage > LBMICE_STORAGE_BF16) return LBMICE_EINVAL;
  if (p.stencil != 0 && p.stencil != 2 && p.stencil != 4 && p.stencil != 6 && p.stencil != 8)
    return LBMICE_EINVAL;
  if (p.fold != 0 && p.fold != 4 && p.fold != 6) return LBMICE_EINVAL;
  if (!std::isfinite(p.u_in) || std::fabs(p.u_in) >= std::sqrt(1.0 / 3.0)) return LBMICE_EUNSTABLE;
  if (p.flow && !(p.nu > 0)) return LBMICE_EUNSTABLE;  // tau_f = 3 nu + 1/2 must exceed 1/2
  return LBMICE_OK;
}

void derive(lbmice_t* h) {
  const lbmice_params& p = h->p;
  Consts& C = h->C;
  std::memset(&C, 0, sizeof(C));
  C.nx = p.nx;
  C.ny = p.ny;
  C.pitch = (p.nx + 31) / 32 * 32;
  C.pstride = (long long)C.pitch * p.ny;  // plane-major: [plane][ny][pitch]
  C.rstride = C.pitch;
  for (int f = 0; f < 4; ++f) C.bc[f] = p.bc[f];
  C.stencil = p.stencil == 0 ? 4 : p.stencil;
  C.fold = p.fold == 0 ? 6 : p.fold;
  const double Dphi = (p.W0 * p.W0 / p.tau0) * p.dt / (p.dx * p.dx);
  h->Dphi3 = 3.0 * Dphi;
  h->lambda = p.lambda > 0 ? p.lambda : p.tau0 * p.D / (kA2 * p.W0 * p.W0);
  const double Wlat = p.W0 / p.dx;
  const double tau_f = p.nu * 3.0 + 0.5;
  C.Dphi3 = (float)h->Dphi3;
  C.dt_tau0 = (float)(p.dt / p.tau0);
  C.lambda = (float)h->lambda;
  C.Dlat3 = (float)(3.0 * p.D * p.dt / (p.dx * p.dx));
  C.half_Lsat = (float)(0.5 * p.L_sat);
  C.eps = (float)p.eps;
  C.kNkeps = (float)(p.kappa_N * C.fold * p.eps);
  C.kdrag = (float)(kHdrag * p.nu / (4.0 * Wlat * Wlat));
  C.inv_tau_f = (float)(1.0 / tau_f);
  C.guo = (float)(1.0 - 0.5 / tau_f);
  C.U_in = (float)p.U_in;
  const double nxs[4] = {1, -1, 0, 0}, nys[4] = {0, 0, 1, -1};
  for (int f = 0; f < 4; ++f) {
    C.uin_x[f] = (float)(p.u_in * nxs[f]);
    C.uin_y[f] = (float)(p.u_in * nys[f]);
  }
}

void release(lbmice_t* h) {
  for (cudaGraphExec_t g : h->graph) if (g) cudaGraphExecDestroy(g);
  if (h->slab) cudaFree(h->slab);
  if (h->stat_host) cudaFreeHost(h->stat_host);
  if (h->capture) cudaStreamDestroy(h->capture);
  delete h;
}

// bytes of one population buffer: nplanes planes of ny rows of pitch values, whatever the
// interleaving of planes and rows
size_t pop_bytes(const lbmice_t* h) {
  return h->elem * (size_t)h->nplanes * (size_t)h->C.pitch * (size_t)h->C.ny;
}
size_t field_bytes(const lbmice_t* h) {
  return sizeof(float) * (size_t)h->C.pitch * (size_t)h->C.ny;
}
bool dev16(const lbmice_t* h) { return h->p.storage != LBMICE_STORAGE_F32; }
// phi^n and phi^{n-1} of the current state
float* phi_now(const lbmice_t* h) { return h->phi[h->ring % h->nphi]; }
float* phi_prev(const lbmice_t* h) { return h->phi[(h->ring + h->nphi - 1) % h->nphi]; }
// The plane that the next step writes: free until then, it takes one contiguous field at a time on
// its way to the host, so that the fourth plane of a grid in pairs costs no memory beside it. The
// field runs over the padding columns, which only a state shows (clear_plane_padding).
float* free_plane(const lbmice_t* h) { return h->phi[(h->ring + 1) % h->nphi]; }

// Where the buffers of a grid stand: the population slot and the count s whose plane, s mod nphi,
// is phi^n. A launch of one or two steps reads slot cur and writes the other.
struct Phase {
  int cur;
  int64_t s;
  // 0 .. 5: the next of six single steps that go twice around three of the planes, phi^{n-1}, phi^n
  // and the one after, and so end where they began (cur and s are those of the beginning)
  int turn = -1;
  void advance(int steps) {
    if (turn >= 0) {
      turn = turn == 5 ? -1 : turn + 1;
      return;
    }
    cur ^= 1;
    s += steps;
  }
};
Phase phase_of(const lbmice_t* h) { return {h->cur, h->ring}; }
int phase_index(const lbmice_t* h, Phase f) { return f.cur * h->nphi + (int)(f.s % h->nphi); }

// cuTensorMapEncodeTiled of the driver, through the runtime's entry-point query (no link
// against the driver library).
PFN_cuTensorMapEncodeTiled_v12000 encode_tiled() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// A tiled tensor map of rank 2 or 3 over base: dims[0] the contiguous extent (elements),
// strides[i] the bytes between steps of dimension i + 1, box the box extents.
bool encode_map(CUtensorMap* m, CUtensorMapDataType t, int rank, const void* base,
                const uint64_t* dims, const uint64_t* strides, const uint32_t* box) {
  auto fn = encode_tiled();
  if (!fn) return false;
  cuuint64_t d[3], st[2];
  cuuint32_t b[3], es[3] = {1, 1, 1};
  for (int i = 0; i < rank; ++i) {
    d[i] = dims[i];
    b[i] = box[i];
  }
  for (int i = 0; i + 1 < rank; ++i) st[i] = strides[i];
  return fn(m, t, (cuuint32_t)rank, const_cast<void*>(base), d, st, b, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

// The maps of every step phase (the boxes of one march pass: 8 rows of a strip), encoded on
// the host and copied to the device once; the buffers never move.
int make_tensor_maps(lbmice_t* h) {
  // Every storage: phi^n in boxes of 8 rows x 40 columns, the march's phi ring blocks (slot
  // 5). The L2 prefetch boxes (slots 0..4) for 16-bit storage only: FP32 storage runs the
  // plain march, since prefetching its bandwidth-bound steps measured 15 B per node of
  // extra DRAM reads and no gain, while the issue-bound 16-bit steps gain 3%.
  const int phases = 2 * h->nphi;
  std::vector<CUtensorMap> maps(phases * kMapsPerPhase);
  std::memset(maps.data(), 0, sizeof(CUtensorMap) * maps.size());
  const uint64_t P = h->C.pitch, NY = h->C.ny, Q = h->C.pstride;
  const uint32_t R = kMarchRows;
  bool ok = true;
  for (int ph = 0; ph < phases && ok; ++ph) {  // phase: population slot x nphi + phi plane
    const int cur = ph / h->nphi, i = ph % h->nphi;
    CUtensorMap* m = &maps[ph * kMapsPerPhase];
    const char* pin = static_cast<const char*>(h->pops[cur]);
    const uint64_t d1[2] = {P, NY}, s1[1] = {P * 4};
    const uint32_t b1[2] = {36, R}, b5[2] = {kMarchPW, R};
    ok = ok && encode_map(&m[5], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, h->phi[i], d1, s1, b5);
    if (!dev16(h)) continue;
    const uint32_t L = h->p.flow ? 3 : 2;
    const uint64_t dv[3] = {8 * P, NY, L}, sv[2] = {16 * P, 18 * Q};
    const uint32_t bv[3] = {256, R, L};
    ok = ok && encode_map(&m[0], CU_TENSOR_MAP_DATA_TYPE_UINT16, 3, pin, dv, sv, bv);
    ok = ok && encode_map(&m[1], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, h->Um[cur], d1, s1, b1);
    if (h->p.flow)
      ok = ok && encode_map(&m[2], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, h->rhom[cur], d1, s1, b1);
    ok = ok && encode_map(&m[4], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
                          h->phi[(i + h->nphi - 1) % h->nphi], d1, s1, b1);
  }
  if (!ok) return LBMICE_ECUDA;
  LB_TRY(cudaMemcpy(h->tmaps, maps.data(), sizeof(CUtensorMap) * maps.size(),
                    cudaMemcpyHostToDevice));
  return LBMICE_OK;
}

// Run f with a tag value of the handle's storage type.
template <class Fn>
int with_storage(const lbmice_t* h, Fn&& fn) {
  switch (h->p.storage) {
    case LBMICE_STORAGE_F16: return fn(F16{});
    case LBMICE_STORAGE_BF16: return fn(BF16{});
    default: return fn(F32{});
  }
}

// Segment height of the march for one grid on a device of sms SMs (4 CTAs per SM). Each
// segment collides two rows below its first in a prologue pass, and the last wave of CTAs
// may fill the GPU only in part; among heights of 40 .. 96 rows (multiples of the 8-row pass)
// that give at least one and a half waves, take the one that maximises
// (waves / waves begun) x H / (H + 2). A grid too small for any of them takes the tallest of
// 32, 16 rows that gives one and a half waves, else 8. (A batch, which has CTAs enough, walks
// every member in segments of 64.) At 2048 x 2048 on 152 SMs: 80 rows, 1794 CTAs, 2.95 waves.
int march_seg_rows(int nx, int ny, int sms) {
  const long long slots = 4LL * sms;
  const auto units = [&](int H) { return (long long)march_strips(nx) * ((ny + H - 1) / H); };
  int best = 0;
  double best_score = 0.0;
  for (int H = 40; H <= 96; H += kMarchRows) {
    const long long u = units(H);
    if (2 * u < 3 * slots) continue;
    const double waves = (double)u / (double)slots;
    const double score = waves / std::ceil(waves) * H / (H + 2.0);
    if (score > best_score) {
      best_score = score;
      best = H;
    }
  }
  if (best) return best;
  for (int H = 32; H > kMarchRows; H /= 2)
    if (2 * units(H) >= 3 * slots) return H;
  return kMarchRows;
}

// Segments of the two-step march: H rows each (a multiple of 8), the first one beginning
// two_pad(ny) rows below row 0.
int two_segments(int ny, int H) { return (ny + two_pad(ny) + H - 1) / H; }
// Tiles of W warps above one another.
int two_tiles(int ny, int W, int v = TWO_DEFAULT) {
  const int rows = W - 2 * two_rim(v);
  return (ny + rows - 1) / rows;
}
int two_variant(const Consts& C) {
  if (C.stencil > 4) return TWO_FAR;
  return C.stencil == 4 && C.fold == 6 ? TWO_DEFAULT : TWO_NEAR;
}
// Whether a grid takes its steps in pairs where a fourth phi plane fits: FP32 storage; stencils that
// reach two nodes on periodic grids only (their ghosts at other faces would be two deep), where the
// rim of four costs less than the second launch or the second pass over memory. E8 without flow, us
// per step, pairs / single steps: 100^2 2.1 / 2.7, 200^2 2.9 / 3.1, 500^2 9.5 / 8.8, 700^2 16.1 / 15.5,
// 800^2 20.2 / 21.3, 900^2 25.4 / 28.7, 1500^2 59 / 73; with flow 800^2 29.1 / 30.5, 900^2 35.1 / 38.1;
// the four-fold E4 500^2 7.4 / 8.3, 1500^2 51 / 72.
bool two_possible(const lbmice_params& p, const Consts& C) {
  if (p.storage != LBMICE_STORAGE_F32)
    return two_variant(C) == TWO_DEFAULT && (long long)C.nx * C.ny <= kTwoDevMaxNodes;
  if (two_variant(C) != TWO_FAR) return true;
  for (int f = 0; f < 4; ++f)
    if (C.bc[f] != BC_PERIODIC) return false;
  const long long nodes = (long long)C.nx * C.ny;
  return C.nx >= 8 && C.ny >= 8 && (nodes <= kTwoFarSmall || nodes >= kTwoFarLarge);
}

// Warps of the tile CTAs a grid takes its two-step launches with; 0: the two-step march. Small
// grids are bound by the chain of dependent phases, so the fewest rows per CTA whose CTAs still
// all fit at two per SM; then the largest that fills the SM with two CTAs (16 warps; without flow,
// whose state is smaller, 20: 400^2 5.6 -> 5.2 us per step, 1024^2 26.7 -> 24.9) until the march's
// fewer collisions win. us per step, tiles of 8 / 12 / 16 warps / march, without flow:
// 64^2 1.65 / 1.86 / 2.12 / 3.3, 128^2 1.96 / 1.90 / 2.10 / 3.4, 256^2 4.2 / 3.2 / 2.7 / 4.4,
// 512^2 12.3 / 9.0 / 7.4 / 9.2; 1024^2 26.7 of 16 warps, and one CTA per SM of 24, 28 or 32 warps
// 33.3, 31.7, 30.1; 20 warps / march: 800^2 15.8 / 17.6, 1024^2 24.9 / 26.8, 1200^2 33.2 / 34.2,
// 1300^2 38.0 / 39.1, 1400^2 44.1 / 43.9, 1448^2 46.6 / 47.5; E8, 20 warps / march: 800^2 20.2 / 21.2,
// 1024^2 31.5 / 32.4, 1200^2 42.4 / 42.1, 1254^2 46.3 / 43.7 (the limit lies 50^2 too high since the
// march has a split barrier); with flow, 16 warps / march: 700^2 18.6 / 19.6, 750^2 21.1 / 23.0, 800^2
// 23.6 / 25.2, 840^2 26.1 / 25.5, 1024^2 37.0 / 36.1, 1800 x 500 32.4 / 30.1, 2048^2 140 / 116.
int two_tile_warps(const Consts& C, bool flow, bool dev, int sms) {
  const int v = two_variant(C);
  const long long most = v == TWO_FAR ? (flow ? kTwoFarSmall : kTwoFarTileNodes)
                                      : two_tile_max(flow);
  if ((long long)C.nx * C.ny > most) return 0;
  for (int W : {8, 12, 16}) {
    if (W == 8 && (v != TWO_DEFAULT || dev)) continue;
    if ((long long)two_strips(C.nx, v) * two_tiles(C.ny, W, v) <= 2LL * sms) return W;
  }
  return flow || dev ? 16 : kTileWide<false>;
}

// Whether single steps of the other stencils and folds go by tile_kernel, not row_kernel (four CTAs
// of either per SM): where row tiles need more than one wave and 32 x 8 tiles do not, or need over 1.55
// times as many CTAs, what a tile's CTA takes longer. us per step, row / tile, E6 and E8 without flow:
// 126 x 786 5.48 / 4.92, 277 x 531 6.18 / 5.86, 128 x 1929 9.19 / 9.00, 32 x 10159 17.8 / 12.5; 800^2
// 21.3 / 22.8, 100^2 2.7 / 3.7.
bool one_step_tiles(const Consts& C, int sms) {
  const long long slots = 4LL * sms, rows = (long long)march_strips(C.nx) * ((C.ny + 5) / 6);
  const long long tiles = (long long)((C.nx + 31) / 32) * ((C.ny + 7) / 8);
  return rows > slots && (C.ny + 7) / 8 <= kMaxGridY && (tiles <= slots || 1.55 * tiles < rows);
}

// Whether a narrow grid loses by steps in pairs: one that fills the GPU, where a pair's strips of 26
// (or 24) columns are half as many again as a single step's, or where a single strip is all there is,
// mostly empty, and a pair's rim of rows costs more than the launch and the L2 traffic it saves. us per
// step, pairs / single steps, with flow: the four-fold 27 x 9658 26.7 / 14.8, 17 x 9246 15.0 / 13.5; the
// default scheme 9 x 19156 26.9 / 24.1, 57 x 3621 13.5 / 12.8; without flow: E2 30 x 13508 23.8 / 13.8,
// 32 x 4108 7.9 / 5.3, 56 x 1751 5.1 / 4.2; E6 51 x 18210 46.1 / 39.2.
bool too_narrow_for_pairs(const Consts& C, bool flow, bool dev, int sms) {
  const int v = two_variant(C), W = two_tile_warps(C, flow, dev, sms), two = two_strips(C.nx, v);
  if (W && (long long)two * two_tiles(C.ny, W, v) <= 2LL * sms) return false;
  const int one = v == TWO_DEFAULT ? march_strips(C.nx) : std::min(march_strips(C.nx), (C.nx + 31) / 32);
  return 2 * two >= 3 * one || (flow && one == 1);
}

// Segment height of the two-step march on slots CTA places: the rounds of CTAs it takes and about 3
// more of first and last ones that run partly full, times the rows and the 36 rows' time that a
// CTA's prologue pass and first loads cost. Fitted to the times of 18 grids (1200^2 to 4096^2 with
// and without flow, 1800 x 900, E8) at 24 to 128 rows: 0.6% above each grid's best height on
// average, 2.2% at most (with a full barrier where the march now has a split one, which takes about
// 6% off each). Fractional rounds + 0.5 and a prologue of 5 rows, the model before, chose heights
// 2.7% above on average: 1200^2 with flow 51.3 -> 48.9 us per step, 1600^2 81.3 -> 78.2, 900 x 1800
// 55.7 -> 53.6; without flow 2400^2 116 -> 113.6, 4096^2 311 -> 305.
int two_seg_rows(int nx, int ny, int v, int slots) {
  int best = kTwoRows;
  double best_time = 0.0;
  for (int H = kTwoRows; H <= 128; H += kTwoRows) {
    const double units = (double)two_strips(nx, v) * two_segments(ny, H);
    const double t = (std::ceil(units / slots) + 3.0) * (H + 36.0);
    if (best_time == 0.0 || t < best_time) {
      best_time = t;
      best = H;
    }
  }
  return best;
}

// Launch grid of the march over one grid: one CTA per (strip, segment of H rows).
long long march_units(const Consts& C, int H) {
  return (long long)march_strips(C.nx) * ((C.ny + H - 1) / H);
}
dim3 march_grid(const Consts& C) {
  return dim3(march_strips(C.nx), (C.ny + C.seg_rows - 1) / C.seg_rows);
}

// Opt the march kernels of this storage into the shared memory they use (above 48 KB).
int march_attributes(const lbmice_t* h) {
  return with_storage(h, [&](auto tag) -> int {
    using S = decltype(tag);
    cudaError_t e = cudaSuccess;
    auto set = [&](auto kern, size_t bytes) {
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    const auto set_tiles = [&](auto width) {
      constexpr int W = decltype(width)::value;
      set(two_tile_kernel<true, W>, TileTwoSmem<true, W>::bytes());
      set(two_tile_kernel<false, W>, TileTwoSmem<false, W>::bytes());
      set(two_tile_kernel<true, W, true>, TileTwoSmem<true, W>::bytes());
      set(two_tile_kernel<false, W, true>, TileTwoSmem<false, W>::bytes());
    };
    (void)set_tiles;
    set(march_kernel<true, S, MARCH_PREFETCH>, march_smem_bytes<true>());
    set(march_kernel<false, S, MARCH_PREFETCH>, march_smem_bytes<false>());
    set(march_kernel<true, S, MARCH_PLAIN>, march_smem_bytes<true>());
    set(march_kernel<false, S, MARCH_PLAIN>, march_smem_bytes<false>());
    constexpr int M = Storage<S>::DEV ? MARCH_PREFETCH : MARCH_PLAIN;
    set(batch_march_kernel<true, S, M>, march_smem_bytes<true>());
    set(batch_march_kernel<false, S, M>, march_smem_bytes<false>());
    if constexpr (Storage<S>::DEV) {
      set(two_tile_kernel<true, 12, false, TWO_DEFAULT, S>, TileTwoSmem<true, 12>::bytes());
      set(two_tile_kernel<true, 16, false, TWO_DEFAULT, S>, TileTwoSmem<true, 16>::bytes());
      set(two_tile_kernel<false, 12, false, TWO_DEFAULT, S>, TileTwoSmem<false, 12>::bytes());
      set(two_tile_kernel<false, 16, false, TWO_DEFAULT, S>, TileTwoSmem<false, 16>::bytes());
    } else {
      set_tiles(std::integral_constant<int, 8>{});
      set_tiles(std::integral_constant<int, 12>{});
      set_tiles(std::integral_constant<int, 16>{});
      set(batch_two_tile_kernel<true, kBatchTileWarps>, TileTwoSmem<true, kBatchTileWarps>::bytes());
      set(batch_two_tile_kernel<false, kBatchTileWarps>, TileTwoSmem<false, kBatchTileWarps>::bytes());
      constexpr int WIDE = kTileWide<false>;
      set(two_tile_kernel<false, WIDE>, TileTwoSmem<false, WIDE>::bytes());
      set(two_tile_kernel<false, WIDE, true>, TileTwoSmem<false, WIDE>::bytes());
      set(two_tile_kernel<false, WIDE, false, TWO_NEAR>, TileTwoSmem<false, WIDE, TWO_NEAR>::bytes());
      set(two_tile_kernel<false, WIDE, false, TWO_FAR>, TileTwoSmem<false, WIDE, TWO_FAR>::bytes());
      set(two_kernel<true, TWO_DEFAULT>, TwoSmem<true>::bytes());
      set(two_kernel<false, TWO_DEFAULT>, TwoSmem<false>::bytes());
      set(two_kernel<true, TWO_NEAR>, TwoSmem<true>::bytes());
      set(two_kernel<false, TWO_NEAR>, TwoSmem<false>::bytes());
      set(two_kernel<true, TWO_FAR>, TwoSmem<true, TWO_FAR>::bytes());
      set(two_kernel<false, TWO_FAR>, TwoSmem<false, TWO_FAR>::bytes());
      set(two_tile_kernel<true, 16, false, TWO_NEAR>, TileTwoSmem<true, 16, TWO_NEAR>::bytes());
      set(two_tile_kernel<false, 16, false, TWO_NEAR>, TileTwoSmem<false, 16, TWO_NEAR>::bytes());
      set(two_tile_kernel<true, 16, false, TWO_FAR>, TileTwoSmem<true, 16, TWO_FAR>::bytes());
      set(two_tile_kernel<false, 16, false, TWO_FAR>, TileTwoSmem<false, 16, TWO_FAR>::bytes());
      set(batch_two_kernel<true>, TwoSmem<true>::bytes());
      set(batch_two_kernel<false>, TwoSmem<false>::bytes());
    }
    return cuda_err(e);
  });
}

// Launch a kernel that begins with start_after_previous(): its CTAs may become resident while
// the launch before drains, which hides the launch's own latency.
template <class... Params, class... Args>
int launch_overlapped(void (*kern)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                      const Args&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cuda_err(cudaLaunchKernelEx(&cfg, kern, args...));
}

// One step of grid h on the given buffers.
int launch_step_ptrs(const lbmice_t* h, const StepPtrs& P, cudaStream_t st) {
  if (h->C.stencil == 4 && h->C.fold == 6) {
    // the default scheme (E4, six-fold): the column march, its populations prefetched into
    // L2 by TMA when the step's buffers have tensor maps (16-bit storage)
    const dim3 grid = march_grid(h->C);
    return with_storage(h, [&](auto tag) {
      using S = decltype(tag);
      auto go = [&](auto flow, auto pref) {
        constexpr bool F = decltype(flow)::value;
        constexpr int M = decltype(pref)::value ? MARCH_PREFETCH : MARCH_PLAIN;
        return launch_overlapped(march_kernel<F, S, M>, grid, kMarchThreads, march_smem_bytes<F>(),
                                 st, h->C, P);
      };
      const bool pref = dev16(h) && P.tm != nullptr;
      if (h->p.flow)
        return pref ? go(std::true_type{}, std::true_type{}) : go(std::true_type{}, std::false_type{});
      return pref ? go(std::false_type{}, std::true_type{}) : go(std::false_type{}, std::false_type{});
    });
  }
  // every other stencil and fold: tiles of radius 2 (E6 and E8 reach two nodes out: phi halo 3)
  return with_storage(h, [&](auto tag) {
    using S = decltype(tag);
    if (h->tile_step) {
      using T = Tile<32, 8, 2>;
      const dim3 grd((h->C.nx + 31) / 32, (h->C.ny + 7) / 8);
      return h->p.flow ? launch_overlapped(tile_kernel<true, S>, grd, T::NT,
                                           T::template smem_bytes<true>(), st, h->C, P)
                       : launch_overlapped(tile_kernel<false, S>, grd, T::NT,
                                           T::template smem_bytes<false>(), st, h->C, P);
    }
    const auto go = [&](auto width) {
      constexpr int W = decltype(width)::value;
      using T = RowTile<W, 2>;
      const int rows = (h->C.ny + W - 3) / (W - 2), z = (rows + kMaxGridY - 1) / kMaxGridY;
      const dim3 grd(march_strips(h->C.nx), (rows + z - 1) / z, z);
      return h->p.flow ? launch_overlapped(row_kernel<W, true, S, 2>, grd, 32 * W,
                                           T::template smem_bytes<true>(), st, h->C, P)
                       : launch_overlapped(row_kernel<W, false, S, 2>, grd, 32 * W,
                                           T::template smem_bytes<false>(), st, h->C, P);
    };
    return go(std::integral_constant<int, 8>{});
  });
}

StepPtrs step_ptrs(const lbmice_t* h, Phase f, int steps);

// Whether launches of this grid take two steps (create gives those a fourth phi plane).
bool two_step(const lbmice_t* h) { return h->nphi == kMaxPhi; }

// Two steps of grid h in tiles of h->tile_warps warps. keep (default scheme): store step n + 1 at
// P.rmid, too.
int launch_tiles(const lbmice_t* h, const StepPtrs& P, bool keep, cudaStream_t st) {
  if (dev16(h))
    return with_storage(h, [&](auto tag) -> int {
      using S = decltype(tag);
      const auto go = [&](auto width) {
        constexpr int W = decltype(width)::value;
        const dim3 grid(two_strips(h->C.nx), two_tiles(h->C.ny, W));
        return h->p.flow
                   ? launch_overlapped(two_tile_kernel<true, W, false, TWO_DEFAULT, S>, grid, 32 * W,
                                       TileTwoSmem<true, W>::bytes(), st, h->C, P)
                   : launch_overlapped(two_tile_kernel<false, W, false, TWO_DEFAULT, S>, grid, 32 * W,
                                       TileTwoSmem<false, W>::bytes(), st, h->C, P);
      };
      if constexpr (!Storage<S>::DEV) return LBMICE_EINVAL;  // (not reached)
      else
        return h->tile_warps == 12 ? go(std::integral_constant<int, 12>{})
                                   : go(std::integral_constant<int, 16>{});
    });
  const auto go = [&](auto width, auto kept, auto var) {
    constexpr int W = decltype(width)::value, V = decltype(var)::value;
    constexpr bool K = decltype(kept)::value;
    const dim3 grid(two_strips(h->C.nx, V), two_tiles(h->C.ny, W, V));
    if constexpr (W <= kTileWide<true>) {
      if (h->p.flow)
        return launch_overlapped(two_tile_kernel<true, W, K, V>, grid, 32 * W,
                                 TileTwoSmem<true, W, V>::bytes(), st, h->C, P);
    }
    return launch_overlapped(two_tile_kernel<false, W, K, V>, grid, 32 * W,
                             TileTwoSmem<false, W, V>::bytes(), st, h->C, P);
  };
  const auto pick = [&](auto kept, auto var) {
    constexpr int V = decltype(var)::value;
    if constexpr (V == TWO_DEFAULT)
      if (h->tile_warps == 8) return go(std::integral_constant<int, 8>{}, kept, var);
    if (h->tile_warps == 12) return go(std::integral_constant<int, 12>{}, kept, var);
    if (h->tile_warps == kTileWide<false>)
      return go(std::integral_constant<int, kTileWide<false>>{}, kept, var);
    return go(std::integral_constant<int, 16>{}, kept, var);
  };
  const int v = two_variant(h->C);
  if (v == TWO_NEAR) return pick(std::false_type{}, std::integral_constant<int, TWO_NEAR>{});
  if (v == TWO_FAR) return pick(std::false_type{}, std::integral_constant<int, TWO_FAR>{});
  return keep ? pick(std::true_type{}, std::integral_constant<int, TWO_DEFAULT>{})
              : pick(std::false_type{}, std::integral_constant<int, TWO_DEFAULT>{});
}

// One launch of grid h from phase f: steps (1 or 2) time steps on its rotating buffers.
int launch_step(const lbmice_t* h, Phase f, int steps, cudaStream_t st) {
  const StepPtrs P = step_ptrs(h, f, steps);
  if (steps == 1) return launch_step_ptrs(h, P, st);
  if (h->tile_warps) return launch_tiles(h, P, false, st);
  const int v = two_variant(h->C);
  const dim3 grid(two_strips(h->C.nx, v), two_segments(h->C.ny, h->C.two_rows));
  const auto go = [&](auto var) {
    constexpr int V = decltype(var)::value, threads = kTwoRows * kTwoCols;
    return h->p.flow ? launch_overlapped(two_kernel<true, V>, grid, threads,
                                         TwoSmem<true, V>::bytes(), st, h->C, P)
                     : launch_overlapped(two_kernel<false, V>, grid, threads,
                                         TwoSmem<false, V>::bytes(), st, h->C, P);
  };
  return v == TWO_DEFAULT ? go(std::integral_constant<int, TWO_DEFAULT>{})
         : v == TWO_NEAR  ? go(std::integral_constant<int, TWO_NEAR>{})
                          : go(std::integral_constant<int, TWO_FAR>{});
}

// Whether a call of nsteps steps of a grid with four phi planes is to end with six that turn in
// place (Phase::turn). A call captured on its stream is bound to the buffers it was captured with,
// and its graph may be launched again if it leaves them as it found them: pairs do after multiples
// of four steps, single steps in four planes after multiples of twelve, so a captured call of an odd
// number of half dozens takes its last six this way.
constexpr int kTurnSteps = 6;
bool ends_in_turn(int64_t nsteps, cudaStream_t st) {
  if (nsteps % (2 * kTurnSteps) != kTurnSteps) return false;
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &status) != cudaSuccess) {
    cudaGetLastError();  // the legacy stream beside another stream's capture: not captured itself
    return false;
  }
  return status == cudaStreamCaptureStatusActive;
}

// Steps of the next launch when left are to be taken.
int launch_steps(const lbmice_t* h, int64_t left) { return two_step(h) && left >= 2 ? 2 : 1; }

// The graph of kGraphSteps steps from the grid's buffer phase, captured when first needed.
int ensure_graph(lbmice_t* h, cudaGraphExec_t* out) {
  Phase f = phase_of(h);
  cudaGraphExec_t& slot = h->graph[phase_index(h, f)];
  if (!slot) {
    cudaGraph_t g = nullptr;
    LB_TRY(cudaStreamBeginCapture(h->capture, cudaStreamCaptureModeThreadLocal));
    int rc = LBMICE_OK;
    for (int64_t left = kGraphSteps; left > 0 && rc == LBMICE_OK;) {
      const int n = launch_steps(h, left);
      rc = launch_step(h, f, n, h->capture);
      f.advance(n);
      left -= n;
    }
    cudaError_t e = cudaStreamEndCapture(h->capture, &g);
    if (rc != LBMICE_OK) { if (g) cudaGraphDestroy(g); return rc; }
    if (e != cudaSuccess) return cuda_err(e);
    e = cudaGraphInstantiate(&slot, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) { slot = nullptr; return cuda_err(e); }
  }
  *out = slot;
  return LBMICE_OK;
}

// The pinned block of a grid's host results, allocated with the grid: queries allocate nothing.
// The driver carves small blocks out of a chunk that it maps for the first of them and unmaps with
// the last (105 + 155 us); one of 64 bytes, held until the process ends, keeps the chunk (2 + 2 us
// for every grid after the first).
cudaError_t allocate_results(lbmice_t* h) {
  static std::once_flag once;
  std::call_once(once, [] {
    void* chunk = nullptr;
    if (cudaMallocHost(&chunk, 64) != cudaSuccess) cudaGetLastError();  // only the time is lost
  });
  void* p = nullptr;
  const cudaError_t e = cudaMallocHost(&p, sizeof(double) * (8 + 3 * LBMICE_MAX_RAYS));
  if (e != cudaSuccess) return e;
  h->stat_host = static_cast<double*>(p);
  h->tip_host = h->stat_host + 8;
  return e;
}

int run_stats(lbmice_t* h) {
  const int s = h->cur;
  int rc = with_storage(h, [&](auto tag) {
    using S = decltype(tag);
    stats_partial_kernel<S><<<kStatBlocks, kStatThreads, 0, h->stream>>>(
        h->C, h->p.flow, 0.5 * h->p.dx * h->p.dx, 0.5 * h->p.L_sat, h->pops[s], phi_now(h),
        phi_prev(h), h->Um[s], h->rhom[s], h->stat_partial);
    return cuda_err(cudaGetLastError());
  });
  if (rc != LBMICE_OK) return rc;
  // the sums and the word of the bounded device-side waits (lbmice_tma.cuh) that gave up
  // since the last check, written straight to pinned host memory
  stats_final_kernel<<<1, kStatFinalThreads, 0, h->stream>>>(h->stat_partial, kStatBlocks,
                                                             h->stat_host, 1);
  LB_TRY(cudaGetLastError());
  LB_TRY(cudaStreamSynchronize(h->stream));
  return h->stat_host[kNStat] != 0.0 ? LBMICE_ETIMEOUT : LBMICE_OK;
}

// Zero the padding columns of the free population buffer after it served as staging space, so
// that the padding of every state is zero whichever buffer it ends up in (a grid that steps in
// pairs or singly does not keep to the step's parity).
int clear_staging(lbmice_t* h) {
  // 16-bit buffers have unused parts beside the padding
  if (dev16(h))
    return two_step(h) ? cuda_err(cudaMemsetAsync(h->pops[1 - h->cur], 0, pop_bytes(h), h->stream))
                       : LBMICE_OK;
  if (h->C.pitch == h->C.nx) return LBMICE_OK;
  const int n = (h->C.pitch - h->C.nx) * h->C.ny;
  clear_padding_kernel<<<(n + 255) / 256, 256, 0, h->stream>>>(
      h->C, h->p.flow, static_cast<float*>(h->pops[1 - h->cur]));
  return cuda_err(cudaGetLastError());
}

int equilibrium_from(lbmice_t* h, const double* phi, const double* U, const double* rho,
                     const double* ux, const double* uy) {
  if (!h->p.flow) ux = uy = rho = nullptr;  // fluid at rest: g^eq sees u = 0
  const dim3 blk(32, 8);
  const dim3 grd = node_grid(h->C, blk);
  const double eps = h->p.eps, kNkeps = h->p.kappa_N * h->C.fold * h->p.eps;
  int rc = with_storage(h, [&](auto tag) {
    using S = decltype(tag);
    if (h->p.flow)
      equilibrium_kernel<true, S><<<grd, blk, 0, h->stream>>>(
          h->C, h->Dphi3, eps, kNkeps, phi, U, rho, ux, uy, h->pops[0], h->phi[0], h->phi[h->nphi - 1],
          h->Um[0], h->rhom[0]);
    else
      equilibrium_kernel<false, S><<<grd, blk, 0, h->stream>>>(
          h->C, h->Dphi3, eps, kNkeps, phi, U, rho, ux, uy, h->pops[0], h->phi[0], h->phi[h->nphi - 1],
          h->Um[0], h->rhom[0]);
    return cuda_err(cudaGetLastError());
  });
  if (rc != LBMICE_OK) return rc;
  h->step = 0;
  h->ring = 0;
  h->cur = 0;
  return LBMICE_OK;
}

// member: the grid steps with others in a batch, in pairs whatever its shape.
int create_grid(const lbmice_params* p, void* stream, bool member, lbmice_t** out) {
  if (!out) return LBMICE_EINVAL;
  *out = nullptr;
  if (!p) return LBMICE_EINVAL;
  int rc = validate(*p);
  if (rc != LBMICE_OK) return rc;
  lbmice_t* h = new (std::nothrow) lbmice_ctx();
  if (!h) return LBMICE_ENOMEM;
  h->p = *p;
  derive(h);
  h->stream = static_cast<cudaStream_t>(stream);
  h->nplanes = p->flow ? 27 : 18;
  h->elem = p->storage == LBMICE_STORAGE_F32 ? 4 : 2;
  cudaError_t e = cudaGetDevice(&h->device);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&h->capture, cudaStreamNonBlocking);
  const auto allocate = [&](int nphi) {
    const size_t phi_bytes = field_bytes(h);
    Slab s;
    for (void*& b : h->pops) s.place(&b, pop_bytes(h));
    for (int i = 0; i < nphi; ++i) s.place(&h->phi[i], phi_bytes);
    if (dev16(h)) {
      for (float*& b : h->Um) s.place(&b, phi_bytes);
      if (p->flow)
        for (float*& b : h->rhom) s.place(&b, phi_bytes);
    }
    const size_t zeroed = s.bytes();
    s.place(&h->stat_partial, sizeof(double) * kStatBlocks * kNStat);
    s.place(&h->tmaps, sizeof(CUtensorMap) * kMaxPhases * kMapsPerPhase);
    const cudaError_t ea = s.allocate(&h->slab);
    if (ea != cudaSuccess) return ea;
    h->nphi = nphi;
    return cudaMemsetAsync(h->slab, 0, zeroed, h->stream);
  };
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device) != cudaSuccess ||
      sms < 1)
    sms = 1;
  // steps in pairs need a fourth phi plane; a grid so large that this plane does not fit any more
  // takes them one by one
  const bool pairs = two_possible(h->p, h->C) &&
                     (member || !too_narrow_for_pairs(h->C, p->flow != 0, dev16(h), sms));
  if (e == cudaSuccess) e = allocate(pairs ? kMaxPhi : 3);
  if (e == cudaErrorMemoryAllocation && pairs) {
    cudaGetLastError();
    e = allocate(3);
  }
  if (e == cudaSuccess) e = allocate_results(h);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) {
    release(h);
    cudaGetLastError();  // clear a sticky-free error state left by a failed allocation
    return cuda_err(e);
  }
  h->C.seg_rows = march_seg_rows(h->C.nx, h->C.ny, sms);
  h->C.two_rows = two_seg_rows(h->C.nx, h->C.ny, two_variant(h->C),
                               two_ctas(p->flow != 0) * sms);
  h->tile_step = one_step_tiles(h->C, sms);
  h->tile_warps = two_tile_warps(h->C, p->flow != 0, dev16(h), sms);
  rc = march_attributes(h);
  if (rc == LBMICE_OK) rc = make_tensor_maps(h);
  if (rc != LBMICE_OK) {
    release(h);
    cudaGetLastError();
    return rc;
  }
  *out = h;
  return LBMICE_OK;
}

}  // namespace

extern "C" {

int lbmice_params_default(lbmice_params* p, int32_t nx, int32_t ny) {
  if (!p) return LBMICE_EINVAL;
  std::memset(p, 0, sizeof(*p));
  p->nx = nx;
  p->ny = ny;
  p->dx = 0.4;
  p->dt = 0.008;
  p->W0 = 1.0;
  p->tau0 = 1.0;
  p->D = 2.0;
  p->lambda = 0.0;
  p->L_sat = 1.0;
  p->eps = 0.05;
  p->kappa_N = 1.0;
  p->nu = 0.016;
  for (int f = 0; f < 4; ++f) p->bc[f] = LBMICE_BC_PERIODIC;
  p->stencil = 4;
  p->fold = 6;
  return LBMICE_OK;
}

int lbmice_create(const lbmice_params* p, void* stream, lbmice_t** out) {
  return create_grid(p, stream, false, out);
}

int lbmice_init_seed(lbmice_t* h, double cx, double cy, double R0, double U0) {
  if (!h || !std::isfinite(cx) || !std::isfinite(cy) || !std::isfinite(R0) ||
      !std::isfinite(U0))
    return LBMICE_EINVAL;
  // The second population buffer is free before the first step: it holds the double seed
  // fields (phi and U, plus rho and u with flow: 16 or 40 bytes per node; it has at least 36
  // or 54).
  const size_t n = (size_t)h->p.nx * h->p.ny;
  double* f = reinterpret_cast<double*>(h->pops[1]);
  const bool fl = h->p.flow != 0;
  // velocity of the first inlet face along its inward normal (the fluid rests otherwise)
  double ux = 0.0, uy = 0.0;
  const double nxs[4] = {1, -1, 0, 0}, nys[4] = {0, 0, 1, -1};
  for (int face = 0; face < 4; ++face)
    if (h->p.flow && h->p.bc[face] == LBMICE_BC_INLET) {
      ux = h->p.u_in * nxs[face];
      uy = h->p.u_in * nys[face];
      break;
    }
  const dim3 blk(32, 8);
  const dim3 grd = node_grid(h->C, blk);
  double* rho = fl ? f + 2 * n : nullptr;
  double* uxf = fl ? f + 3 * n : nullptr;
  double* uyf = fl ? f + 4 * n : nullptr;
  seed_kernel<<<grd, blk, 0, h->stream>>>(h->p.nx, h->p.ny, cx, cy, R0, U0,
                                          std::sqrt(2.0) * h->p.W0 / h->p.dx, ux, uy, f,
                                          f + n, rho, uxf, uyf);
  LB_TRY(cudaGetLastError());
  const int rc = equilibrium_from(h, f, f + n, rho, uxf, uyf);
  return rc != LBMICE_OK ? rc : clear_staging(h);
}

int lbmice_set_fields(lbmice_t* h, const double* phi, const double* U, const double* rho,
                      const double* ux, const double* uy, int32_t on_device) {
  if (!h || !phi || !U || (on_device != 0 && on_device != 1)) return LBMICE_EINVAL;
  if (on_device) return equilibrium_from(h, phi, U, rho, ux, uy);
  const size_t n = (size_t)h->p.nx * h->p.ny;
  double* f = reinterpret_cast<double*>(h->pops[1]);
  const bool fl = h->p.flow != 0;  // without flow the velocity inputs are ignored
  const double* src[5] = {phi, U, fl ? rho : nullptr, fl ? ux : nullptr, fl ? uy : nullptr};
  const double* dev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
  for (int k = 0; k < 5; ++k) {
    if (!src[k]) continue;
    LB_TRY(cudaMemcpyAsync(f + k * n, src[k], n * sizeof(double), cudaMemcpyHostToDevice,
                           h->stream));
    dev[k] = f + k * n;
  }
  int rc = equilibrium_from(h, dev[0], dev[1], dev[2], dev[3], dev[4]);
  if (rc == LBMICE_OK) rc = clear_staging(h);
  if (rc != LBMICE_OK) return rc;
  // pageable sources may be reused by the caller once this returns
  LB_TRY(cudaStreamSynchronize(h->stream));
  return LBMICE_OK;
}

int lbmice_step(lbmice_t* h, int64_t nsteps) {
  if (!h || nsteps < 0) return LBMICE_EINVAL;
  const int64_t every = h->p.check_every;
  const bool turn = two_step(h) && every == 0 && ends_in_turn(nsteps, h->stream);
  int64_t left = turn ? nsteps - kTurnSteps : nsteps;
  while (left > 0) {
    int64_t chunk = left;
    if (every > 0) chunk = std::min<int64_t>(left, every - (h->step % every));
    int64_t done = 0;
    while (done < chunk) {
      if (chunk - done >= kGraphSteps && h->taken >= kGraphAfter) {
        cudaGraphExec_t g = nullptr;
        int rc = ensure_graph(h, &g);
        if (rc != LBMICE_OK) return rc;
        LB_TRY(cudaGraphLaunch(g, h->stream));
        h->step += kGraphSteps;
        h->ring += kGraphSteps;
        done += kGraphSteps;
      } else {
        const int n = launch_steps(h, chunk - done);
        int rc = launch_step(h, phase_of(h), n, h->stream);
        if (rc != LBMICE_OK) return rc;
        h->cur ^= 1;
        h->step += n;
        h->ring += n;
        h->taken += n;
        done += n;
      }
    }
    left -= chunk;
    if (every > 0 && h->step % every == 0) {
      int rc = run_stats(h);
      if (rc != LBMICE_OK) return rc;
      if (h->stat_host[4] != 0.0) return LBMICE_ENONFINITE;
    }
  }
  if (turn) {
    Phase f = phase_of(h);
    for (f.turn = 0; f.turn >= 0; f.advance(1)) {
      const int rc = launch_step(h, f, 1, h->stream);
      if (rc != LBMICE_OK) return rc;
    }
    h->step += kTurnSteps;
    h->taken += kTurnSteps;
  }
  return LBMICE_OK;
}

}  // extern "C"

namespace {

// The pieces of the exact state, in blob order: populations, phi^n, phi^{n-1}, and with
// 16-bit storage U and rho of the current slot.
struct StatePart {
  void* ptr;
  size_t bytes;
};
int state_parts(lbmice_t* h, StatePart parts[5]) {
  int n = 0;
  parts[n++] = {h->pops[h->cur], pop_bytes(h)};
  parts[n++] = {phi_now(h), field_bytes(h)};
  parts[n++] = {phi_prev(h), field_bytes(h)};
  if (h->Um[0]) parts[n++] = {h->Um[h->cur], field_bytes(h)};
  if (h->rhom[0]) parts[n++] = {h->rhom[h->cur], field_bytes(h)};
  return n;
}

}  // namespace

extern "C" size_t lbmice_state_bytes(const lbmice_t* h) {
  if (!h) return 0;
  StatePart parts[5];
  const int n = state_parts(const_cast<lbmice_t*>(h), parts);
  size_t total = 0;
  for (int k = 0; k < n; ++k) total += parts[k].bytes;
  return total;
}

namespace {

// Zero the padding columns of the phi planes before they are shown in a state, if a field on its way
// to the host ran over them. (Zeroed after each such field instead, they cost it 8 us: 24 -> 33 us
// for a field of 500^2.)
int clear_plane_padding(lbmice_t* h) {
  if (!h->pad_used) return LBMICE_OK;
  const size_t pitch = sizeof(float) * h->C.pitch, pad = pitch - sizeof(float) * h->C.nx;
  for (int i = 0; i < h->nphi; ++i)
    LB_TRY(cudaMemset2DAsync(h->phi[i] + h->C.nx, pitch, 0, pad, h->C.ny, h->stream));
  h->pad_used = false;
  return LBMICE_OK;
}

int copy_state(lbmice_t* h, void* blob, bool out, cudaMemcpyKind kind) {
  StatePart parts[5];
  const int n = state_parts(h, parts);
  char* b = static_cast<char*>(blob);
  for (int k = 0; k < n; ++k) {
    if (out)
      LB_TRY(cudaMemcpyAsync(b, parts[k].ptr, parts[k].bytes, kind, h->stream));
    else
      LB_TRY(cudaMemcpyAsync(parts[k].ptr, b, parts[k].bytes, kind, h->stream));
    b += parts[k].bytes;
  }
  return LBMICE_OK;
}

}  // namespace

extern "C" int lbmice_fields(lbmice_t* h, int32_t which, void* dst, size_t bytes,
                             int32_t dst_on_device) {
  if (!h || !dst || which < 0 || which > LBMICE_FIELD_STATE ||
      (dst_on_device != 0 && dst_on_device != 1))
    return LBMICE_EINVAL;
  const int s = h->cur;
  const size_t nx = h->p.nx, ny = h->p.ny;
  const cudaMemcpyKind kind = dst_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  const dim3 blk(32, 8);
  float* scratch = free_plane(h);
  if (which != LBMICE_FIELD_STATE && !dst_on_device && h->C.pitch != h->C.nx) h->pad_used = true;
  if (which == LBMICE_FIELD_STATE) {
    if (bytes < lbmice_state_bytes(h)) return LBMICE_EINVAL;
    int rc = clear_plane_padding(h);
    if (rc == LBMICE_OK) rc = copy_state(h, dst, true, kind);
    if (rc != LBMICE_OK) return rc;
  } else if (which == LBMICE_FIELD_POPS) {
    const size_t need = sizeof(float) * h->nplanes * nx * ny;
    if (bytes < need) return LBMICE_EINVAL;
    // decode one plane at a time (into dst directly, or through the field buffer)
    for (int q = 0; q < h->nplanes; ++q) {
      float* out = dst_on_device ? static_cast<float*>(dst) + (size_t)q * nx * ny : scratch;
      int rc = with_storage(h, [&](auto tag) {
        using S = decltype(tag);
        decode_plane_kernel<S><<<node_grid(h->C, blk), blk, 0, h->stream>>>(
            h->C, h->pops[s], q / 9, q % 9, phi_now(h), h->Um[s], h->rhom[s],
            out);
        return cuda_err(cudaGetLastError());
      });
      if (rc != LBMICE_OK) return rc;
      if (!dst_on_device)
        LB_TRY(cudaMemcpyAsync(static_cast<float*>(dst) + (size_t)q * nx * ny, scratch,
                               sizeof(float) * nx * ny, cudaMemcpyDeviceToHost, h->stream));
    }
  } else {
    const size_t need = sizeof(float) * nx * ny;
    if (bytes < need) return LBMICE_EINVAL;
    float* out = dst_on_device ? static_cast<float*>(dst) : scratch;
    int rc = with_storage(h, [&](auto tag) {
      using S = decltype(tag);
      moment_kernel<S><<<node_grid(h->C, blk), blk, 0, h->stream>>>(
          h->C, which, h->p.flow, h->pops[s], phi_now(h), phi_prev(h), h->Um[s], h->rhom[s], out);
      return cuda_err(cudaGetLastError());
    });
    if (rc != LBMICE_OK) return rc;
    if (!dst_on_device)
      LB_TRY(cudaMemcpyAsync(dst, scratch, need, cudaMemcpyDeviceToHost, h->stream));
  }
  if (!dst_on_device) LB_TRY(cudaStreamSynchronize(h->stream));
  return LBMICE_OK;
}

extern "C" int lbmice_load(lbmice_t* h, int32_t which, const void* src, size_t bytes,
                           int32_t src_on_device) {
  if (!h || !src || (src_on_device != 0 && src_on_device != 1)) return LBMICE_EINVAL;
  if (which != LBMICE_FIELD_POPS && which != LBMICE_FIELD_PHI_PREV &&
      which != LBMICE_FIELD_STATE)
    return LBMICE_EINVAL;
  const int s = h->cur;
  const size_t nx = h->p.nx, ny = h->p.ny;
  const cudaMemcpyKind kind = src_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  const dim3 blk(32, 8);
  if (which == LBMICE_FIELD_STATE) {
    if (bytes < lbmice_state_bytes(h)) return LBMICE_EINVAL;
    int rc = copy_state(h, const_cast<void*>(src), false, kind);
    if (rc != LBMICE_OK) return rc;
  } else if (which == LBMICE_FIELD_POPS) {
    if (bytes < sizeof(float) * h->nplanes * nx * ny) return LBMICE_EINVAL;
    // stage the 9 float planes of each lattice in the free population buffer (it holds at
    // least 9 nx ny floats), then encode them into the current one; the h lattice's moment
    // is the phi^n plane, and with 16-bit storage U and rho are kept too
    float* stage = static_cast<float*>(h->pops[1 - s]);
    for (int L = 0; L < h->nplanes / 9; ++L) {
      LB_TRY(cudaMemcpyAsync(stage, static_cast<const float*>(src) + (size_t)9 * L * nx * ny,
                             sizeof(float) * 9 * nx * ny, kind, h->stream));
      float* M = L == 0 ? phi_now(h) : L == 1 ? h->Um[s] : h->rhom[s];
      int rc = with_storage(h, [&](auto tag) {
        using S = decltype(tag);
        encode_lattice_kernel<S><<<node_grid(h->C, blk), blk, 0, h->stream>>>(
            h->C, stage, L, h->pops[s], M);
        return cuda_err(cudaGetLastError());
      });
      if (rc != LBMICE_OK) return rc;
    }
    const int rc = clear_staging(h);
    if (rc != LBMICE_OK) return rc;
  } else {
    if (bytes < sizeof(float) * nx * ny) return LBMICE_EINVAL;
    LB_TRY(cudaMemcpy2DAsync(phi_prev(h), h->C.pitch * sizeof(float), src,
                             nx * sizeof(float), nx * sizeof(float), ny, kind, h->stream));
  }
  if (!src_on_device) LB_TRY(cudaStreamSynchronize(h->stream));
  return LBMICE_OK;
}

extern "C" {

int lbmice_stats(lbmice_t* h, double out[LBMICE_NSTATS]) {
  if (!h || !out) return LBMICE_EINVAL;
  int rc = run_stats(h);
  if (rc != LBMICE_OK) return rc;
  for (int k = 0; k < kNStat; ++k) out[k] = h->stat_host[k];
  out[5] = (double)h->step;
  return LBMICE_OK;
}

int lbmice_tips(lbmice_t* h, double cx, double cy, double step, int32_t nrays,
                const double* angles_deg, double* radii) {
  if (!h || !angles_deg || !radii || nrays < 1 || nrays > LBMICE_MAX_RAYS ||
      !(step > 0.0) || !std::isfinite(step) || !std::isfinite(cx) || !std::isfinite(cy))
    return LBMICE_EINVAL;
  const double deg = 3.14159265358979323846 / 180.0;
  for (int i = 0; i < nrays; ++i) {
    if (!std::isfinite(angles_deg[i])) return LBMICE_EINVAL;
    h->tip_host[2 * i] = std::cos(angles_deg[i] * deg);
    h->tip_host[2 * i + 1] = std::sin(angles_deg[i] * deg);
  }
  // a few numbers each way: the kernel reads and writes the pinned host buffer itself
  tips_kernel<<<nrays, kTipThreads, 0, h->stream>>>(phi_now(h), h->C.nx, h->C.ny, h->C.pitch, cx, cy,
                                                    step, h->tip_host,
                                                    h->tip_host + 2 * LBMICE_MAX_RAYS);
  LB_TRY(cudaGetLastError());
  LB_TRY(cudaStreamSynchronize(h->stream));
  for (int i = 0; i < nrays; ++i) radii[i] = h->tip_host[2 * LBMICE_MAX_RAYS + i];
  return LBMICE_OK;
}

int lbmice_sync(lbmice_t* h) {
  if (!h) return LBMICE_EINVAL;
  LB_TRY(cudaStreamSynchronize(h->stream));
  LB_TRY(cudaGetLastError());
  return LBMICE_OK;
}

int64_t lbmice_steps_done(const lbmice_t* h) { return h ? h->step : -1; }

int lbmice_destroy(lbmice_t* h) {
  if (!h) return LBMICE_OK;
  cudaError_t e = cudaStreamSynchronize(h->stream);
  release(h);
  return cuda_err(e);
}

const char* lbmice_last_error(void) { return g_last_cuda_error; }

const char* lbmice_strerror(int code) {
  switch (code) {
    case LBMICE_OK: return "ok";
    case LBMICE_EINVAL: return "invalid argument";
    case LBMICE_ECUDA: return "CUDA error";
    case LBMICE_ENOMEM: return "out of memory";
    case LBMICE_ENONFINITE: return "non-finite value in phi, U or rho";
    case LBMICE_EUNSTABLE: return "unstable parameters (relaxation time or inflow speed)";
    case LBMICE_ETIMEOUT: return "device-side wait timed out";
    case LBMICE_ENOTSUP: return "not supported by this build";
    default: return "unknown error";
  }
}

int lbmice_debug_flags(uint32_t* flags, int32_t clear) {
  if (!flags || (clear != 0 && clear != 1)) return LBMICE_EINVAL;
  *flags = 0;
#ifdef LBMICE_CHECKED
  LB_TRY(cudaDeviceSynchronize());  // every queued step, on any stream, has run
  unsigned w = 0;
  LB_TRY(cudaMemcpyFromSymbol(&w, lbmice::oob_word, sizeof(w)));
  *flags = w;
  if (clear) {
    const unsigned z = 0;
    LB_TRY(cudaMemcpyToSymbol(lbmice::oob_word, &z, sizeof(z)));
  }
  return LBMICE_OK;
#else
  return LBMICE_ENOTSUP;
#endif
}

int lbmice_debug_wait_selftest(void) {
  unsigned int w = 0;
  const unsigned int z = 0;
  LB_TRY(cudaDeviceSynchronize());
  LB_TRY(cudaMemcpyToSymbol(lbmice::wait_word, &z, sizeof(z)));
  lbmice::wait_selftest_kernel<<<1, 32>>>();
  LB_TRY(cudaGetLastError());
  LB_TRY(cudaDeviceSynchronize());
  LB_TRY(cudaMemcpyFromSymbol(&w, lbmice::wait_word, sizeof(w)));
  LB_TRY(cudaMemcpyToSymbol(lbmice::wait_word, &z, sizeof(z)));
  return w ? LBMICE_ETIMEOUT : LBMICE_OK;
}

int lbmice_debug_set_margin(int64_t margin) {
  if (margin < 0) return LBMICE_EINVAL;
#ifdef LBMICE_CHECKED
  LB_TRY(cudaDeviceSynchronize());
  const long long m = margin;
  LB_TRY(cudaMemcpyToSymbol(lbmice::oob_margin, &m, sizeof(m)));
  return LBMICE_OK;
#else
  return LBMICE_ENOTSUP;
#endif
}

}  // extern "C"

// ---------------------------------------------------------------------------------------
// FP64 diagnostics without allocation (declared in include/lbmice.h as lbmice_stats_noalloc).
//
// Some callers cannot allocate device memory at the moment they want these diagnostics:
// a host application whose device memory is reserved up front by its own pool allocator
// (so a cudaMalloc from this library would fail or fragment that budget), or a
// time-critical loop for which the implicit device synchronisation and unbounded latency of
// cudaMalloc/cudaFree are not acceptable. For them the per-block partial sums of the
// reduction live in the fixed array below, which every GPU that loads this library holds
// until the process exits.
// ---------------------------------------------------------------------------------------
namespace {

constexpr int kNoallocMaxBlocks = 2048;                  // partial rows in the fixed array
constexpr long long kNoallocNodesPerBlock = 8192;        // nodes summed by one block
constexpr int kNoallocMaxDevices = 64;
static_assert(kNoallocMaxBlocks * kNoallocNodesPerBlock == LBMICE_NOALLOC_MAX_NODES,
              "the fixed partial array must cover LBMICE_NOALLOC_MAX_NODES nodes");

// 2048 rows x 5 doubles = 80 KB. Every row a call reads is written by that same call before
// it is read, so nothing has to start at zero; the array keeps the last call's partials.
static __device__ __align__(256) double g_noalloc_partial[kNoallocMaxBlocks * kNStat];

std::atomic<double*> g_noalloc_ptr[kNoallocMaxDevices];

// Device address of the fixed array on the current device. Host code only holds a host-side
// stand-in for the symbol, so the address is asked for once per device, with that device
// current, and cached for the life of the process (valid while the device's primary context
// lives: a cudaDeviceReset makes it stale, as the header states).
int noalloc_scratch(double** out) {
  int dev = 0;
  LB_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kNoallocMaxDevices) return LBMICE_EINVAL;
  double* p = g_noalloc_ptr[dev].load(std::memory_order_acquire);
  if (!p) {
    void* q = nullptr;
    LB_TRY(cudaGetSymbolAddress(&q, g_noalloc_partial));
    p = static_cast<double*>(q);
    g_noalloc_ptr[dev].store(p, std::memory_order_release);
  }
  *out = p;
  return LBMICE_OK;
}

}  // namespace

extern "C" int lbmice_stats_noalloc(const float* pops, const float* phi, const float* phi_prev,
                                    int32_t nx, int32_t ny, int32_t pitch, int32_t flow,
                                    double dx, double L_sat, double* out, void* stream) {
  if (!pops || !phi || !phi_prev || !out || nx < 1 || ny < 1 || pitch < nx ||
      (flow != 0 && flow != 1) || !(dx > 0) || !std::isfinite(L_sat))
    return LBMICE_EINVAL;
  const long long nodes = (long long)nx * ny;
  if (nodes > LBMICE_NOALLOC_MAX_NODES) return LBMICE_EINVAL;  // beyond the fixed array
  const int nblocks = (int)((nodes + kNoallocNodesPerBlock - 1) / kNoallocNodesPerBlock);
  double* partial = nullptr;
  int rc = noalloc_scratch(&partial);
  if (rc != LBMICE_OK) return rc;
  Consts C;
  std::memset(&C, 0, sizeof(C));
  C.nx = nx;
  C.ny = ny;
  C.pitch = pitch;
  C.pstride = (long long)pitch * ny;  // caller's layout: [plane][ny][pitch]
  C.rstride = pitch;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  stats_partial_kernel<F32P><<<nblocks, kStatThreads, 0, st>>>(
      C, flow, 0.5 * dx * dx, 0.5 * L_sat, pops, phi, phi_prev, nullptr, nullptr, partial);
  LB_TRY(cudaGetLastError());
  stats_final_kernel<<<1, kStatFinalThreads, 0, st>>>(partial, nblocks, out, 0);
  LB_TRY(cudaGetLastError());
  return LBMICE_OK;
}

// ---------------------------------------------------------------------------------------
// Batches: many member grids advanced by one launch per tile shape and step.
// ---------------------------------------------------------------------------------------
struct lbmice_batch {
  std::vector<lbmice_t*> members;
  std::vector<int> shape;             // tile shape id of each member
  cudaStream_t stream = nullptr;
  cudaStream_t capture = nullptr;     // private stream used only to record graphs
  int flow = 0, storage = 0;
  std::unique_ptr<BatchLaunch> block; // host scratch for one launch's parameter block
  bool two = false;                   // members of the march shape take their steps in pairs
  // graphs of kGraphSteps steps, each with the buffer phase of every member that it starts from
  struct Graph {
    std::vector<int> from;
    cudaGraphExec_t exec;
  };
  std::vector<Graph> graphs;
};

namespace {

// The batch has no step counter of its own: its members step together, and their common
// count (which re-initialising every member resets) decides the buffer phase.
int64_t batch_steps(const lbmice_batch_t* b) { return b->members[0]->step; }

// What a batched launch computes: single steps in one of the shapes, or two steps of members of the
// march shape, in tiles or by the two-step march.
enum : int { FORM_TWO_TILE = kNumShapes, FORM_TWO_MARCH };

// Work units of a member in a launch of this form: tiles, or (strip, segment) pairs of a march.
long long member_units(const lbmice_t* m, int form) {
  if (form == LBMICE_SHAPE_MARCH) return march_units(m->C, kMarchMaxSegRows);
  if (form >= kNumShapes)
    return (long long)two_strips(m->C.nx) * (form == FORM_TWO_TILE
                                                 ? two_tiles(m->C.ny, kBatchTileWarps)
                                                 : two_segments(m->C.ny, kBatchTwoRows));
  const int tx = shape_tx(form), ty = shape_ty(form);
  return (long long)((m->C.nx + tx - 1) / tx) * ((m->C.ny + ty - 1) / ty);
}

// The region bases of a step's population buffers (StepPtrs::rin, rout): element offsets
// 4pQ (p = 0..3), 16Q, 18Q, 22Q, 26Q of an FP32 buffer, 9LQ (L = 0, 1, 2) of a 16-bit one.
void step_regions(StepPtrs& P, const Consts& C, bool dev16) {
  const long long Q = C.pstride;
  const long long f32_off[kRegions] = {0, 4 * Q, 8 * Q, 12 * Q, 16 * Q, 18 * Q, 22 * Q, 26 * Q};
  std::memset(P.rmid, 0, sizeof(P.rmid));
  for (int r = 0; r < kRegions; ++r) {
    const long long bytes = dev16 ? (r < 3 ? 2 * 9 * r * Q : 0) : 4 * f32_off[r];
    const bool used = dev16 ? r < 3 : true;
    P.rin[r] = used ? static_cast<const char*>(P.pin) + bytes : nullptr;
    P.rout[r] = used ? static_cast<char*>(P.pout) + bytes : nullptr;
  }
}

// Buffer roles of a launch of steps (1 or 2) time steps from phase f.
StepPtrs step_ptrs(const lbmice_t* h, Phase f, int steps) {
  const int n = h->nphi;
  int now = (int)(f.s % n), before = (now + n - 1) % n, out = (now + steps) % n;
  if (f.turn >= 0) {
    const int three[3] = {before, now, (now + 1) % n};
    f.cur ^= f.turn & 1;
    before = three[f.turn % 3];
    now = three[(f.turn + 1) % 3];
    out = three[(f.turn + 2) % 3];
  }
  StepPtrs P;
  P.pin = h->pops[f.cur];
  P.pout = h->pops[1 - f.cur];
  P.phi_n = h->phi[now];
  P.phi_nm1 = h->phi[before];
  P.phi_np1 = h->phi[out];
  P.phi_mid = steps == 2 ? h->phi[(now + 1) % n] : nullptr;
  P.U_n = h->Um[f.cur];
  P.U_np1 = h->Um[1 - f.cur];
  P.rho_n = h->rhom[f.cur];
  P.rho_np1 = h->rhom[1 - f.cur];
  P.tm = h->tmaps ? h->tmaps + kMapsPerPhase * (f.cur * n + now) : nullptr;
  step_regions(P, h->C, dev16(h));
  return P;
}

template <int TX, int TY>
int launch_block(const lbmice_batch_t* b, long long tiles, cudaStream_t st) {
  return with_storage(b->members[0], [&](auto tag) {
    using S = decltype(tag);
    using T = Tile<TX, TY>;
    return b->flow ? launch_overlapped(batch_step_kernel<TX, TY, true, S>, dim3((unsigned)tiles), TX * TY,
                                       T::template smem_bytes<true>(), st, *b->block)
                   : launch_overlapped(batch_step_kernel<TX, TY, false, S>, dim3((unsigned)tiles), TX * TY,
                                       T::template smem_bytes<false>(), st, *b->block);
  });
}

int launch_march_block(const lbmice_batch_t* b, long long units, cudaStream_t st) {
  return with_storage(b->members[0], [&](auto tag) {
    using S = decltype(tag);
    // members with tensor maps (16-bit storage) prefetch, as their single-grid steps do
    constexpr int M = Storage<S>::DEV ? MARCH_PREFETCH : MARCH_PLAIN;
    const dim3 grid((unsigned)units);
    return b->flow ? launch_overlapped(batch_march_kernel<true, S, M>, grid, kMarchThreads,
                                       march_smem_bytes<true>(), st, *b->block)
                   : launch_overlapped(batch_march_kernel<false, S, M>, grid, kMarchThreads,
                                       march_smem_bytes<false>(), st, *b->block);
  });
}

int launch_two_block(const lbmice_batch_t* b, int form, long long units, cudaStream_t st) {
  constexpr int threads = kTwoRows * kTwoCols, W = kBatchTileWarps;
  const dim3 grid((unsigned)units);
  if (form == FORM_TWO_TILE)
    return b->flow ? launch_overlapped(batch_two_tile_kernel<true, W>, grid, 32 * W,
                                       TileTwoSmem<true, W>::bytes(), st, *b->block)
                   : launch_overlapped(batch_two_tile_kernel<false, W>, grid, 32 * W,
                                       TileTwoSmem<false, W>::bytes(), st, *b->block);
  return b->flow ? launch_overlapped(batch_two_kernel<true>, grid, threads, TwoSmem<true>::bytes(), st,
                                     *b->block)
                 : launch_overlapped(batch_two_kernel<false>, grid, threads, TwoSmem<false>::bytes(), st,
                                     *b->block);
}

// The form of a launch of steps (1, or 2 with the march shape) time steps of members of shape s that
// have nodes nodes together.
int launch_form(const lbmice_batch_t* b, int s, int steps, long long nodes) {
  if (s != LBMICE_SHAPE_MARCH) return s;
  if (steps == 2) return nodes <= kBatchTileMaxNodes ? FORM_TWO_TILE : FORM_TWO_MARCH;
  return b->two && nodes <= batch_single_tile_nodes(b->flow != 0) ? LBMICE_SHAPE_32x8
                                                                  : LBMICE_SHAPE_MARCH;
}

// One launch of steps (1, or 2 with the march shape) time steps of the members of shape s among
// the listed ones, or several where they are more than kBatchMaxMembers; f[i] is member i's
// buffer phase.
int launch_shape(lbmice_batch_t* b, const std::vector<int>& idx, int s, std::vector<Phase>& f,
                 int steps, cudaStream_t st) {
  for (size_t k = 0; k < idx.size();) {
    BatchLaunch& L = *b->block;
    L.n = 0;
    L.tile_start[0] = 0;
    int in[kBatchMaxMembers];  // the members of this launch
    long long nodes = 0;
    for (; k < idx.size() && L.n < kBatchMaxMembers; ++k)
      if (b->shape[idx[k]] == s) {
        in[L.n++] = idx[k];
        nodes += (long long)b->members[idx[k]]->C.nx * b->members[idx[k]]->C.ny;
      }
    if (L.n == 0) break;
    const int form = launch_form(b, s, steps, nodes);
    for (int j = 0; j < L.n; ++j) {
      const lbmice_t* h = b->members[in[j]];
      BatchDesc& d = L.d[j];
      d.C = h->C;
      d.C.seg_rows = kMarchMaxSegRows;
      d.C.two_rows = kBatchTwoRows;
      d.P = step_ptrs(h, f[in[j]], steps);
      d.tiles_x = form >= kNumShapes           ? two_strips(h->C.nx)
                  : form == LBMICE_SHAPE_MARCH ? march_strips(h->C.nx)
                                               : (h->C.nx + shape_tx(form) - 1) / shape_tx(form);
      d.pad_ = 0;
      L.tile_start[j + 1] = L.tile_start[j] + member_units(h, form);
      f[in[j]].advance(steps);
    }
    const long long units = L.tile_start[L.n];
    const int rc = form >= kNumShapes           ? launch_two_block(b, form, units, st)
                   : form == LBMICE_SHAPE_MARCH ? launch_march_block(b, units, st)
                   : form == LBMICE_SHAPE_32x8  ? launch_block<32, 8>(b, units, st)
                   : form == LBMICE_SHAPE_64x4  ? launch_block<64, 4>(b, units, st)
                                                : launch_block<16, 16>(b, units, st);
    if (rc != LBMICE_OK) return rc;
  }
  return LBMICE_OK;
}

// steps (1 or 2) time steps of the listed members from the buffer phases f, which advance: one
// launch per shape in use and per kBatchMaxMembers members of that shape (the tile shapes take
// two steps in two launches).
int launch_members(lbmice_batch_t* b, const std::vector<int>& idx, std::vector<Phase>& f, int steps,
                   cudaStream_t st) {
  for (int s = 0; s < kNumShapes; ++s) {
    const int each = s == LBMICE_SHAPE_MARCH ? steps : 1;
    for (int done = 0; done < steps; done += each) {
      const int rc = launch_shape(b, idx, s, f, each, st);
      if (rc != LBMICE_OK) return rc;
    }
  }
  return LBMICE_OK;
}

int batch_launch_steps(const lbmice_batch_t* b, int64_t left) { return b->two && left >= 2 ? 2 : 1; }

std::vector<Phase> batch_phases(const lbmice_batch_t* b) {
  std::vector<Phase> f;
  for (const lbmice_t* m : b->members) f.push_back(phase_of(m));
  return f;
}
// The members after steps steps, which ended in the buffer phases f.
void set_phases(lbmice_batch_t* b, const std::vector<Phase>& f, int64_t steps) {
  for (size_t i = 0; i < f.size(); ++i) {
    b->members[i]->cur = f[i].cur;
    b->members[i]->ring = f[i].s;
    b->members[i]->step += steps;
  }
}

void batch_release(lbmice_batch_t* b) {
  for (const auto& g : b->graphs) cudaGraphExecDestroy(g.exec);
  for (lbmice_t* m : b->members) if (m) lbmice_destroy(m);
  if (b->capture) cudaStreamDestroy(b->capture);
  delete b;
}

std::vector<int> all_members(const lbmice_batch_t* b) {
  std::vector<int> v(b->members.size());
  for (size_t i = 0; i < v.size(); ++i) v[i] = (int)i;
  return v;
}

bool in_lockstep(const lbmice_batch_t* b) {
  for (const lbmice_t* m : b->members)
    if (m->step != batch_steps(b)) return false;
  return true;
}

void drop_graphs(lbmice_batch_t* b) {
  for (const auto& g : b->graphs) cudaGraphExecDestroy(g.exec);
  b->graphs.clear();
}

// The graph of kGraphSteps steps from the members' buffer phases, captured when first needed; at
// most kMaxPhases are kept.
int batch_graph(lbmice_batch_t* b, cudaGraphExec_t* out) {
  std::vector<int> from;
  for (const lbmice_t* m : b->members) from.push_back(phase_index(m, phase_of(m)));
  for (const auto& g : b->graphs)
    if (g.from == from) {
      *out = g.exec;
      return LBMICE_OK;
    }
  if (b->graphs.size() >= kMaxPhases) drop_graphs(b);
  const std::vector<int> all = all_members(b);
  std::vector<Phase> f = batch_phases(b);
  cudaGraph_t g = nullptr;
  LB_TRY(cudaStreamBeginCapture(b->capture, cudaStreamCaptureModeThreadLocal));
  int rc = LBMICE_OK;
  for (int64_t left = kGraphSteps; left > 0 && rc == LBMICE_OK;) {
    const int n = batch_launch_steps(b, left);
    rc = launch_members(b, all, f, n, b->capture);
    left -= n;
  }
  cudaError_t e = cudaStreamEndCapture(b->capture, &g);
  if (rc != LBMICE_OK) { if (g) cudaGraphDestroy(g); return rc; }
  if (e != cudaSuccess) return cuda_err(e);
  cudaGraphExec_t exec = nullptr;
  e = cudaGraphInstantiate(&exec, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) return cuda_err(e);
  b->graphs.push_back({std::move(from), exec});
  *out = exec;
  return LBMICE_OK;
}

}  // namespace

extern "C" {

int lbmice_batch_create(const lbmice_params* params, int32_t count, void* stream,
                        lbmice_batch_t** out) {
  if (!out) return LBMICE_EINVAL;
  *out = nullptr;
  if (!params || count < 1) return LBMICE_EINVAL;
  for (int i = 0; i < count; ++i) {
    if (params[i].flow != params[0].flow || params[i].storage != params[0].storage)
      return LBMICE_EINVAL;
    // the batched tile is the default one: E4 gradient, six-fold anisotropy
    if ((params[i].stencil != 0 && params[i].stencil != 4) ||
        (params[i].fold != 0 && params[i].fold != 6))
      return LBMICE_EINVAL;
    const int rc = validate(params[i]);
    if (rc != LBMICE_OK) return rc;
  }
  lbmice_batch_t* b = new (std::nothrow) lbmice_batch();
  if (!b) return LBMICE_ENOMEM;
  b->block.reset(new (std::nothrow) BatchLaunch());
  if (!b->block) {
    delete b;
    return LBMICE_ENOMEM;
  }
  b->stream = static_cast<cudaStream_t>(stream);
  b->flow = params[0].flow;
  b->storage = params[0].storage;
  b->members.assign(count, nullptr);
  b->shape.assign(count, LBMICE_SHAPE_MARCH);
  for (int i = 0; i < count; ++i) {
    const int rc = create_grid(&params[i], stream, true, &b->members[i]);
    if (rc != LBMICE_OK) {
      batch_release(b);
      return rc;
    }
  }
  b->two = params[0].storage == LBMICE_STORAGE_F32;
  for (const lbmice_t* m : b->members) b->two = b->two && two_step(m);
  const cudaError_t e = cudaStreamCreateWithFlags(&b->capture, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    batch_release(b);
    return cuda_err(e);
  }
  *out = b;
  return LBMICE_OK;
}

int32_t lbmice_batch_size(const lbmice_batch_t* b) { return b ? (int32_t)b->members.size() : 0; }

lbmice_t* lbmice_batch_member(lbmice_batch_t* b, int32_t i) {
  if (!b || i < 0 || i >= (int32_t)b->members.size()) return nullptr;
  return b->members[i];
}

int lbmice_batch_set_shape(lbmice_batch_t* b, int32_t i, int32_t shape) {
  if (!b || i < 0 || i >= (int32_t)b->members.size() || shape < 0 || shape >= kNumShapes)
    return LBMICE_EINVAL;
  b->shape[i] = shape;
  drop_graphs(b);  // launches already queued keep the parameter blocks they were given
  return LBMICE_OK;
}

int lbmice_batch_step(lbmice_batch_t* b, int64_t nsteps) {
  if (!b || nsteps < 0) return LBMICE_EINVAL;
  if (!in_lockstep(b)) return LBMICE_EINVAL;
  const std::vector<int> all = all_members(b);
  bool turn = false;
  for (const lbmice_t* m : b->members) turn = turn || two_step(m);
  turn = turn && ends_in_turn(nsteps, b->stream);
  int64_t left = turn ? nsteps - kTurnSteps : nsteps;
  while (left > 0) {
    if (left >= kGraphSteps) {
      cudaGraphExec_t g = nullptr;
      const int rc = batch_graph(b, &g);
      if (rc != LBMICE_OK) return rc;
      LB_TRY(cudaGraphLaunch(g, b->stream));
      for (lbmice_t* m : b->members) {
        m->step += kGraphSteps;
        m->ring += kGraphSteps;
      }
      left -= kGraphSteps;
    } else {
      const int n = batch_launch_steps(b, left);
      std::vector<Phase> f = batch_phases(b);
      const int rc = launch_members(b, all, f, n, b->stream);
      if (rc != LBMICE_OK) return rc;
      set_phases(b, f, n);
      left -= n;
    }
  }
  if (turn) {
    std::vector<Phase> f = batch_phases(b);
    for (Phase& p : f) p.turn = 0;
    for (int k = 0; k < kTurnSteps; ++k) {
      const int rc = launch_members(b, all, f, 1, b->stream);
      if (rc != LBMICE_OK) return rc;
    }
    set_phases(b, f, kTurnSteps);
  }
  return LBMICE_OK;
}

int lbmice_batch_autotune(lbmice_batch_t* b, int32_t steps_per_trial, int32_t* shapes,
                          int64_t* steps_taken) {
  if (!b || steps_per_trial < 1) return LBMICE_EINVAL;
  if (!in_lockstep(b)) return LBMICE_EINVAL;
  const int n = (int)b->members.size();
  drop_graphs(b);
  // size classes
  std::vector<std::pair<int, int>> classes;
  for (const lbmice_t* m : b->members) {
    const std::pair<int, int> key(m->C.nx, m->C.ny);
    if (std::find(classes.begin(), classes.end(), key) == classes.end()) classes.push_back(key);
  }
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  LB_TRY(cudaEventCreate(&e0));
  LB_TRY(cudaEventCreate(&e1));
  int64_t taken = 0;
  int rc = LBMICE_OK;
  for (const auto& cls : classes) {
    std::vector<int> in, rest;
    for (int i = 0; i < n; ++i)
      (b->members[i]->C.nx == cls.first && b->members[i]->C.ny == cls.second ? in : rest)
          .push_back(i);
    float best = 0.0f;
    int best_shape = 0;
    for (int s = 0; s < kNumShapes && rc == LBMICE_OK; ++s) {
      for (int i : in) b->shape[i] = s;
      // one untimed step, then the timed steps of this class; the other members take the same number
      // of steps untimed, so the batch stays in lockstep. A batch in pairs is timed in pairs: with
      // an odd count the untimed launch leaves the phase where it is (the timed ones write the same
      // results again) and the step it stood for is timed, too
      std::vector<Phase> f = batch_phases(b);
      const auto take = [&](const std::vector<int>& idx, int64_t left) {
        while (left > 0 && rc == LBMICE_OK) {
          const int n = batch_launch_steps(b, left);
          rc = launch_members(b, idx, f, n, b->stream);
          left -= n;
        }
      };
      const bool whole = b->two && steps_per_trial % 2 == 1;
      if (whole) {
        std::vector<Phase> again = f;
        rc = launch_members(b, in, again, s == LBMICE_SHAPE_MARCH ? 2 : 1, b->stream);
      } else {
        take(in, 1);
      }
      if (rc == LBMICE_OK) rc = cuda_err(cudaEventRecord(e0, b->stream));
      take(in, (int64_t)steps_per_trial + (whole ? 1 : 0));
      if (rc == LBMICE_OK) rc = cuda_err(cudaEventRecord(e1, b->stream));
      if (!rest.empty()) take(rest, (int64_t)steps_per_trial + 1);
      if (rc == LBMICE_OK) set_phases(b, f, (int64_t)steps_per_trial + 1);
      if (rc == LBMICE_OK) rc = cuda_err(cudaStreamSynchronize(b->stream));
      float ms = 0.0f;
      if (rc == LBMICE_OK) rc = cuda_err(cudaEventElapsedTime(&ms, e0, e1));
      if (rc == LBMICE_OK) {
        taken += steps_per_trial + 1;
        if (s == 0 || ms < best) {
          best = ms;
          best_shape = s;
        }
      }
    }
    for (int i : in) b->shape[i] = best_shape;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc != LBMICE_OK) return rc;
  if (shapes)
    for (int i = 0; i < n; ++i) shapes[i] = b->shape[i];
  if (steps_taken) *steps_taken = taken;
  return LBMICE_OK;
}

int lbmice_batch_destroy(lbmice_batch_t* b) {
  if (!b) return LBMICE_OK;
  cudaError_t e = cudaStreamSynchronize(b->stream);
  batch_release(b);
  return cuda_err(e);
}

}  // extern "C"

// ---------------------------------------------------------------------------------------
// Tape: a checkpointed forward record of one grid and the discrete adjoint of its steps
// (periodic faces, FP32 storage). Checkpoints are state blobs every `every` steps; the
// reverse sweep restores each segment's checkpoint, recomputes the segment's states with the
// step kernel and runs the adjoint kernels backwards through them.
// ---------------------------------------------------------------------------------------
struct lbmice_tape {
  lbmice_t* h = nullptr;           // the recorded grid (borrowed)
  int every = 100;                 // checkpoint interval
  int64_t steps = 0;               // steps recorded
  std::vector<void*> ckpt;         // states at steps 0, every, 2 every, ...
  // reverse-sweep work space, allocated by the first backward
  void* work = nullptr;            // the device allocation holding every buffer below
  int work_len = 0;                // steps of the longest segment it has room for
  std::vector<float*> seg_pops;    // work_len population buffers: states of one segment
  std::vector<float*> seg_phi;     // work_len + 1 phi planes: phi^{s0-1}, phi^{s0}, ...
  float* pb[2] = {nullptr, nullptr};
  float* Phib[2] = {nullptr, nullptr};
  float* Psib[2] = {nullptr, nullptr};
  std::vector<float*> plane;       // scratch planes, see enum below
  double* partial = nullptr;       // [blocks][kAdjParams]
  int nblocks = 0;
  // the pull's own-population term inside the collision adjoint (grids whose reverse working
  // set, about 4 x 116 B per node, exceeds the L2), else in a separate read-modify-write pass
  bool fused = false;
  // a full segment's recompute and reverse steps as a CUDA graph, one per starting parity of
  // the adjoint ping-pong (every argument is the same for every full segment)
  cudaGraphExec_t seg_graph[2] = {nullptr, nullptr};
};

namespace {

enum : int {
  TP_PHIB_LOC = 0, TP_GBX, TP_GBY, TP_BN, TP_SEED_PHI, TP_SEED_U, TP_PHI0B, TP_U0B, TP_RHO0B,
  TP_UX0B, TP_UY0B, TP_NPLANES
};

bool tape_supported(const lbmice_t* h) {
  if (h->p.storage != LBMICE_STORAGE_F32) return false;
  for (int f = 0; f < 4; ++f)
    if (h->p.bc[f] != LBMICE_BC_PERIODIC) return false;
  return true;
}

// State blob of the current step, kept when the step is a multiple of the interval.
int tape_checkpoint(lbmice_tape_t* t) {
  const size_t c = (size_t)(t->steps / t->every);
  if (c < t->ckpt.size()) return LBMICE_OK;
  void* blob = nullptr;
  LB_TRY(cudaMalloc(&blob, lbmice_state_bytes(t->h)));
  t->ckpt.push_back(blob);
  return copy_state(t->h, blob, true, cudaMemcpyDeviceToDevice);
}

void tape_drop_graphs(lbmice_tape_t* t) {
  for (cudaGraphExec_t& g : t->seg_graph) {
    if (g) cudaGraphExecDestroy(g);
    g = nullptr;
  }
}

// Work space for segments of up to len steps in one allocation.
int tape_take_work(lbmice_tape_t* t, int len) {
  const lbmice_t* h = t->h;
  t->seg_pops.assign(len, nullptr);
  t->seg_phi.assign(len + 1, nullptr);
  t->plane.assign(TP_NPLANES, nullptr);
  t->nblocks = ((h->C.nx + 31) / 32) * ((h->C.ny + 7) / 8);
  Slab s;
  for (float*& b : t->plane) s.place(&b, field_bytes(h));
  const size_t zeroed = s.bytes();  // planes are read over their full pitch by the copies out
  for (float*& b : t->seg_pops) s.place(&b, pop_bytes(h));
  for (float*& b : t->seg_phi) s.place(&b, field_bytes(h));
  for (int k = 0; k < 2; ++k) {
    s.place(&t->pb[k], pop_bytes(h));
    s.place(&t->Phib[k], field_bytes(h));
    s.place(&t->Psib[k], field_bytes(h));
  }
  s.place(&t->partial, sizeof(double) * kAdjParams * t->nblocks);
  LB_TRY(s.allocate(&t->work));
  t->work_len = len;
  LB_TRY(cudaMemsetAsync(t->work, 0, zeroed, h->stream));
  return LBMICE_OK;
}

// Work space for segments of up to len steps, kept for the next sweep. A tape swept again and again
// while its first segment is still being recorded needs more each time: space that has to grow
// grows to twice the need where that fits, so that such a tape allocates a few times, not at every
// sweep.
int tape_alloc_work(lbmice_tape_t* t, int len) {
  if (t->work && t->work_len >= len) return LBMICE_OK;
  if (t->work) {
    LB_TRY(cudaStreamSynchronize(t->h->stream));
    tape_drop_graphs(t);
    LB_TRY(cudaFree(t->work));
    t->work = nullptr;
    const int more = (int)std::min<int64_t>(t->every, 2LL * len);
    if (more > len) {
      const int rc = tape_take_work(t, more);
      if (rc != LBMICE_ENOMEM) return rc;
      cudaGetLastError();
    }
  }
  return tape_take_work(t, len);
}

void tape_free(lbmice_tape_t* t) {
  tape_drop_graphs(t);
  for (void* b : t->ckpt) cudaFree(b);
  if (t->work) cudaFree(t->work);
  delete t;
}

// Checkpoint c into the first state of the segment buffers (blob: populations, phi^n,
// phi^{n-1}, as copy_state writes it for FP32 storage).
int tape_restore(lbmice_tape_t* t, size_t c) {
  const lbmice_t* h = t->h;
  const char* b = static_cast<const char*>(t->ckpt[c]);
  LB_TRY(cudaMemcpyAsync(t->seg_pops[0], b, pop_bytes(h), cudaMemcpyDeviceToDevice, h->stream));
  b += pop_bytes(h);
  LB_TRY(cudaMemcpyAsync(t->seg_phi[1], b, field_bytes(h), cudaMemcpyDeviceToDevice,
                         h->stream));
  b += field_bytes(h);
  LB_TRY(cudaMemcpyAsync(t->seg_phi[0], b, field_bytes(h), cudaMemcpyDeviceToDevice,
                         h->stream));
  return LBMICE_OK;
}

// State j of the segment to state j + steps (steps = 2: to j + 1 as well).
StepPtrs tape_step_ptrs(const lbmice_tape_t* t, int j, int steps) {
  StepPtrs P{};
  P.pin = t->seg_pops[j];
  P.pout = t->seg_pops[j + steps];
  P.phi_n = t->seg_phi[j + 1];
  P.phi_nm1 = t->seg_phi[j];
  P.phi_np1 = t->seg_phi[j + 1 + steps];
  step_regions(P, t->h->C, dev16(t->h));
  if (steps == 2) {
    StepPtrs M{};
    M.pin = M.pout = t->seg_pops[j + 1];
    step_regions(M, t->h->C, dev16(t->h));
    std::memcpy(P.rmid, M.rout, sizeof(P.rmid));
    P.phi_mid = t->seg_phi[j + 2];
  }
  return P;
}

dim3 adj_grid(const lbmice_t* h) { return dim3((h->C.nx + 31) / 32, (h->C.ny + 7) / 8); }

// Reverse step through segment state j: adjoint buffers cur -> 1 - cur.
int tape_reverse_step(lbmice_tape_t* t, int j, int cur, cudaStream_t st) {
  const lbmice_t* h = t->h;
  AdjPtrs A;
  A.pops = t->seg_pops[j];
  A.phi_n = t->seg_phi[j + 1];
  A.phi_nm1 = t->seg_phi[j];
  A.pb_in = t->pb[cur];
  A.Phib_in = t->Phib[cur];
  A.Psib_in = t->Psib[cur];
  A.pb_out = t->pb[1 - cur];
  A.Phib_out = t->Phib[1 - cur];
  A.Psib_out = t->Psib[1 - cur];
  A.phib_loc = t->plane[TP_PHIB_LOC];
  A.gbx = t->plane[TP_GBX];
  A.gby = t->plane[TP_GBY];
  A.Bn = t->plane[TP_BN];
  A.partial = t->partial;
  const auto go = [&](void (*kern)(Consts, AdjPtrs)) {
    return launch_overlapped(kern, adj_grid(h), 256, 0, st, h->C, A);
  };
  int rc = LBMICE_OK;
  if (t->fused) {
    rc = go(adj_b_kernel);
    if (rc == LBMICE_OK)
      rc = go(h->p.flow ? adj_collide_kernel<true, true> : adj_collide_kernel<false, true>);
    if (rc == LBMICE_OK) rc = go(adj_stencil_kernel);
  } else {
    rc = go(h->p.flow ? adj_collide_kernel<true, false> : adj_collide_kernel<false, false>);
    if (rc == LBMICE_OK) rc = go(adj_pull_kernel);
  }
  return rc;
}

// Recompute the states of a segment of len steps from its restored first state, then run
// the reverse steps through them, starting from adjoint buffer cur.
int tape_segment(lbmice_tape_t* t, int len, int cur, cudaStream_t st) {
  int rc = LBMICE_OK;
  // two states per launch for small grids; storing both, a launch of a larger one moves about as
  // much per step as a single step does (reverse sweep, us per step, pairs / single: 96^2 without
  // flow 10.0 / 11.1, 256^2 14.2 / 15.8, 512^2 39.0 / 39.2, 1024^2 140.5 / 138.5)
  const lbmice_t* h = t->h;
  const bool pairs =
      two_step(h) && h->tile_warps != 0 && (long long)h->C.nx * h->C.ny <= kTapePairsMaxNodes;
  for (int j = 0; j + 1 < len && rc == LBMICE_OK;) {
    if (pairs && j + 2 < len) {
      rc = launch_tiles(h, tape_step_ptrs(t, j, 2), true, st);
      j += 2;
    } else {
      rc = launch_step_ptrs(t->h, tape_step_ptrs(t, j, 1), st);
      j += 1;
    }
  }
  for (int j = len - 1; j >= 0 && rc == LBMICE_OK; --j) {
    rc = tape_reverse_step(t, j, cur, st);
    cur = 1 - cur;
  }
  return rc;
}

// [ny][nx] float array (host or device) <-> [ny][pitch] plane.
int plane_in(const lbmice_t* h, float* plane, const float* src) {
  const size_t w = sizeof(float) * h->C.nx;
  LB_TRY(cudaMemcpy2DAsync(plane, sizeof(float) * h->C.pitch, src, w, w, h->C.ny,
                           cudaMemcpyDefault, h->stream));
  return LBMICE_OK;
}
int plane_out(const lbmice_t* h, float* dst, const float* plane) {
  const size_t w = sizeof(float) * h->C.nx;
  LB_TRY(cudaMemcpy2DAsync(dst, w, plane, sizeof(float) * h->C.pitch, w, h->C.ny,
                           cudaMemcpyDefault, h->stream));
  return LBMICE_OK;
}

}  // namespace

extern "C" {

int lbmice_tape_create(lbmice_t* h, int32_t every, lbmice_tape_t** out) {
  if (!out) return LBMICE_EINVAL;
  *out = nullptr;
  if (!h || every < 1 || !tape_supported(h) || h->step != 0) return LBMICE_EINVAL;
  if (h->C.stencil != 4 || h->C.fold != 6) return LBMICE_EINVAL;  // the adjoint's E4, six-fold
  lbmice_tape_t* t = new (std::nothrow) lbmice_tape();
  if (!t) return LBMICE_ENOMEM;
  t->h = h;
  t->every = every;
  {
    // the fused reverse pull for grids whose reverse working set exceeds the L2;
    // LBMICE_ADJ_FUSED=0 or 1 in the environment forces one form (both give the same bits)
    int l2 = 0;
    if (cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, h->device) != cudaSuccess) l2 = 0;
    t->fused = 4.0 * 116.0 * (double)h->C.nx * (double)h->C.ny > (double)l2;
    if (const char* e = std::getenv("LBMICE_ADJ_FUSED")) {
      if (e[0] == '0' && e[1] == 0) t->fused = false;
      if (e[0] == '1' && e[1] == 0) t->fused = true;
    }
  }
  const int rc = tape_checkpoint(t);
  if (rc != LBMICE_OK) {
    tape_free(t);
    return rc;
  }
  *out = t;
  return LBMICE_OK;
}

int64_t lbmice_tape_steps(const lbmice_tape_t* t) { return t ? t->steps : -1; }

int lbmice_tape_record(lbmice_tape_t* t, int64_t nsteps) {
  if (!t || nsteps < 0) return LBMICE_EINVAL;
  if (t->h->step != t->steps) return LBMICE_EINVAL;  // stepped outside the tape
  int64_t left = nsteps;
  while (left > 0) {
    const int64_t chunk = std::min<int64_t>(left, t->every - t->steps % t->every);
    const int rc = lbmice_step(t->h, chunk);
    t->steps = t->h->step;
    if (rc != LBMICE_OK) return rc;
    left -= chunk;
    if (t->steps % t->every == 0) {
      const int rc2 = tape_checkpoint(t);
      if (rc2 != LBMICE_OK) return rc2;
    }
  }
  return LBMICE_OK;
}

int lbmice_tape_backward(lbmice_tape_t* t, const float* phi_bar, const float* U_bar,
                         double grads[3], float* phi0_bar, float* U0_bar, float* rho0_bar,
                         float* ux0_bar, float* uy0_bar) {
  if (!t) return LBMICE_EINVAL;
  lbmice_t* h = t->h;
  if (h->step != t->steps) return LBMICE_EINVAL;
  // a segment of len steps keeps len states (its last step's result is not read back)
  const int longest = (int)std::max<int64_t>(1, std::min<int64_t>(t->every, t->steps));
  int rc = tape_alloc_work(t, longest);
  if (rc != LBMICE_OK) return rc;
  const dim3 g = adj_grid(h);
  // seed: dL/dphi_T into the phi-plane adjoint, dL/dU_T into the g adjoints
  if (phi_bar && (rc = plane_in(h, t->plane[TP_SEED_PHI], phi_bar)) != LBMICE_OK) return rc;
  if (U_bar && (rc = plane_in(h, t->plane[TP_SEED_U], U_bar)) != LBMICE_OK) return rc;
  const float* sp = phi_bar ? t->plane[TP_SEED_PHI] : nullptr;
  const float* su = U_bar ? t->plane[TP_SEED_U] : nullptr;
  if (h->p.flow)
    adj_seed_kernel<true><<<g, 256, 0, h->stream>>>(h->C, sp, su, t->pb[0], t->Phib[0],
                                                    t->Psib[0]);
  else
    adj_seed_kernel<false><<<g, 256, 0, h->stream>>>(h->C, sp, su, t->pb[0], t->Phib[0],
                                                     t->Psib[0]);
  LB_TRY(cudaGetLastError());
  LB_TRY(cudaMemsetAsync(t->partial, 0, sizeof(double) * kAdjParams * t->nblocks, h->stream));
  int cur = 0;
  // segments from the last: restore, recompute its states, reverse through them
  const int64_t nseg = (t->steps + t->every - 1) / t->every;
  for (int64_t c = nseg - 1; c >= 0; --c) {
    const int64_t s0 = c * t->every;
    const int len = (int)std::min<int64_t>(t->every, t->steps - s0);
    if ((rc = tape_restore(t, (size_t)c)) != LBMICE_OK) return rc;
    // full segments replay a graph where there are enough of them to pay for its capture and
    // instantiation (about as long as queueing the launches of two segments)
    if (len == t->every && t->steps / t->every >= kTapeGraphSegments) {
      if (!t->seg_graph[cur]) {
        cudaGraph_t gr = nullptr;
        LB_TRY(cudaStreamBeginCapture(h->capture, cudaStreamCaptureModeThreadLocal));
        rc = tape_segment(t, len, cur, h->capture);
        const cudaError_t e = cudaStreamEndCapture(h->capture, &gr);
        if (rc != LBMICE_OK) { if (gr) cudaGraphDestroy(gr); return rc; }
        if (e != cudaSuccess) return cuda_err(e);
        const cudaError_t ei = cudaGraphInstantiate(&t->seg_graph[cur], gr, 0);
        cudaGraphDestroy(gr);
        if (ei != cudaSuccess) { t->seg_graph[cur] = nullptr; return cuda_err(ei); }
      }
      LB_TRY(cudaGraphLaunch(t->seg_graph[cur], h->stream));
    } else if ((rc = tape_segment(t, len, cur, h->stream)) != LBMICE_OK) {
      return rc;
    }
    if (len & 1) cur = 1 - cur;
  }
  if (nseg == 0 && (rc = tape_restore(t, 0)) != LBMICE_OK) return rc;
  // initial state: adjoints of the moments it was built from
  InitAdjPtrs I;
  I.pops = t->seg_pops[0];
  I.phi0 = t->seg_phi[1];
  I.pb = t->pb[cur];
  I.Phib = t->Phib[cur];
  I.Psib = t->Psib[cur];
  I.phib_loc = t->plane[TP_PHIB_LOC];
  I.gbx = t->plane[TP_GBX];
  I.gby = t->plane[TP_GBY];
  I.Ub = t->plane[TP_U0B];
  I.rhob = t->plane[TP_RHO0B];
  I.uxb = t->plane[TP_UX0B];
  I.uyb = t->plane[TP_UY0B];
  I.partial = t->partial;
  if (h->p.flow)
    adj_init_kernel<true><<<g, 256, 0, h->stream>>>(h->C, I);
  else
    adj_init_kernel<false><<<g, 256, 0, h->stream>>>(h->C, I);
  adj_gather_kernel<<<g, 256, 0, h->stream>>>(h->C, t->plane[TP_PHIB_LOC], t->plane[TP_GBX],
                                              t->plane[TP_GBY], t->plane[TP_PHI0B]);
  LB_TRY(cudaGetLastError());
  const float* outs[5] = {t->plane[TP_PHI0B], t->plane[TP_U0B], t->plane[TP_RHO0B],
                          t->plane[TP_UX0B], t->plane[TP_UY0B]};
  float* dsts[5] = {phi0_bar, U0_bar, rho0_bar, ux0_bar, uy0_bar};
  for (int k = 0; k < 5; ++k)
    if (dsts[k] && (rc = plane_out(h, dsts[k], outs[k])) != LBMICE_OK) return rc;
  std::vector<double> part((size_t)kAdjParams * t->nblocks);
  LB_TRY(cudaMemcpyAsync(part.data(), t->partial, sizeof(double) * part.size(),
                         cudaMemcpyDeviceToHost, h->stream));
  LB_TRY(cudaStreamSynchronize(h->stream));
  double sum[kAdjParams] = {0.0, 0.0, 0.0, 0.0};
  for (int b = 0; b < t->nblocks; ++b)
    for (int k = 0; k < kAdjParams; ++k) sum[k] += part[(size_t)b * kAdjParams + k];
  if (grads) {
    const lbmice_params& p = h->p;
    // eps enters as eps and as kappa_N 6 eps; D as D_lat3 = 3 D dt/dx^2 and, when lambda is
    // not given, through the beta = 0 lambda = tau0 D / (a2 W0^2) (Sec. 2.1)
    grads[0] = sum[ADJ_EPS] + 6.0 * p.kappa_N * sum[ADJ_KN6EPS];
    grads[1] = sum[ADJ_DLAT3] * 3.0 * p.dt / (p.dx * p.dx);
    if (!(p.lambda > 0)) grads[1] += sum[ADJ_LAMBDA] * p.tau0 / (kA2 * p.W0 * p.W0);
    grads[2] = sum[ADJ_LAMBDA];
  }
  return LBMICE_OK;
}

int lbmice_tape_destroy(lbmice_tape_t* t) {
  if (!t) return LBMICE_OK;
  const cudaError_t e = cudaStreamSynchronize(t->h->stream);
  tape_free(t);
  return cuda_err(e);
}

}  // extern "C"

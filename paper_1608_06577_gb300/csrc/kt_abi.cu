// kt_abi.cu -- host side of libkt: the C ABI declared in include/kt.h.
//
// A context holds one or more events.  Every field array spans all events: component n of
// event e starts at n * gs + base_e (gs = sum of the events' padded sizes), so one persistent
// launch per Runge-Kutta stage can walk a table of (event, tile) work items.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include "../../include/kt.h"
#include "kt_split.cuh"

using namespace kt;

namespace {

constexpr int KSTAT_WORDS = 12;  // device stats block: status, max speed bits, pad, 3 u64 counters from word 4

struct Shape {
  int x, y, z;
};
// candidate tile shapes of the autotuner (threads per block; x stays 32 so a warp is one x-row)
constexpr Shape kShapes[] = {{32, 4, 2}, {32, 8, 1}, {32, 2, 4}, {32, 1, 8}, {32, 4, 1}, {32, 2, 2}};
constexpr int kNumShapes = sizeof(kShapes) / sizeof(kShapes[0]);
// candidates: every shape with a persistent grid (blocks resident at once) and with one block per tile,
// each (mixed precision) as a right-hand-side and an update launch per stage, the update reading
// its inputs directly or staged by TMA, or as one fused launch per stage.  The autotuner times the
// split launches with direct reads (0-11) and, where the context can run them, the fused ones
// (24-35); the TMA-staged update measured slower over a whole step and is selected only by
// kt_set_tuning.
constexpr int kNumBase = 2 * kNumShapes;
constexpr int kNumCandidates = 3 * kNumBase;
constexpr int kFusedFirst = 2 * kNumBase;

// A run of events [ev0, ev1) that the mixed-precision kernels take in one launch: their lattices lie within
// kSpanElements of `base`, where the launch's field pointers start.  tile0, ntiles: their tiles.
struct Span {
  int ev0, ev1;
  long long base;
  int tile0, ntiles;
};

struct Ctx {
  kt_options opt;
  Params P;
  int mixed = 0;         // 1: float u, e, p and float stencil
  size_t esz = 8;        // bytes per u/e/p element
  int device = 0;        // the device its memory and kernels are on
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  // events
  int nev = 0;
  std::vector<Lattice> lat;
  std::vector<Span> spans;  // mixed precision: the events of each launch
  long long gs = 0;      // component stride of every field array
  size_t max_cells = 0;  // physical cells of the largest event
  std::vector<char> ev_set;
  // device memory
  void* base = nullptr;  // owned allocation (null if caller arena)
  size_t bytes = 0;
  double* q = nullptr;   // 15 components
  double* qs = nullptr;  // 15 components
  float* qf = nullptr;   // mixed mode: FP32 copies of q and qs read by the stencil
  float* qsf = nullptr;
  void* U[3] = {};       // 3 x 4 components
  void* E[2] = {};
  void* Pb[2] = {};
  double* stage = nullptr;  // staging: 18 packed fields of the largest event
  EosSeg<double>* seg_d = nullptr;
  RootSeg* seg_r = nullptr;
  RootSegM* seg_m = nullptr;
  FaceSeg* seg_face = nullptr;
  SourceSeg* seg_src = nullptr;
  TauSlot* d_tau = nullptr;  // three slots, used in rotation with the u buffers: tau^n is in slot cur
  unsigned* d_stat = nullptr;
  float* d_mlp = nullptr;
  uint32_t* d_mlp_packed = nullptr;
  Lattice* d_lat = nullptr;        // mixed precision: bases relative to the event's span
  Tile* d_tiles = nullptr;
  CUtensorMap map0[2] = {};        // mixed precision: the first event's maps of qf and qsf (kernel parameters)
  CUtensorMap* d_tmaps = nullptr;  // mixed precision: per event, the 4-d maps of qf (first nev) and qsf
  CUtensorMap* d_umaps = nullptr;  // mixed precision: per event, the kUpdMaps maps of the staged update
  int staged = 0;                  // the update kernels read their inputs staged by TMA
  int fused = 0;                   // one fused launch per stage (right-hand side + update)
  int upd_nbuf = 1;                // staged update: buffers per block (2 on a persistent grid)
  float* reg = nullptr;            // regulation factor of the last step, per cell (diagnostics)
  float* z_net = nullptr;          // learned start: the network's output per cell for the current step
  int grid_mlp = 1;                // blocks of mlp_start_kernel
  int max_tiles = 0;
  // work decomposition
  int shape = 0;
  int ntiles = 0;
  int grid_blocks = 0;    // the stage kernel's blocks (FP64), or grid_rhs
  int team = 0;           // FP64: four warps per strip (stage_team_kernel)
  int grid_rhs = 0;       // mixed precision: right-hand-side kernel
  int grid_upd = 0;       // mixed precision: update kernel
  bool tuned = false;
  int cand = 0;
  float tune_ms[kNumCandidates] = {};
  int learned = 0;
  int pi32 = 0;          // KT_STORE_PI_FP32: pi, Pi live in the FP32 array qf (components 4-14)
  int cur = 0, prev = 1, spare = 2;
  double tau = 0.0;
  long long steps = 0;
  cudaGraphExec_t graph[3] = {nullptr, nullptr, nullptr};  // 3-step graph per rotation phase
  kt_stats last{};
  char err[512] = {0};
};

int fail(Ctx* c, int code, const char* fmt, ...) {
  if (c) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(c->err, sizeof(c->err), fmt, ap);
    va_end(ap);
  }
  return code;
}

// NVTX range for the duration of a host call (visible in Nsight timelines; no cost without a tool)
struct Range {
  explicit Range(const char* name) { nvtxRangePushA(name); }
  ~Range() { nvtxRangePop(); }
};

#define CK(call)                                                                                 \
  do {                                                                                           \
    cudaError_t e_ = (call);                                                                     \
    if (e_ != cudaSuccess) return fail(c, KT_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

// Whether this context's kernels may read and write the caller's device array in place: memory of their own
// device, aligned for doubles.  Anything else that a copy can reach (another device's memory without peer
// access, an array at an odd offset) is copied.
bool in_place(const Ctx* c, const void* p) {
  if ((uintptr_t)p % alignof(double)) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();  // not an error of this call
    return false;
  }
  return a.type == cudaMemoryTypeDevice && a.device == c->device;
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

bool grids_ok(int nev, const kt_grid* grids) {
  if (nev < 1 || !grids) return false;
  for (int e = 0; e < nev; ++e)
    if (grids[e].nx < 1 || grids[e].ny < 1 || grids[e].neta < 1) return false;
  return true;
}

// padded lattices of all events and the shared component stride
void layout(int nev, const kt_grid* grids, std::vector<Lattice>& lat, long long& gs, size_t& max_cells) {
  lat.resize(nev);
  long long off = 0;
  max_cells = 0;
  for (int e = 0; e < nev; ++e) {
    Lattice& L = lat[e];
    L.nx = grids[e].nx; L.ny = grids[e].ny; L.nz = grids[e].neta;
    L.pitch = (int)align_up((size_t)L.nx + 4, 4);
    L.NY = L.ny + 4;
    L.NZ = L.nz + 4;
    L.plane = (long long)L.pitch * L.NY;
    L.base = off;
    off += (long long)align_up((size_t)(L.plane * L.NZ), 32);
    max_cells = std::max(max_cells, (size_t)L.nx * L.ny * L.nz);
  }
  gs = off;
  for (auto& L : lat) L.fstride = gs;
}

// first element after event e's lattice
long long end_of(const std::vector<Lattice>& lat, long long gs, size_t e) {
  return (e + 1 < lat.size()) ? lat[e + 1].base : gs;
}

// the events in as few runs of less than kSpanElements as their order allows (almost always one); false if
// an event alone is larger
bool make_spans(const std::vector<Lattice>& lat, long long gs, std::vector<Span>& spans) {
  spans.clear();
  for (size_t e = 0; e < lat.size(); ++e) {
    if (end_of(lat, gs, e) - lat[e].base >= kSpanElements) return false;
    if (spans.empty() || end_of(lat, gs, e) - spans.back().base >= kSpanElements)
      spans.push_back(Span{(int)e, (int)e, lat[e].base, 0, 0});
    spans.back().ev1 = (int)e + 1;
  }
  return true;
}

long long tiles_of(const Lattice& L, const Shape& s) {
  return (long long)((L.nx + s.x - 1) / s.x) * ((L.ny + s.y - 1) / s.y) * ((L.nz + s.z - 1) / s.z);
}
int tiles_for(const std::vector<Lattice>& lat, const Shape& s) {
  long long n = 0;
  for (const auto& L : lat) n += tiles_of(L, s);
  return (int)n;
}

// the FP64 stage's blocks: 32 consecutive cells of an event each
long long strips_of(const Lattice& L) { return ((long long)L.nx * L.ny * L.nz + 31) / 32; }
long long strips_for(const std::vector<Lattice>& lat) {
  long long n = 0;
  for (const auto& L : lat) n += strips_of(L);
  return n;
}

// entries of the work table: the tiles of the shape with most of them (mixed precision), or the
// strips of a batch (FP64; a single event needs no table)
long long table_entries(const std::vector<Lattice>& lat, int mixed) {
  if (!mixed) return lat.size() > 1 ? strips_for(lat) : 1;
  int n = 0;
  for (const auto& s : kShapes) n = std::max(n, tiles_for(lat, s));
  return n;
}

void build_tiles(const std::vector<Lattice>& lat, const Shape& s, std::vector<Tile>& out) {
  out.clear();
  for (int e = 0; e < (int)lat.size(); ++e) {
    const Lattice& L = lat[e];
    // eta fastest: a block of a persistent grid walks a contiguous run of tiles up an eta column
    for (int j = 0; j < L.ny; j += s.y)
      for (int i = 0; i < L.nx; i += s.x)
        for (int k = 0; k < L.nz; k += s.z) out.push_back(Tile{e, i, j, k});
  }
}

size_t state_bytes(const std::vector<Lattice>& lat, long long gs, size_t max_cells, int mixed, int eos_n) {
  const size_t fs = (size_t)gs;
  const size_t es = mixed ? 4 : 8;
  size_t b = 0;
  b += align_up(30 * fs * 8, 256);             // q, qs
  if (mixed) b += align_up(30 * fs * 4, 256);  // FP32 copies of q, qs
  b += align_up(12 * fs * es, 256);            // U[3]
  b += align_up(4 * fs * es, 256);             // E[2], P[2]
  b += align_up(18 * max_cells * 8, 256);      // staging
  b += align_up((size_t)(eos_n > 0 ? eos_n : 1) * sizeof(EosSeg<double>), 256);
  b += align_up((size_t)(eos_n > 0 ? eos_n : 1) * sizeof(RootSeg), 256);
  b += align_up((size_t)(eos_n > 0 ? eos_n : 1) * sizeof(RootSegM), 256);
  b += align_up((size_t)(eos_n > 0 ? eos_n : 1) * sizeof(FaceSeg), 256);
  b += align_up((size_t)(eos_n > 0 ? eos_n : 1) * sizeof(SourceSeg), 256);
  b += 256;                                    // tau
  b += 256;                                    // stats
  b += align_up(KT_MLP_NPARAM * 4, 256);       // MLP weights
  b += align_up(KT_MLP_PACKED_BYTES, 256);     // packed MLP weights
  b += align_up(lat.size() * sizeof(Lattice), 256);
  b += align_up((size_t)table_entries(lat, mixed) * sizeof(Tile), 256);
  if (mixed) b += align_up(2 * lat.size() * sizeof(CUtensorMap), 256);
  if (mixed) b += align_up(kUpdMaps * lat.size() * sizeof(CUtensorMap), 256);
  b += align_up(fs * 4, 256);                  // regulation factors
  b += align_up(fs * 4, 256);                  // network outputs (learned start)
  return b;
}

void coef_from(Coef& d, const kt_coef* s) {
  d.kind = s ? s->kind : KT_COEF_CONST;
  d.c0 = s ? s->c0 : 0.0;
  d.c1 = s ? s->c1 : 0.0;
  d.c2 = s ? s->c2 : 1.0;
  d.ln_c0 = (d.c0 > 0.0) ? std::log(d.c0) : -INFINITY;
}

template <typename R>
void fill_pr(PR<R>& o, const Params& P) {
  o.inv_d[0] = (R)(1.0 / P.dx);
  o.inv_d[1] = (R)(1.0 / P.dy);
  o.inv_d[2] = (R)(1.0 / P.deta);
  o.half_inv_d[0] = (R)(0.5 / P.dx);
  o.half_inv_d[1] = (R)(0.5 / P.dy);
  o.half_inv_d[2] = (R)(0.5 / P.deta);
  o.theta = (R)P.theta;
  o.inv_dtau = (R)(1.0 / P.dtau);
  o.dtau = (R)P.dtau;
  o.half_dtau = (R)(0.5 * P.dtau);
  o.rate_max = (R)P.rate_max;
  o.tpp = (R)P.tpp;
  o.inv_rho_max = (R)(1.0 / P.rho_max);
  o.inv_xi0_rho_max = (R)(1.0 / (P.xi0 * P.rho_max));
  o.eos_a = (R)P.eos_a;
  o.eta_c0 = (R)P.eta.c0; o.eta_c1 = (R)P.eta.c1; o.eta_inv_c2 = (R)(1.0 / P.eta.c2); o.eta_ln_c0 = (R)P.eta.ln_c0;
  o.eta_inv_c1 = (R)(1.0 / P.eta.c1);
  o.eta_inv_5c0 = (R)(1.0 / (5.0 * P.eta.c0));
  o.zeta_c0 = (R)P.zeta.c0; o.zeta_c1 = (R)P.zeta.c1; o.zeta_inv_c2 = (R)(1.0 / P.zeta.c2);
  o.zeta_ln_c0 = (R)P.zeta.ln_c0; o.zeta_inv_c1 = (R)(1.0 / P.zeta.c1);
}

// Per-interval cubic coefficients of the table EOS (see kt_eos in kt.h).
template <typename R>
void build_segments(const kt_eos* eos, std::vector<EosSeg<R>>& out) {
  int n = eos->n;
  out.resize(n);
  for (int i = 0; i + 1 < n; ++i) {
    double e0 = eos->e[i], e1 = eos->e[i + 1];
    double de = e1 - e0;
    double P0 = eos->p[i], P1 = eos->p[i + 1];
    double m0 = eos->cs2[i] * de, m1 = eos->cs2[i + 1] * de;
    double T0 = eos->T[i], T1 = eos->T[i + 1];
    double s0 = eos->cs2[i] * T0 / (e0 + P0) * de, s1 = eos->cs2[i + 1] * T1 / (e1 + P1) * de;
    EosSeg<R> s;
    s.e0 = (R)e0; s.inv_de = (R)(1.0 / de);
    s.P0 = (R)P0; s.mP = (R)m0; s.cP2 = (R)(3.0 * (P1 - P0) - 2.0 * m0 - m1); s.cP3 = (R)(2.0 * (P0 - P1) + m0 + m1);
    s.T0 = (R)T0; s.mT = (R)s0; s.cT2 = (R)(3.0 * (T1 - T0) - 2.0 * s0 - s1); s.cT3 = (R)(2.0 * (T0 - T1) + s0 + s1);
    s.l0 = (R)eos->lndelta[i]; s.dl = (R)(eos->lndelta[i + 1] - eos->lndelta[i]);
    const double c2 = 3.0 * (P1 - P0) - 2.0 * m0 - m1, c3 = 2.0 * (P0 - P1) + m0 + m1;
    s.a1 = (R)(m0 / de); s.a2 = (R)(c2 / (de * de)); s.a3 = (R)(c3 / (de * de * de));
    out[i] = s;
  }
  out[n - 1] = out[n - 2];
  out[n - 1].e0 = (R)eos->e[n - 1];  // sentinel: only its e0 is read by the interval search
}

// The root-find's records (RootSeg) from the FP64 and FP32 segments.
void build_root_segments(const std::vector<EosSeg<double>>& sd, const std::vector<EosSeg<float>>& sf,
                         std::vector<RootSeg>& out) {
  const int n = (int)sd.size();
  out.resize(n);
  for (int i = 0; i < n; ++i) {
    RootSeg r;
    r.e0 = sd[i].e0;
    r.e1 = (i + 2 < n) ? sd[i + 1].e0 : INFINITY;  // the last interval (n - 2) and the sentinel are open
    r.P0 = sd[i].P0;
    r.a1 = sd[i].a1;
    r.a2 = sd[i].a2;
    r.a3 = sd[i].a3;
    const float two = 2.f, three = 3.f;
    r.b1 = sf[i].a1;
    r.b2 = two * sf[i].a2;
    r.b3 = three * sf[i].a3;
    r.unused = 0.f;
    out[i] = r;
  }
}

// The mixed-precision root-find's records: the FP64 ones with a2, a3 rounded to single precision.
void build_mixed_root_segments(const std::vector<RootSeg>& sr, std::vector<RootSegM>& out) {
  out.resize(sr.size());
  for (size_t i = 0; i < sr.size(); ++i) {
    const RootSeg& r = sr[i];
    RootSegM m;
    m.e0 = r.e0;
    m.e1 = r.e1;
    m.P0 = r.P0;
    m.a1 = r.a1;
    m.a2 = (float)r.a2;
    m.a3 = (float)r.a3;
    m.b1 = r.b1;
    m.b2 = r.b2;
    m.b3 = r.b3;
    m.unused0 = m.unused1 = m.unused2 = 0.f;
    out[i] = m;
  }
}

// ------------------------------------------------------------------ small kernels
// The primaries of kt_set_state: packed physical arrays on the device, null where not given
struct Primaries {
  const double *e, *u, *pi, *Pi, *u_prev;
};

// padded coordinates of physical cell o (x fastest)
__device__ __forceinline__ void cell_coords(const Lattice& L, unsigned o, int& i, int& j, int& k) {
  const unsigned row = o / (unsigned)L.nx;
  i = (int)(o - row * (unsigned)L.nx) + 2;
  k = (int)(row / (unsigned)L.ny);
  j = (int)row - k * L.ny + 2;
  k += 2;
}

// Conserved variables from primaries (Eqs. Ttt, Tti) for one event, with its ghost copies; also tau.
// Bound by memory (18 values read, 30 to 43 written per cell) once it stays off the FP64 pipe: tests on
// bit patterns, conversions on the integer pipe, no division.  It reads the caller's device arrays
// themselves (host arrays come through the staging area).  With the gather below, set and get of a 128^3
// event on the device: six learned steps between them 7.13 -> 6.79 ms, six steps of a 16-event batch
// 26.5 -> 22.7 ms.  (An output into new host arrays is bound by the host's copies: no gain there.)
constexpr int kSetThreads = 128;
template <typename R>
__global__ void __launch_bounds__(kSetThreads, 4)
    set_state_kernel(const Params P, const Lattice L, const Primaries in, double tau, double g, double gp, TauSlot* slot,
                     double* q, float* qf, R* U, R* Up, R* E, R* Pb, float* reg, unsigned* status) {
  const unsigned ncp = (unsigned)L.nx * (unsigned)L.ny * (unsigned)L.nz;
  const unsigned o = blockIdx.x * kSetThreads + threadIdx.x;
  if (o == 0) *slot = tau_slot(tau, P.dtau, P.milne);
  if (o >= ncp) return;
  int i, j, k;
  cell_coords(L, o, i, j, k);
  const double e = in.e[o];
  double u4[4] = {1.0, 0.0, 0.0, 0.0}, up4[4], pi[10];
  if (in.u) {
#pragma unroll
    for (int m = 0; m < 3; ++m) u4[m + 1] = in.u[(size_t)m * ncp + o];
    u4[0] = sqrt(fma(g * u4[3], u4[3], fma(u4[2], u4[2], fma(u4[1], u4[1], 1.0))));
  }
#pragma unroll
  for (int m = 0; m < 10; ++m) pi[m] = in.pi ? in.pi[(size_t)m * ncp + o] : 0.0;
  const double Pi = in.Pi ? in.Pi[o] : 0.0;
#pragma unroll
  for (int m = 0; m < 4; ++m) up4[m] = u4[m];
  if (in.u_prev) {
#pragma unroll
    for (int m = 0; m < 3; ++m) up4[m + 1] = in.u_prev[(size_t)m * ncp + o];
    up4[0] = sqrt(fma(gp * up4[3], up4[3], fma(up4[2], up4[2], fma(up4[1], up4[1], 1.0))));
  }
  const double P0 = eos_P(P, e), Pt = P0 + Pi, w = (e + Pt) * u4[0];
  double qn[NQ];
  qn[0] = fma(w, u4[0], -Pt) + pi[0];
#pragma unroll
  for (int m = 1; m < 4; ++m) qn[m] = fma(w, u4[m], pi[m]);
#pragma unroll
  for (int m = 0; m < 10; ++m) qn[4 + m] = pi[m];
  qn[14] = Pi;
  // non-finite input, or e < 0 (the sign bit of a non-zero e)
  const long long be = __double_as_longlong(e);
  bool bad = !kt::finite(e) || (be < 0 && (be << 1) != 0) || !kt::finite(u4[0]) || !kt::finite(Pi) || !kt::finite(up4[0]);
#pragma unroll
  for (int m = 0; m < 10; ++m) bad |= !kt::finite(pi[m]);
  if (bad) atomicOr(status, ST_NONFINITE);
  // the inversion of Eq. (eInferred) needs E = T^{tau tau} - pi^{tau tau} > 0 and M^2 < E^2 with
  // M^i = T^{tau i} - pi^{tau i}, M^2 = M_x^2 + M_y^2 + g_{eta eta} M_eta^2 (Sec. 2.4)
  // Decided in single precision where that is certain: every operand below 2^60 and g above 2^-60 (in the
  // doubles' exponents: the truncated values say nothing beyond 2^128), E above 2^-60, M^2 < 0.99 E^2 and a
  // pi^{tau mu} no larger than E, so that the difference's rounding stays far inside the margin.
  const auto ex = [](double x) { return (unsigned)__double2hiint(x) & 0x7ff00000u; };
  unsigned top = ex(g);
#pragma unroll
  for (int m = 0; m < 8; ++m) top = max(top, ex(qn[m]));
  const bool in_range = top < ((1023u + 60u) << 20) && ex(g) >= ((1023u - 60u) << 20);
  const float Ef = d2f_trunc(qn[0]) - d2f_trunc(qn[4]), gf = d2f_trunc(g);
  const float mx = d2f_trunc(qn[1]) - d2f_trunc(qn[5]), my = d2f_trunc(qn[2]) - d2f_trunc(qn[6]),
              mn = d2f_trunc(qn[3]) - d2f_trunc(qn[7]);
  const bool sure = in_range && Ef > 0x1p-60f && fmaf(gf * mn, mn, fmaf(my, my, mx * mx)) < 0.99f * Ef * Ef &&
                    fabsf(d2f_trunc(qn[4])) < Ef && fabsf(d2f_trunc(qn[5])) < Ef && fabsf(d2f_trunc(qn[6])) < Ef &&
                    gf * d2f_trunc(qn[7]) * d2f_trunc(qn[7]) < Ef * Ef;
  if (!bad && !sure) {
    const double Ei = qn[0] - qn[4], Mx = qn[1] - qn[5], My = qn[2] - qn[6], Mn = qn[3] - qn[7];
    if (!(pos(Ei) && obits(Mx * Mx + My * My + g * Mn * Mn) < obits(Ei * Ei))) atomicOr(status, ST_INVERSION);
  }
  const long long fs = L.fstride;
  reg[L.idx(i, j, k)] = 1.f;  // no regulation recorded yet
  // The stored precision.  FP32: to nearest by d2f_bits, which flushes results below the smallest normal float;
  // a cell that has one (the smallest non-zero magnitude says so: its upper word - 1, so that zeros are
  // largest) converts again by the instruction (FP64 pipe).  A branch per value instead of the one per cell:
  // 335 against 262 us for kt_set_state of 128^3 cells.
  float qs[NQ];
  R ur[4], upr[4], er, pr0;
  unsigned least = 0xffffffffu;
  auto convert = [&](auto&& to) {
    if (qf) {
#pragma unroll
      for (int n = 0; n < NQ; ++n) qs[n] = to(qn[n]);
    }
    if constexpr (sizeof(R) == 4) {
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        ur[m] = to(u4[m]);
        upr[m] = to(up4[m]);
      }
      er = to(e);
      pr0 = to(P0);
    }
  };
  convert([&](double x) {
    least = min(least, ((unsigned)__double2hiint(x) & 0x7fffffffu) - 1u);
    return d2f_bits(x);
  });
  if (least < (897u << 20) - 1u) convert([](double x) { return (float)x; });
  if constexpr (sizeof(R) == 8) {
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      ur[m] = u4[m];
      upr[m] = up4[m];
    }
    er = e;
    pr0 = P0;
  }
  for_cell_and_ghosts(P, L, L.idx(i, j, k), i, j, k, [&](long long c) {
#pragma unroll
    for (int n = 0; n < NQ; ++n) q[n * fs + c] = qn[n];
    if (qf) {
#pragma unroll
      for (int n = 0; n < NQ; ++n) qf[n * fs + c] = qs[n];
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      U[m * fs + c] = ur[m];
      Up[m * fs + c] = upr[m];
    }
    E[c] = er;
    Pb[c] = pr0;
  });
}

// float -> double, exact for every float: on the integer pipe, the conversion instruction (FP64 pipe)
// for subnormals, infinities and NaN only
__device__ __forceinline__ double f2d_exact(float f) {
  const unsigned ex = (__float_as_uint(f) >> 23) & 0xffu;
  if (ex == 0xffu || (ex == 0u && f != 0.f)) return (double)f;
  return f2d_bits(f);
}

// Rows of one event (double or float fields) gathered into packed physical arrays: one launch for up to
// kRows rows, kRowsPerThread of them per thread (blockIdx.y picks the group), their loads in flight
// together; the destination is the caller's device array itself or the staging area of a copy.
constexpr int kRows = 18, kRowsPerThread = 6;
struct GatherRows {
  const void* src[kRows];
  double* dst[kRows];
  unsigned f32;  // bit r: row r is float
  int n;
};
__global__ void __launch_bounds__(256) gather_kernel(const Lattice L, const GatherRows rows) {
  const unsigned ncp = (unsigned)L.nx * (unsigned)L.ny * (unsigned)L.nz;
  const unsigned o = blockIdx.x * 256u + threadIdx.x;
  if (o >= ncp) return;
  int i, j, k;
  cell_coords(L, o, i, j, k);
  const long long c = L.idx(i, j, k);
  const int r0 = kRowsPerThread * (int)blockIdx.y;
  double v[kRowsPerThread];
  float f[kRowsPerThread];
#pragma unroll
  for (int r = 0; r < kRowsPerThread; ++r) {
    if (r0 + r >= rows.n) break;
    if ((rows.f32 >> (r0 + r)) & 1u) f[r] = __ldg((const float*)rows.src[r0 + r] + c);
    else v[r] = __ldg((const double*)rows.src[r0 + r] + c);
  }
#pragma unroll
  for (int r = 0; r < kRowsPerThread; ++r) {
    if (r0 + r >= rows.n) break;
    rows.dst[r0 + r][o] = ((rows.f32 >> (r0 + r)) & 1u) ? f2d_exact(f[r]) : v[r];
  }
}

// scatter one packed physical array into a field (double or float) at every physical cell and
// the ghost copies it owns (checkpoint restore; float fields round to nearest, which is exact
// for values that were float to begin with)
template <typename S>
__global__ void scatter_kernel(const Params P, const Lattice L, const double* __restrict__ in, S* f) {
  long long ncp = (long long)L.nx * L.ny * L.nz;
  long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= ncp) return;
  int i = (int)(o % L.nx), j = (int)((o / L.nx) % L.ny), k = (int)(o / ((long long)L.nx * L.ny));
  const S v = (S)in[o];
  for_cell_and_ghosts(P, L, L.idx(i + 2, j + 2, k + 2), i + 2, j + 2, k + 2, [&](long long t) { f[t] = v; });
}

// smallest and largest e and smallest regulation factor over one event's physical cells (all
// positive, so their float bit patterns order like the values): out[0] min e, [1] max e, [2] min f
template <typename R>
__global__ void state_extrema_kernel(const Lattice L, const R* __restrict__ e, const float* __restrict__ reg,
                                     unsigned* out) {
  const long long ncp = (long long)L.nx * L.ny * L.nz;
  unsigned lo = 0x7f800000u, hi = 0u, rl = 0x7f800000u;
  for (long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x; o < ncp; o += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(o % L.nx), j = (int)((o / L.nx) % L.ny), k = (int)(o / ((long long)L.nx * L.ny));
    const long long c = L.idx(i + 2, j + 2, k + 2);
    const unsigned b = __float_as_uint(fmaxf(to_f32(e[c]), 0.f));
    lo = min(lo, b);
    hi = max(hi, b);
    rl = min(rl, __float_as_uint(fmaxf(reg[c], 0.f)));
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  rl = __reduce_min_sync(0xffffffffu, rl);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(out, lo);
    atomicMax(out + 1, hi);
    atomicMin(out + 2, rl);
  }
}

// self-test of the integer-pipe double -> float conversions (rounded and truncating)
__global__ void cvt_selftest_kernel(const double* __restrict__ x, float* rn, float* rz, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    rn[i] = d2f_bits(x[i]);
    rz[i] = d2f_trunc(x[i]);
  }
}

// self-test of the FP64 division of the stencil (vdiv) on caller-given operands
__global__ void div_selftest_kernel(const double* __restrict__ a, const double* __restrict__ b, double* q,
                                    long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) q[i] = vdiv(a[i], b[i]);
}

// Self-test of the bounded waits: every thread waits on an mbarrier that nothing arms, with the
// given poll limit, exactly as the stage kernels wait for their TMA copies; the block records
// ST_TIMEOUT and returns.
__global__ void wait_selftest_kernel(unsigned polls, unsigned* status) {
  __shared__ alignas(8) uint64_t bar;
  if (threadIdx.x == 0) {
    kt::mbar_init(&bar, 1);
    kt::fence_barrier_init();
  }
  __syncthreads();
  const bool ok = kt::mbar_wait(&bar, 0u, polls);
  if (__syncthreads_or(!ok) && threadIdx.x == 0) atomicOr(status, ST_TIMEOUT);
}

// validity diagnostics of Sec. 7 at the current state of one event (kt_get_diagnostics): the
// stage-1 right-hand side's kinematics and coefficients, evaluated per physical cell into the
// packed output [7][cells], the last column the recorded regulation factor
template <typename R>
__global__ void diag_kernel(const Params P, const Lattice L, const StageIO<R> io, double tau, const float* reg,
                            double* out) {
  const long long ncp = (long long)L.nx * L.ny * L.nz;
  const long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= ncp) return;
  const int i = (int)(o % L.nx), j = (int)((o / L.nx) % L.ny), k = (int)(o / ((long long)L.nx * L.ny));
  const Idx<R> c = cell_idx<R>(L, i + 2, j + 2, k + 2);
  const CellGeom<R> G = cell_geom<R>(P, tau);
  R dq[NQ], du[4][4], dv, dg[6];
  float amax = 0.f;
  Faces<R> Fx, Fy, Fz;
  R uc[4];
  cell_faces<R, false, false>(P, L, io, c, u_global(L, io, c), G, dq, uc, du, dv, amax, Fx, Fy, Fz);
  cell_sources<R, true>(P, L, io, c, G, uc, du, dv, dq, dg);
  for (int m = 0; m < 6; ++m) {
    if constexpr (sizeof(R) == 4) out[m * ncp + o] = f2d_exact(dg[m]);  // a quotient may be infinite
    else out[m * ncp + o] = dg[m];
  }
  out[6 * ncp + o] = f2d_bits(reg[c]);  // (finite)
}

// training samples of the learned start: features as the stage kernel forms them, the exact
// FP64 root and the target 10 ln(e / e_conf)
__global__ void mlp_features_kernel(const Params P, const Lattice L, const double* __restrict__ q,
                                    const float* __restrict__ qf, int pi32, double tau, long long n,
                                    const long long* __restrict__ cells, float* X, float* Y, double* Eexact,
                                    unsigned* status) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const long long ncp = (long long)L.nx * L.ny * L.nz;
  const long long o = cells[s];
  if (o < 0 || o >= ncp) {
    atomicOr(status, ST_INVERSION);
    return;
  }
  const int i = (int)(o % L.nx), j = (int)((o / L.nx) % L.ny), k = (int)(o / ((long long)L.nx * L.ny));
  const long long c = L.idx(i + 2, j + 2, k + 2);
  double qn[NQ];
  for (int m = 0; m < NQ; ++m) qn[m] = (pi32 && m >= 4) ? (double)qf[m * L.fstride + c] : q[m * L.fstride + c];
  const float Ef = d2f_bits(qn[0] - qn[4]);
  const double Mx = qn[1] - qn[5], My = qn[2] - qn[6], Mn = qn[3] - qn[7];
  const double g = P.milne ? tau * tau : 1.0;
  const float M2f = d2f_bits(fma(Mx, Mx, fma(My, My, g * Mn * Mn)));
  float x[MLP_IN], ecE;
  mlp_features(fmaxf(Ef, 1e-30f), M2f, d2f_bits(qn[14]), x, ecE);
  double e, P0, uo[4];
  unsigned it = 0;
  const unsigned st = invert_fp64(P, tau, qn, qn[0] - qn[4], e, P0, uo, it);
  if (st) atomicOr(status, st);
  for (int m = 0; m < MLP_IN; ++m) X[s * MLP_IN + m] = x[m];
  Y[s] = (float)(10.0 * log(e / ((double)Ef * (double)ecE)));
  Eexact[s] = e;
}

// ------------------------------------------------------------------ launches
template <typename R>
StageIO<R> make_io(Ctx* c, int stage) {
  StageIO<R> io;
  R* U0 = (R*)c->U[c->cur];
  R* Uprev = (R*)c->U[c->prev];
  R* Usp = (R*)c->U[c->spare];
  if (stage == 1) {
    io.q_in = c->q; io.q_base = nullptr; io.q_out = c->qs;
    io.u_in = U0; io.u_prev = Uprev; io.u_out = Uprev;        // u^* over u^{n-1}
    io.e_in = (R*)c->E[0]; io.p_in = (R*)c->Pb[0];
    io.e_out = (R*)c->E[1]; io.p_out = (R*)c->Pb[1];
  } else {
    io.q_in = c->qs; io.q_base = c->q; io.q_out = c->q;       // q^{n+1} over q^n
    io.u_in = Uprev; io.u_prev = U0; io.u_out = Usp;          // u^{n+1} into the spare buffer
    io.e_in = (R*)c->E[1]; io.p_in = (R*)c->Pb[1];
    io.e_out = (R*)c->E[0]; io.p_out = (R*)c->Pb[0];
  }
  if constexpr (sizeof(R) == 4) {
    io.qr_in = (stage == 1) ? c->qf : c->qsf;
    io.qr_out = (stage == 1) ? c->qsf : c->qf;
    // Six components that nothing else holds while a stage's faces are in use: k_2 in the first stage, the
    // FP32 copy of q^n in the second (its update writes q^{n+1} there, ghosts included); with FP32 pi
    // storage, which reads that copy there, the FP64 pi and Pi that it does not use.
    io.fv = !c->P.iface_invert ? nullptr
            : c->pi32          ? (const R*)(c->q + 4 * c->gs)
            : (stage == 1)     ? (const R*)((float*)c->qs + 15 * c->gs)
                               : (const R*)c->qf;
  } else {
    io.qr_in = (const R*)io.q_in;
    io.qr_out = nullptr;
    io.fv = nullptr;
  }
  io.tau = c->d_tau + c->cur;
  io.tau_next = (stage == 2) ? c->d_tau + c->spare : nullptr;  // the next step's u^n buffer and tau slot
  io.status = c->d_stat;
  io.max_speed_bits = c->d_stat + 1;
  io.counters = (unsigned long long*)(c->d_stat + 4);
  io.mlp_packed = c->learned ? c->d_mlp_packed : nullptr;
  io.reg_out = (stage == 2) ? c->reg : nullptr;
  return io;
}

// the same fields from element `off` of every component on
template <typename R>
StageIO<R> from(StageIO<R> io, long long off) {
  auto move = [&](auto& p) { if (p) p += off; };
  move(io.q_in); move(io.q_base); move(io.q_out); move(io.qr_in); move(io.qr_out);
  move(io.u_in); move(io.u_prev); move(io.u_out);
  move(io.e_in); move(io.p_in); move(io.e_out); move(io.p_out);
  move(io.reg_out); move(io.fv);
  return io;
}
UpdIO from(UpdIO u, long long off) {
  auto move = [&](auto& p) { if (p) p += off; };
  move(u.q); move(u.qf_n); move(u.qsf); move(u.k1); move(u.k2); move(u.qr_out);
  move(u.u_out); move(u.e_out); move(u.p_out); move(u.e_guess); move(u.reg_out); move(u.z_net);
  return u;
}

// Mixed precision: the Runge-Kutta increments k_1, k_2 (FP32, 15 components each) live in the
// memory of the FP64 q* array, which that path never stores.
float* k_buf(Ctx* c, int stage) { return (float*)c->qs + (stage == 1 ? 0 : 15 * c->gs); }

UpdIO make_uio(Ctx* c, int stage) {
  UpdIO u;
  StageIO<float> io = make_io<float>(c, stage);
  u.q = c->q;
  u.qf_n = c->qf;
  u.qsf = c->qsf;
  u.k1 = k_buf(c, 1);
  u.k2 = k_buf(c, 2);
  u.qr_out = io.qr_out;
  u.u_out = io.u_out;
  u.e_out = io.e_out;
  u.p_out = io.p_out;
  u.e_guess = io.e_in;
  u.tau = io.tau;
  u.tau_next = io.tau_next;
  u.status = c->d_stat;
  u.counters = (unsigned long long*)(c->d_stat + 4);
  u.reg_out = io.reg_out;
  u.z_net = c->z_net;
  return u;
}

template <int STAGE>
void launch_stage(Ctx* c, const StageIO<double>& io) {
  const bool t1 = (c->P.theta == 1.0), inv = c->P.iface_invert;
  auto go = [&](auto kernel) {
    kernel<<<c->grid_blocks, 32, 0, c->stream>>>(c->P, io, c->lat[0], c->d_lat, c->d_tiles, c->nev);
  };
  if (c->team) {
    auto team = [&](auto kernel) {
      kernel<<<c->grid_blocks, 128, 0, c->stream>>>(c->P, io, c->lat[0], c->d_lat, c->d_tiles, c->nev);
    };
    if (t1) team(stage_team_kernel<double, STAGE, true>);
    else team(stage_team_kernel<double, STAGE, false>);
    return;
  }
  if (t1 && !inv) go(stage_kernel<double, STAGE, true, false>);
  else if (!inv) go(stage_kernel<double, STAGE, false, false>);
  else if (t1) go(stage_kernel<double, STAGE, true, true>);
  else go(stage_kernel<double, STAGE, false, true>);
}

Work make_work(Ctx* c, const Span& sp) {
  const Shape& s = kShapes[c->shape];
  Work w;
  w.L0 = c->lat[sp.ev0];
  w.L0.base = 0;
  w.tk = (unsigned)((w.L0.nz + s.z - 1) / s.z);
  w.ti = (unsigned)((w.L0.nx + s.x - 1) / s.x);
  w.ntiles = sp.ntiles;
  w.lats = c->d_lat;
  w.tiles = c->d_tiles + sp.tile0;
  return w;
}

// f(integral constants...) with every run-time flag as a template argument
template <typename F>
void with_flags(F&& f) { f(); }
template <typename F, typename... B>
void with_flags(F&& f, bool b, B... rest) {
  if (b) with_flags([&](auto... r) { f(std::true_type{}, r...); }, rest...);
  else with_flags([&](auto... r) { f(std::false_type{}, r...); }, rest...);
}

// the right-hand-side kernel of a stage, with the minmod specialised when theta = 1
template <int STAGE>
void launch_rhs(Ctx* c, const StageIO<float>& io) {
  const Shape& s = kShapes[c->shape];
  if (c->P.iface_invert) {
    unsigned faces = 1;  // of the event and direction with the most
    for (const Lattice& L : c->lat)
      for (int d = 0; d < 3; ++d)
        faces = std::max(faces, (unsigned)(L.nx + (d == 0)) * (unsigned)(L.ny + (d == 1)) * (unsigned)(L.nz + (d == 2)));
    for (const Span& sp : c->spans) {
      const int n = sp.ev1 - sp.ev0;
      const dim3 grid((faces + kt::kFaceThreads - 1) / kt::kFaceThreads, 3, (unsigned)std::min(n, 65535));
      with_flags([&](auto t1) {
        kt::face_velocity_kernel<t1.value><<<grid, kt::kFaceThreads, 0, c->stream>>>(
            c->P, io.qr_in + sp.base, io.e_in + sp.base, io.tau, STAGE, c->d_lat + sp.ev0, n, (float*)io.fv + sp.base);
      }, c->P.theta == 1.0);
    }
  }
  const CUtensorMap* maps = c->d_tmaps + (STAGE == 1 ? 0 : c->nev);
  for (const Span& sp : c->spans)
    with_flags([&](auto single, auto t1, auto inv, auto fixed) {
      constexpr int f = fixed.value ? 2 : 0;
      rhs_kernel<single.value, t1.value, inv.value, f, f>
          <<<std::min(c->grid_rhs, sp.ntiles), dim3(s.x, s.y, s.z), rhs_smem_bytes(s.x, s.y, s.z), c->stream>>>(
              c->P, from(io, sp.base), STAGE, k_buf(c, STAGE) + sp.base, make_work(c, sp), c->map0[STAGE - 1], maps);
    }, c->nev == 1, c->P.theta == 1.0, c->P.iface_invert != 0, s.y == 2 && s.z == 2);
}

// every rhs kernel may take the dynamic shared memory of the largest tile shape
int allow_rhs_smem(Ctx* c) {
  int bytes = 0;
  for (const auto& sh : kShapes) bytes = std::max(bytes, rhs_smem_bytes(sh.x, sh.y, sh.z));
  cudaError_t e = cudaSuccess;
  auto set = [&](const void* f) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  for (int f = 0; f < 16; ++f) {
    with_flags([&](auto a, auto b, auto d, auto fixed) {
      constexpr int x = fixed.value ? 2 : 0;
      set((const void*)rhs_kernel<a.value, b.value, d.value, x, x>);
      set((const void*)fused_kernel<a.value, 1, b.value, d.value, x, x>);
      set((const void*)fused_kernel<a.value, 2, b.value, d.value, x, x>);
    }, (f & 1) != 0, (f & 2) != 0, (f & 4) != 0, (f & 8) != 0);
  }
  if (e != cudaSuccess) return fail(c, KT_ERR_CUDA, "rhs shared memory: %s", cudaGetErrorString(e));
  bytes = 0;
  for (const auto& sh : kShapes) bytes = std::max(bytes, upd_smem_bytes(sh.x, sh.y, sh.z, 2));
  set((const void*)update_staged_kernel<1, true>);
  set((const void*)update_staged_kernel<1, false>);
  set((const void*)update_staged_kernel<2, true>);
  set((const void*)update_staged_kernel<2, false>);
  if (e != cudaSuccess) return fail(c, KT_ERR_CUDA, "update shared memory: %s", cudaGetErrorString(e));
  return KT_OK;
}

// the update kernel of a stage for the context's root-find start and pi storage
template <int STAGE>
void launch_update(Ctx* c, const UpdIO& uio) {
  const Shape& s = kShapes[c->shape];
  const dim3 blk(s.x, s.y, s.z);
  if (c->staged && !c->pi32) {
    const size_t sm = upd_smem_bytes(s.x, s.y, s.z, c->upd_nbuf);
    for (const Span& sp : c->spans)
      with_flags([&](auto learned) {
        update_staged_kernel<STAGE, learned.value><<<std::min(c->grid_upd, sp.ntiles), blk, sm, c->stream>>>(
            c->P, from(uio, sp.base), c->d_lat, c->d_tiles + sp.tile0, sp.ntiles, c->d_umaps, c->upd_nbuf);
      }, c->learned != 0);
    return;
  }
  for (const Span& sp : c->spans)
    with_flags([&](auto single, auto learned, auto pi32) {
      update_kernel<single.value, STAGE, learned.value, pi32.value>
          <<<std::min(c->grid_upd, sp.ntiles), blk, 0, c->stream>>>(c->P, from(uio, sp.base), make_work(c, sp));
    }, c->nev == 1, c->learned != 0, c->pi32 != 0);
}

// the fused stage kernel (right-hand side and update in one launch)
template <int STAGE>
void launch_fused(Ctx* c, const StageIO<float>& io, const UpdIO& uio) {
  const Shape& s = kShapes[c->shape];
  const CUtensorMap* maps = c->d_tmaps + (STAGE == 1 ? 0 : c->nev);
  for (const Span& sp : c->spans)
    with_flags([&](auto single, auto t1, auto learned, auto fixed) {
      constexpr int f = fixed.value ? 2 : 0;
      fused_kernel<single.value, STAGE, t1.value, learned.value, f, f>
          <<<std::min(c->grid_rhs, sp.ntiles), dim3(s.x, s.y, s.z), rhs_smem_bytes(s.x, s.y, s.z), c->stream>>>(
              c->P, from(io, sp.base), from(uio, sp.base), make_work(c, sp), c->map0[STAGE - 1], maps);
    }, c->nev == 1, c->P.theta == 1.0, c->learned != 0, s.y == 2 && s.z == 2);
}

template <int STAGE>
void launch_split_stage(Ctx* c, const StageIO<float>& io, const UpdIO& uio) {
  if (c->fused) {
    launch_fused<STAGE>(c, io, uio);
    return;
  }
  launch_rhs<STAGE>(c, io);
  launch_update<STAGE>(c, uio);
}

// ev (optional, kNumTimed + 1 events): recorded between the launches of one step, in the order
// learned start (the network's inference), stage-1 rhs (or fused stage 1), stage-1 update,
// stage-2 rhs (or fused stage 2), stage-2 update, tau advance (always empty: the second stage
// writes tau^{n+1}); intervals of launches a context
// does not make (the network without the learned start, the update launches of the FP64 path and
// of the fused layout) are empty.
constexpr int kNumTimed = 6;
void mark(Ctx* c, cudaEvent_t* ev, int i) {
  if (ev) cudaEventRecord(ev[i], c->stream);
}

// the learned start's network on the state at the start of the step (its FP32 copy)
void launch_mlp_start(Ctx* c) {
  kt::mlp_start_kernel<<<c->grid_mlp, 256, 0, c->stream>>>(c->qf, c->gs, c->d_tau + c->cur, c->P.milne,
                                                           c->d_mlp_packed, c->z_net);
}

template <typename R>
void launch_step_stages(Ctx* c, cudaEvent_t* ev) {
  mark(c, ev, 0);
  if constexpr (sizeof(R) == 4) {
    if (c->learned && c->P.mlp_infer) launch_mlp_start(c);
    mark(c, ev, 1);
    if (c->fused) {  // the fused launches take the right-hand-side slots; the update slots stay empty
      launch_fused<1>(c, make_io<float>(c, 1), make_uio(c, 1));
      mark(c, ev, 2);
      mark(c, ev, 3);
      launch_fused<2>(c, make_io<float>(c, 2), make_uio(c, 2));
      mark(c, ev, 4);
      mark(c, ev, 5);
      return;
    }
    launch_rhs<1>(c, make_io<float>(c, 1));
    mark(c, ev, 2);
    launch_update<1>(c, make_uio(c, 1));
    mark(c, ev, 3);
    launch_rhs<2>(c, make_io<float>(c, 2));
    mark(c, ev, 4);
    launch_update<2>(c, make_uio(c, 2));
    mark(c, ev, 5);
  } else {
    mark(c, ev, 1);
    launch_stage<1>(c, make_io<double>(c, 1));
    mark(c, ev, 2);
    mark(c, ev, 3);
    launch_stage<2>(c, make_io<double>(c, 2));
    mark(c, ev, 4);
    mark(c, ev, 5);
  }
}

// enqueue one full step (two stages; the second advances tau) for the current rotation phase, then rotate
int enqueue_step(Ctx* c, cudaEvent_t* ev = nullptr) {
  if (c->mixed) launch_step_stages<float>(c, ev);
  else launch_step_stages<double>(c, ev);
  mark(c, ev, 6);
  // u^{n-1} <- u^n, u^n <- u^{n+1}; the old u^{n-1} buffer (holding u^*) becomes the spare
  int ncur = c->spare, nprev = c->cur, nspare = c->prev;
  c->cur = ncur; c->prev = nprev; c->spare = nspare;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(c, KT_ERR_CUDA, "stage launch: %s", cudaGetErrorString(e));
  return KT_OK;
}

// persistent grid: as many blocks of kernel K as fit on the device at once
template <typename K>
int occupancy_blocks(K kernel, const Shape& s, size_t dyn_smem = 0) {
  int nb = 0, dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, s.x * s.y * s.z, dyn_smem);
  return std::max(1, nb) * std::max(1, sms);
}

// The TMA descriptors of the FP32 copies of q read by the mixed-precision stencil: per event a
// 4-d map (x: pitch, y: ny + 4, eta: neta + 4, component: 15) with the strides of the padded
// lattice, and a box of the tile plus its two-cell halo for kCompPerBox components,
// (bx + 4) x (by + 4) x (bz + 4) x kCompPerBox.
int encode_tensor_maps(Ctx* c) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn)
      return fail(c, KT_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
    encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
  }
  const Shape& s = kShapes[c->shape];
  if ((s.x + 4) * (s.y + 4) * (s.z + 4) > kBoxMax) return fail(c, KT_ERR_ARG, "tile box exceeds the staging buffer");
  std::vector<CUtensorMap> maps(2 * c->nev);
  for (int w = 0; w < 2; ++w)
    for (int e = 0; e < c->nev; ++e) {
      const Lattice& L = c->lat[e];
      float* base = (w == 0 ? c->qf : c->qsf) + L.base;
      cuuint64_t dims[4] = {(cuuint64_t)L.pitch, (cuuint64_t)L.NY, (cuuint64_t)L.NZ, (cuuint64_t)NQ};
      cuuint64_t strides[3] = {(cuuint64_t)L.pitch * 4, (cuuint64_t)L.plane * 4, (cuuint64_t)c->gs * 4};
      cuuint32_t box[4] = {(cuuint32_t)(s.x + 4), (cuuint32_t)(s.y + 4), (cuuint32_t)(s.z + 4), kCompPerBox};
      cuuint32_t estr[4] = {1, 1, 1, 1};
      CUresult r = encode(&maps[w * c->nev + e], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return fail(c, KT_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d) for event %d", (int)r, e);
    }
  c->map0[0] = maps[0];
  c->map0[1] = maps[c->nev];
  CK(cudaMemcpyAsync(c->d_tmaps, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice, c->stream));
  // the staged update's boxes: the tile's cells in y and eta, bx + 4 cells in x from the tile's
  // padded x, for q (FP64: 8 components, and 1), k_1, k_2 and the FP32 copy of q (15 components)
  std::vector<CUtensorMap> um(kUpdMaps * c->nev);
  for (int e = 0; e < c->nev; ++e) {
    const Lattice& L = c->lat[e];
    struct Src { void* base; CUtensorMapDataType t; int esz; cuuint32_t depth; };
    const Src src[kUpdMaps] = {{c->q + L.base, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 8, 8},
                               {c->q + L.base, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 8, 1},
                               {k_buf(c, 1) + L.base, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, NQ},
                               {k_buf(c, 2) + L.base, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, NQ},
                               {c->qf + L.base, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, NQ}};
    for (int w = 0; w < kUpdMaps; ++w) {
      const cuuint64_t es = (cuuint64_t)src[w].esz;
      cuuint64_t dims[4] = {(cuuint64_t)L.pitch, (cuuint64_t)L.NY, (cuuint64_t)L.NZ, (cuuint64_t)NQ};
      cuuint64_t strides[3] = {(cuuint64_t)L.pitch * es, (cuuint64_t)L.plane * es, (cuuint64_t)c->gs * es};
      cuuint32_t box[4] = {(cuuint32_t)(s.x + 4), (cuuint32_t)s.y, (cuuint32_t)s.z, src[w].depth};
      cuuint32_t estr[4] = {1, 1, 1, 1};
      CUresult r = encode(&um[kUpdMaps * e + w], src[w].t, 4, src[w].base, dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return fail(c, KT_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d), update map %d", (int)r, w);
    }
  }
  CK(cudaMemcpyAsync(c->d_umaps, um.data(), um.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice, c->stream));
  CK(cudaStreamSynchronize(c->stream));
  return KT_OK;
}

// The FP64 mode has one layout (see stage_kernel): blocks of 32 consecutive cells, whatever candidate
// is asked for.  Four warps share a strip while all blocks of stage_team_kernel are resident at once: three
// per SM (164 registers, 22 KB), 456 strips on 152 SMs.  One strip more is a second wave.  12 viscous steps
// (us), one warp / four warps per strip: 64 strips 1598 / 793, 304 strips 1600 / 1010, 456 strips 1623 / 1277,
// 464 strips 1637 / 2167, 608 strips 1692 / 2437.
int select_strips(Ctx* c, int cand) {
  c->grid_blocks = (int)strips_for(c->lat);
  c->team = !c->P.iface_invert && c->grid_blocks <= occupancy_blocks(stage_team_kernel<double, 2, false>, Shape{32, 4, 1});
  if (c->nev > 1 && c->ntiles == 0) {
    std::vector<Tile> strips;
    for (int e = 0; e < c->nev; ++e)
      for (long long s = 0; s < strips_of(c->lat[e]); ++s) strips.push_back(Tile{e, (int)(32 * s), 0, 0});
    CK(cudaMemcpyAsync(c->d_tiles, strips.data(), strips.size() * sizeof(Tile), cudaMemcpyHostToDevice, c->stream));
    CK(cudaStreamSynchronize(c->stream));
  }
  c->ntiles = c->grid_blocks;
  c->cand = cand;
  return KT_OK;
}

int select_shape(Ctx* c, int cand) {
  if (!c->mixed) return select_strips(c, cand);
  const int base = cand % kNumBase, shape = base / 2, one_per_tile = base % 2, variant = cand / kNumBase;
  const bool fusable = !c->pi32 && !c->P.iface_invert;
  c->staged = (variant == 1) && !c->pi32;
  c->fused = (variant == 2) && fusable;
  c->upd_nbuf = one_per_tile ? 1 : 2;
  std::vector<Tile> tiles;
  build_tiles(c->lat, kShapes[shape], tiles);
  if ((int)tiles.size() > c->max_tiles) return fail(c, KT_ERR_OOM, "tile table overflow");
  CK(cudaMemcpyAsync(c->d_tiles, tiles.data(), tiles.size() * sizeof(Tile), cudaMemcpyHostToDevice, c->stream));
  CK(cudaStreamSynchronize(c->stream));
  c->shape = shape;
  c->ntiles = (int)tiles.size();
  int at = 0;
  for (Span& sp : c->spans) {
    long long n = 0;
    for (int e = sp.ev0; e < sp.ev1; ++e) n += tiles_of(c->lat[e], kShapes[shape]);
    sp.tile0 = at;
    sp.ntiles = (int)n;
    at += sp.ntiles;
  }
  int rc = encode_tensor_maps(c);
  if (rc != KT_OK) return rc;
  const Shape& sh = kShapes[shape];
  auto grid = [&](int cap) { return one_per_tile ? c->ntiles : std::max(1, std::min(cap, c->ntiles)); };
  const size_t rsm = rhs_smem_bytes(sh.x, sh.y, sh.z);
  c->grid_rhs = grid(c->fused ? occupancy_blocks(fused_kernel<true, 1, true, true, 0, 0>, sh, rsm)
                              : occupancy_blocks(rhs_kernel<true, true, false, 0, 0>, sh, rsm));
  if (c->staged) {
    const size_t usm = upd_smem_bytes(sh.x, sh.y, sh.z, c->upd_nbuf);
    c->grid_upd = grid(c->learned ? occupancy_blocks(update_staged_kernel<2, true>, sh, usm)
                                  : occupancy_blocks(update_staged_kernel<2, false>, sh, usm));
  } else {
    c->grid_upd = grid(c->learned ? occupancy_blocks(update_kernel<true, 1, true, false>, sh)
                                  : occupancy_blocks(update_kernel<true, 1, false, false>, sh));
  }
  c->grid_blocks = c->grid_rhs;
  c->cand = cand;
  for (int p = 0; p < 3; ++p)
    if (c->graph[p]) { cudaGraphExecDestroy(c->graph[p]); c->graph[p] = nullptr; }
  return KT_OK;
}

// Autotuner: time first-stage launches for every candidate (tile shape, grid size, layout).  The
// launches write only scratch buffers (q*, its FP32 copy, e*, p*, and u* redirected to the spare
// buffer), so the state is untouched; the fastest candidate is kept.
int time_first_stage(Ctx* c, float* ms) {
  StageIO<float> io = make_io<float>(c, 1);
  io.u_out = (float*)c->U[c->spare];
  auto launch = [&]() {  // writes k_1, q*'s FP32 copy, e*, P*, u* (spare buffer)
    UpdIO u = make_uio(c, 1);
    u.u_out = (float*)c->U[c->spare];
    launch_split_stage<1>(c, io, u);
  };
  cudaEvent_t a, b;
  CK(cudaEventCreate(&a));
  CK(cudaEventCreate(&b));
  launch();  // warm-up
  for (int r = 0; r < 3; ++r) {  // the fastest of three timed launches (candidates differ by ~1%)
    CK(cudaEventRecord(a, c->stream));
    launch();
    CK(cudaEventRecord(b, c->stream));
    CK(cudaEventSynchronize(b));
    float t = 0.f;
    CK(cudaEventElapsedTime(&t, a, b));
    if (r == 0 || t < *ms) *ms = t;
  }
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  return KT_OK;
}

int autotune(Ctx* c) {
  Range range_("kt autotune");
  int best = 0;
  for (int s = 0; s < kNumCandidates; ++s) c->tune_ms[s] = 0.f;
  const bool fusable = !c->pi32 && !c->P.iface_invert;
  for (int s = 0; s < kNumCandidates; ++s) {
    if (!(s < kNumBase || (fusable && s >= kFusedFirst))) continue;
    int rc = select_shape(c, s);
    if (rc != KT_OK) return rc;
    float ms = 0.f;
    rc = time_first_stage(c, &ms);
    if (rc != KT_OK) return rc;
    c->tune_ms[s] = ms;
    if (ms < c->tune_ms[best]) best = s;
  }
  int rc = select_shape(c, best);
  if (rc != KT_OK) return rc;
  CK(cudaMemsetAsync(c->d_stat, 0, 256, c->stream));
  c->tuned = true;
  return KT_OK;
}

int build_graph(Ctx* c, int phase) {
  Range range_("kt capture step graph");
  int save[3] = {c->cur, c->prev, c->spare};
  cudaGraph_t gr;
  CK(cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
  int rc = KT_OK;
  for (int s = 0; s < 3 && rc == KT_OK; ++s) rc = enqueue_step(c);
  cudaError_t e = cudaStreamEndCapture(c->stream, &gr);
  c->cur = save[0]; c->prev = save[1]; c->spare = save[2];
  if (rc != KT_OK) return rc;
  if (e != cudaSuccess) return fail(c, KT_ERR_CUDA, "graph capture: %s", cudaGetErrorString(e));
  e = cudaGraphInstantiate(&c->graph[phase], gr, 0);
  cudaGraphDestroy(gr);
  if (e != cudaSuccess) return fail(c, KT_ERR_CUDA, "graph instantiate: %s", cudaGetErrorString(e));
  return KT_OK;
}

}  // namespace

struct kt_ctx : Ctx {};

// ==================================================================== C ABI
extern "C" {

int kt_options_default(kt_options* o) {
  if (!o) return KT_ERR_ARG;
  memset(o, 0, sizeof(*o));
  o->theta_limiter = 1.0;
  o->coords = KT_MILNE;
  o->bc = KT_BC_COPY;
  o->precision = KT_FP64;
  o->inversion = KT_INV_PLAIN;
  o->tau_pipi_on = 1;
  o->regulate = 1;
  o->rho_max = 1.0;
  o->xi0 = 0.1;
  o->e_min = 0.0;
  o->tau_relax_min = 0.0;
  o->use_graph = 1;
  o->autotune = 1;
  o->iface = KT_IFACE_RECON;
  return KT_OK;
}

int kt_state_bytes_batch(int n_events, const kt_grid* grids, const kt_eos* eos, const kt_options* opt,
                         size_t* bytes) {
  if (!bytes || !grids_ok(n_events, grids)) return KT_ERR_ARG;
  if (eos && eos->kind == KT_EOS_TABLE && eos->n < 4) return KT_ERR_EOS;
  kt_options d;
  kt_options_default(&d);
  const kt_options* o = opt ? opt : &d;
  std::vector<Lattice> lat;
  long long gs;
  size_t mc;
  layout(n_events, grids, lat, gs, mc);
  *bytes = state_bytes(lat, gs, mc, o->precision == KT_MIXED, (eos && eos->kind == KT_EOS_TABLE) ? eos->n : 0);
  return KT_OK;
}

int kt_state_bytes(const kt_grid* grid, const kt_eos* eos, const kt_options* opt, size_t* bytes) {
  return kt_state_bytes_batch(1, grid, eos, opt, bytes);
}

int kt_init_batch(kt_ctx** out, int n_events, const kt_grid* grids, double dx, double deta, double dtau,
                  const kt_eos* eos, const kt_coef* eta_over_s, const kt_coef* zeta_over_s, const kt_options* opt) {
  if (!out) return KT_ERR_ARG;
  *out = nullptr;
  kt_ctx* c = new (std::nothrow) kt_ctx();
  if (!c) return KT_ERR_OOM;
  auto bail = [&](int code) { kt_free(c); return code; };
  if (!grids_ok(n_events, grids) || !(dx > 0) || !(deta > 0) || !(dtau > 0) || !eos) {
    fprintf(stderr, "kt_init: invalid grid, spacing or eos\n");
    return bail(KT_ERR_ARG);
  }
  if (opt) c->opt = *opt; else kt_options_default(&c->opt);
  const kt_options& o = c->opt;
  if (o.precision != KT_FP64 && o.precision != KT_MIXED) return bail(KT_ERR_ARG);
  if (!(o.theta_limiter >= 1.0 && o.theta_limiter <= 2.0)) return bail(KT_ERR_ARG);
  if (o.coords != KT_MILNE && o.coords != KT_CARTESIAN) return bail(KT_ERR_ARG);
  if (o.bc != KT_BC_COPY && o.bc != KT_BC_PERIODIC) return bail(KT_ERR_ARG);
  if (o.inversion != KT_INV_PLAIN && o.inversion != KT_INV_LEARNED && o.inversion != KT_INV_CONFORMAL)
    return bail(KT_ERR_ARG);
  // the learned (and the conformal) start serves the mixed-precision path
  if (o.inversion == KT_INV_LEARNED && (!o.mlp_weights || o.precision != KT_MIXED)) return bail(KT_ERR_ARG);
  if (o.inversion == KT_INV_CONFORMAL && o.precision != KT_MIXED) return bail(KT_ERR_ARG);
  c->mixed = (o.precision == KT_MIXED);
  c->esz = c->mixed ? 4 : 8;
  c->learned = (o.inversion == KT_INV_LEARNED || o.inversion == KT_INV_CONFORMAL);
  if (o.pi_storage != KT_STORE_FP64 && o.pi_storage != KT_STORE_PI_FP32) return bail(KT_ERR_ARG);
  if (o.pi_storage == KT_STORE_PI_FP32 && o.precision != KT_MIXED) return bail(KT_ERR_ARG);
  c->pi32 = (o.pi_storage == KT_STORE_PI_FP32);
  c->nev = n_events;
  layout(n_events, grids, c->lat, c->gs, c->max_cells);
  if (c->mixed && !make_spans(c->lat, c->gs, c->spans)) {
    fprintf(stderr, "kt_init: an event of 2^29 or more padded cells in mixed precision\n");
    return bail(KT_ERR_ARG);
  }
  c->ev_set.assign(n_events, 0);

  Params& P = c->P;
  memset(&P, 0, sizeof(P));
  P.dx = dx; P.dy = dx; P.deta = deta; P.dtau = dtau;
  P.theta = o.theta_limiter;
  P.milne = (o.coords == KT_MILNE);
  P.periodic = (o.bc == KT_BC_PERIODIC);
  coef_from(P.eta, eta_over_s);
  coef_from(P.zeta, zeta_over_s);
  for (const Coef* k : {&P.eta, &P.zeta}) {
    const bool ok = (k->kind == KT_COEF_CONST && k->c0 >= 0.0) ||
                    (k->kind == KT_COEF_GAUSS && k->c0 >= 0.0 && k->c2 > 0.0) ||
                    (k->kind == KT_COEF_PAPER_ZETA && k->c0 >= 0.0 && k->c1 > 0.0);
    if (!ok) return bail(KT_ERR_ARG);
  }
  P.eos_table = (eos->kind == KT_EOS_TABLE);
  P.eos_a = eos->a;
  if (eos->kind == KT_EOS_TABLE) {
    if (eos->n < 4 || !eos->e || !eos->p || !eos->cs2 || !eos->T || !eos->lndelta) return bail(KT_ERR_EOS);
    for (int i = 0; i + 1 < eos->n; ++i)
      if (!(eos->e[i + 1] > eos->e[i]) || !(eos->e[i] > 0)) return bail(KT_ERR_EOS);
    P.eos_n = eos->n;
    P.lne0 = (float)std::log(eos->e[0]);
    P.inv_h = (float)((eos->n - 1) / (std::log(eos->e[eos->n - 1]) - std::log(eos->e[0])));
  } else if (eos->kind == KT_EOS_CONFORMAL) {
    if (!(eos->a > 0)) return bail(KT_ERR_EOS);
    P.eos_n = 0;
  } else {
    return bail(KT_ERR_EOS);
  }
  P.shear_on = !(P.eta.kind == KT_COEF_CONST && P.eta.c0 == 0.0);
  P.bulk_on = !(P.zeta.kind == KT_COEF_CONST && P.zeta.c0 == 0.0) && P.eos_table;
  P.tpp = o.tau_pipi_on ? 10.0 / 7.0 : 0.0;
  P.regulate = o.regulate;
  if (o.iface != KT_IFACE_RECON && o.iface != KT_IFACE_INVERT) return bail(KT_ERR_ARG);
  P.iface_invert = (o.iface == KT_IFACE_INVERT);
  P.mlp_infer = (o.inversion == KT_INV_LEARNED);
  P.rho_max = o.rho_max;
  P.xi0 = o.xi0;
  P.e_min = o.e_min;
  P.root_lo = (o.e_min > 0.0) ? o.e_min : 1e-300;
  P.rate_max = (o.tau_relax_min > 0) ? 1.0 / o.tau_relax_min : INFINITY;
  P.ln_rate_max = std::log(P.rate_max);
  fill_pr<double>(P.pd, P);
  fill_pr<float>(P.pf, P);

  int dev_count = 0;
  if (cudaGetDeviceCount(&dev_count) != cudaSuccess || dev_count < 1) {
    fail(c, KT_ERR_CUDA, "no CUDA device");
    fprintf(stderr, "kt_init: no CUDA device (libkt has no CPU fallback)\n");
    return bail(KT_ERR_CUDA);
  }
  // every call synchronises its stream before returning, so a context-owned stream is safe when
  // the caller passes none (the legacy default stream cannot be captured into a graph)
  c->stream = (cudaStream_t)o.stream;
  if (!c->stream) {
    if (cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) != cudaSuccess) {
      fail(c, KT_ERR_CUDA, "stream creation failed");
      return bail(KT_ERR_CUDA);
    }
    c->own_stream = true;
  }

  // ---- device memory, carved from one block
  size_t need = state_bytes(c->lat, c->gs, c->max_cells, c->mixed, P.eos_n);
  char* base;
  if (o.arena) {
    if (o.arena_bytes < need) return bail(KT_ERR_OOM);
    base = (char*)o.arena;
  } else {
    if (cudaMalloc(&c->base, need) != cudaSuccess) { cudaGetLastError(); return bail(KT_ERR_OOM); }
    base = (char*)c->base;
  }
  c->bytes = need;
  size_t off = 0;
  auto carve = [&](size_t b) { void* p = base + off; off += align_up(b, 256); return p; };
  const size_t fs = (size_t)c->gs;
  char* qq = (char*)carve(30 * fs * 8);
  c->q = (double*)qq;
  c->qs = (double*)(qq + 15 * fs * 8);
  if (c->mixed) {
    char* qqf = (char*)carve(30 * fs * 4);
    c->qf = (float*)qqf;
    c->qsf = (float*)(qqf + 15 * fs * 4);
    CK(cudaMemsetAsync(qqf, 0, 30 * fs * 4, c->stream));
  }
  char* uu = (char*)carve(12 * fs * c->esz);
  for (int b = 0; b < 3; ++b) c->U[b] = uu + (size_t)b * 4 * fs * c->esz;
  char* ep = (char*)carve(4 * fs * c->esz);
  c->E[0] = ep; c->E[1] = ep + fs * c->esz; c->Pb[0] = ep + 2 * fs * c->esz; c->Pb[1] = ep + 3 * fs * c->esz;
  c->stage = (double*)carve(18 * c->max_cells * 8);
  int nseg = P.eos_n > 0 ? P.eos_n : 1;
  c->seg_d = (EosSeg<double>*)carve(nseg * sizeof(EosSeg<double>));
  c->seg_r = (RootSeg*)carve(nseg * sizeof(RootSeg));
  c->seg_m = (RootSegM*)carve(nseg * sizeof(RootSegM));
  c->seg_face = (FaceSeg*)carve(nseg * sizeof(FaceSeg));
  c->seg_src = (SourceSeg*)carve(nseg * sizeof(SourceSeg));
  c->d_tau = (TauSlot*)carve(256);
  c->d_stat = (unsigned*)carve(256);
  c->d_mlp = (float*)carve(KT_MLP_NPARAM * 4);
  c->d_mlp_packed = (uint32_t*)carve(KT_MLP_PACKED_BYTES);
  c->d_lat = (Lattice*)carve(c->lat.size() * sizeof(Lattice));
  c->max_tiles = (int)table_entries(c->lat, c->mixed);
  c->d_tiles = (Tile*)carve((size_t)c->max_tiles * sizeof(Tile));
  if (c->mixed) c->d_tmaps = (CUtensorMap*)carve(2 * c->lat.size() * sizeof(CUtensorMap));
  if (c->mixed) c->d_umaps = (CUtensorMap*)carve(kUpdMaps * c->lat.size() * sizeof(CUtensorMap));
  c->reg = (float*)carve(fs * 4);
  c->z_net = (float*)carve(fs * 4);
  CK(cudaMemsetAsync(c->z_net, 0, fs * 4, c->stream));  // z = 0: the conformal start (no network)
  {
    int nb = 0, sms = 0;
    CK(cudaGetDevice(&c->device));
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device));
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kt::mlp_start_kernel, 256, 0));
    c->grid_mlp = (int)std::max(1LL, std::min((long long)std::max(1, nb) * sms, (long long)((fs + 255) / 256)));
  }
  P.seg_d = c->seg_d;
  P.seg_r = c->seg_r;
  P.seg_m = c->seg_m;
  P.seg_face = c->seg_face;
  P.seg_src = c->seg_src;

  CK(cudaMemsetAsync(qq, 0, 30 * fs * 8, c->stream));
  CK(cudaMemsetAsync(ep, 0, 4 * fs * c->esz, c->stream));
  {  // unused corner ghosts hold a fluid at rest (u^tau = 1); they are never read
    std::vector<unsigned char> one(fs * c->esz, 0);
    for (size_t i = 0; i < fs; ++i) {
      if (c->mixed) { float v = 1.f; memcpy(&one[i * 4], &v, 4); }
      else { double v = 1.0; memcpy(&one[i * 8], &v, 8); }
    }
    for (int b = 0; b < 3; ++b) {
      CK(cudaMemcpyAsync(c->U[b], one.data(), one.size(), cudaMemcpyHostToDevice, c->stream));
      CK(cudaMemsetAsync((char*)c->U[b] + fs * c->esz, 0, 3 * fs * c->esz, c->stream));
    }
    CK(cudaStreamSynchronize(c->stream));
  }
  if (P.eos_table) {
    std::vector<EosSeg<double>> sd;
    std::vector<EosSeg<float>> sf;
    build_segments<double>(eos, sd);
    build_segments<float>(eos, sf);
    std::vector<RootSeg> sr;
    build_root_segments(sd, sf, sr);
    std::vector<RootSegM> sm;
    build_mixed_root_segments(sr, sm);
    CK(cudaMemcpyAsync(c->seg_d, sd.data(), sd.size() * sizeof(sd[0]), cudaMemcpyHostToDevice, c->stream));
    CK(cudaMemcpyAsync(c->seg_r, sr.data(), sr.size() * sizeof(sr[0]), cudaMemcpyHostToDevice, c->stream));
    CK(cudaMemcpyAsync(c->seg_m, sm.data(), sm.size() * sizeof(sm[0]), cudaMemcpyHostToDevice, c->stream));
    std::vector<FaceSeg> sface(sr.size());
    for (size_t i = 0; i < sr.size(); ++i)
      sface[i] = FaceSeg{(float)sr[i].e0, (float)sr[i].e1, (float)sr[i].P0, (float)sr[i].a1,
                         (float)sr[i].a2, (float)sr[i].a3, 0.f,             0.f};
    std::vector<SourceSeg> ssrc(sf.size());
    for (size_t i = 0; i < sf.size(); ++i)
      ssrc[i] = SourceSeg{sf[i].e0, sf[i].inv_de, sf[i].l0, sf[i].dl, sf[i].T0, sf[i].mT, sf[i].cT2, sf[i].cT3};
    CK(cudaMemcpyAsync(c->seg_src, ssrc.data(), ssrc.size() * sizeof(SourceSeg), cudaMemcpyHostToDevice, c->stream));
    CK(cudaMemcpyAsync(c->seg_face, sface.data(), sface.size() * sizeof(FaceSeg), cudaMemcpyHostToDevice, c->stream));
  }
  if (o.mlp_weights) {
    CK(cudaMemcpyAsync(c->d_mlp, o.mlp_weights, KT_MLP_NPARAM * 4, cudaMemcpyHostToDevice, c->stream));
    kt::mlp_pack_kernel<<<1, 256, 0, c->stream>>>(c->d_mlp, c->d_mlp_packed);
    CK(cudaGetLastError());
  }
  std::vector<Lattice> dl = c->lat;  // mixed precision: from the start of each event's span
  for (const Span& sp : c->spans)
    for (int e = sp.ev0; e < sp.ev1; ++e) dl[e].base -= sp.base;
  CK(cudaMemcpyAsync(c->d_lat, dl.data(), dl.size() * sizeof(Lattice), cudaMemcpyHostToDevice, c->stream));
  CK(cudaMemsetAsync(c->d_stat, 0, 256, c->stream));
  CK(cudaStreamSynchronize(c->stream));
  int rc = c->mixed ? allow_rhs_smem(c) : KT_OK;
  if (rc == KT_OK) rc = select_shape(c, 0);
  if (rc != KT_OK) return bail(rc);
  *out = c;
  return KT_OK;
}

int kt_init(kt_ctx** out, const kt_grid* grid, double dx, double deta, double dtau, const kt_eos* eos,
            const kt_coef* eta_over_s, const kt_coef* zeta_over_s, const kt_options* opt) {
  return kt_init_batch(out, 1, grid, dx, deta, dtau, eos, eta_over_s, zeta_over_s, opt);
}

int kt_set_state_event(kt_ctx* c, int event, double tau, const double* e, const double* u, const double* pi,
                       const double* Pi, const double* u_prev, int on_device) {
  Range range_("kt_set_state");
  if (!c) return KT_ERR_ARG;
  if (event < 0 || event >= c->nev || !e || !(tau > 0 || !c->P.milne))
    return fail(c, KT_ERR_ARG, "kt_set_state: bad argument");
  const Lattice& L = c->lat[event];
  size_t ncp = (size_t)L.nx * L.ny * L.nz;
  Primaries in = {e, u, pi, Pi, u_prev};
  // what the kernel cannot read in place goes through the staging area: rows 0, 1-3, 4-13, 14, 15-17
  auto up = [&](const double*& p, int row, int rows) {
    if (!p || (on_device && in_place(c, p))) return cudaSuccess;
    double* s = c->stage + row * ncp;
    const cudaError_t r = cudaMemcpyAsync(s, p, rows * ncp * 8, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                                          c->stream);
    p = s;
    return r;
  };
  CK(up(in.e, 0, 1));
  CK(up(in.u, 1, 3));
  CK(up(in.pi, 4, 10));
  CK(up(in.Pi, 14, 1));
  CK(up(in.u_prev, 15, 3));
  CK(cudaMemsetAsync(c->d_stat, 0, 256, c->stream));
  const unsigned nb = (unsigned)((ncp + kSetThreads - 1) / kSetThreads);
  const double g = c->P.milne ? tau * tau : 1.0, gp = c->P.milne ? (tau - c->P.dtau) * (tau - c->P.dtau) : 1.0;
  TauSlot* slot = c->d_tau + c->cur;
  // the state goes into the buffers that hold u^n and u^{n-1} in the current rotation
  if (c->mixed)
    set_state_kernel<float><<<nb, kSetThreads, 0, c->stream>>>(c->P, L, in, tau, g, gp, slot, c->q, c->qf, (float*)c->U[c->cur],
                                                       (float*)c->U[c->prev], (float*)c->E[0], (float*)c->Pb[0],
                                                       c->reg, c->d_stat);
  else
    set_state_kernel<double><<<nb, kSetThreads, 0, c->stream>>>(c->P, L, in, tau, g, gp, slot, c->q, nullptr, (double*)c->U[c->cur],
                                                        (double*)c->U[c->prev], (double*)c->E[0], (double*)c->Pb[0],
                                                        c->reg, c->d_stat);
  CK(cudaGetLastError());
  unsigned st = 0;
  CK(cudaMemcpyAsync(&st, c->d_stat, 4, cudaMemcpyDeviceToHost, c->stream));
  CK(cudaStreamSynchronize(c->stream));
  c->tau = tau;
  c->steps = 0;
  c->ev_set[event] = 1;
  if (st & ST_NONFINITE) return fail(c, KT_ERR_STATE, "kt_set_state: non-finite input or negative e");
  if (st) return fail(c, KT_ERR_STATE, "kt_set_state: T^{tau tau} - pi^{tau tau} <= |T^{tau i} - pi^{tau i}| "
                                       "in some cell (no (e, u) solves Eq. eInferred)");
  return KT_OK;
}

int kt_set_state(kt_ctx* c, double tau, const double* e, const double* u, const double* pi, const double* Pi,
                 const double* u_prev, int on_device) {
  return kt_set_state_event(c, 0, tau, e, u, pi, Pi, u_prev, on_device);
}

}  // extern "C"

namespace {

// One packed row of an event going out: the field component, whether it is float, the destination, and
// which of the caller's arrays that is in.
struct Row {
  const void* f;
  int f32;
  double* dst;
  int array;
};
// Rows to the caller's arrays, one launch per kRows rows: straight to arrays that kernels can write in place,
// else (host arrays among them) through the staging area with one copy per caller's array (its rows adjoin).
// Two arrays that happen to adjoin are copied apart all the same: each may be a pinned allocation of its own,
// and a copy across both is refused.
int gather_rows(Ctx* c, const Lattice& L, const std::vector<Row>& rows, int on_device) {
  const size_t ncp = (size_t)L.nx * L.ny * L.nz;
  const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  int array = -1;  // the caller's array that `direct` is about
  bool direct = false;
  for (size_t b = 0; b < rows.size(); b += kRows) {
    GatherRows g = {};
    unsigned staged = 0;  // bit r: row r goes through the staging area
    g.n = (int)std::min<size_t>(kRows, rows.size() - b);
    for (int r = 0; r < g.n; ++r) {
      const Row& row = rows[b + r];
      if (row.array != array) {
        array = row.array;
        direct = on_device && in_place(c, row.dst);
      }
      if (!direct) staged |= 1u << r;
      g.src[r] = row.f;
      g.dst[r] = direct ? row.dst : c->stage + r * ncp;
      if (row.f32) g.f32 |= 1u << r;
    }
    const dim3 grid((unsigned)((ncp + 255) / 256), (unsigned)((g.n + kRowsPerThread - 1) / kRowsPerThread));
    gather_kernel<<<grid, 256, 0, c->stream>>>(L, g);
    CK(cudaGetLastError());
    for (int r = 0; r < g.n;) {
      int m = 1;
      while (r + m < g.n && rows[b + r + m].array == rows[b + r].array) ++m;
      if ((staged >> r) & 1u)
        CK(cudaMemcpyAsync(rows[b + r].dst, c->stage + r * ncp, m * ncp * 8, kind, c->stream));
      r += m;
    }
  }
  return KT_OK;
}

int begin_steps(Ctx* c, int n_steps) {
  for (int e = 0; e < c->nev; ++e)
    if (!c->ev_set[e]) return fail(c, KT_ERR_ARG, "kt_step: event %d has no state", e);
  if (c->mixed && c->opt.autotune && !c->tuned && n_steps > 0) {
    int rc = autotune(c);
    if (rc != KT_OK) return rc;
  }
  CK(cudaMemsetAsync(c->d_stat, 0, 256, c->stream));
  return KT_OK;
}

// read the statistics of the steps just enqueued (one synchronisation) and advance the host tau
int finish_steps(Ctx* c, int n_steps) {
  unsigned hst[KSTAT_WORDS];
  CK(cudaMemcpyAsync(hst, c->d_stat, sizeof(hst), cudaMemcpyDeviceToHost, c->stream));
  CK(cudaStreamSynchronize(c->stream));
  for (int s = 0; s < n_steps; ++s) c->tau += c->P.dtau;
  c->steps += n_steps;
  unsigned long long cnt[3];
  memcpy(cnt, &hst[4], sizeof(cnt));
  c->last.status = hst[0];
  float ms;
  memcpy(&ms, &hst[1], 4);
  c->last.max_speed = ms;
  c->last.newton_iters = (long long)cnt[0];
  c->last.regulated = (long long)cnt[1];
  c->last.fallbacks = (long long)cnt[2];
  if (hst[0] & ST_TIMEOUT) return fail(c, KT_ERR_TIMEOUT, "kt_step: a shared-memory copy timed out");
  if (hst[0] & ST_NONFINITE) return fail(c, KT_ERR_NONFINITE, "kt_step: non-finite value");
  if (hst[0] & ST_INVERSION) return fail(c, KT_ERR_INVERSION, "kt_step: inversion failed in some cell");
  return KT_OK;
}

}  // namespace

extern "C" {

int kt_step(kt_ctx* c, int n_steps) {
  Range range_("kt_step");
  if (!c || n_steps < 0) return KT_ERR_ARG;
  int rc = begin_steps(c, n_steps);
  if (rc != KT_OK) return rc;
  int done = 0;
  if (c->opt.use_graph) {
    while (n_steps - done >= 3) {
      int ph = c->cur;  // the three rotation phases are told apart by the current u buffer
      if (!c->graph[ph]) {
        rc = build_graph(c, ph);
        if (rc != KT_OK) return rc;
      }
      CK(cudaGraphLaunch(c->graph[ph], c->stream));
      done += 3;  // three steps return the rotation to the same phase
    }
  }
  for (; done < n_steps; ++done) {
    rc = enqueue_step(c);
    if (rc != KT_OK) return rc;
  }
  return finish_steps(c, n_steps);
}

int kt_time_kernels(kt_ctx* c, int n_steps, float* ms, int* n_kernels) {
  Range range_("kt_time_kernels");
  if (!c || n_steps < 1 || !ms || !n_kernels || *n_kernels < kNumTimed) return KT_ERR_ARG;
  int rc = begin_steps(c, n_steps);
  if (rc != KT_OK) return rc;
  cudaEvent_t ev[kNumTimed + 1];
  for (int k = 0; k <= kNumTimed; ++k) CK(cudaEventCreate(&ev[k]));
  double acc[kNumTimed] = {0.0};
  for (int s = 0; s < n_steps && rc == KT_OK; ++s) {
    rc = enqueue_step(c, ev);
    if (rc != KT_OK) break;
    cudaError_t e = cudaEventSynchronize(ev[kNumTimed]);
    if (e != cudaSuccess) { rc = fail(c, KT_ERR_CUDA, "kt_time_kernels: %s", cudaGetErrorString(e)); break; }
    for (int k = 0; k < kNumTimed; ++k) {
      float t = 0.f;
      cudaEventElapsedTime(&t, ev[k], ev[k + 1]);
      acc[k] += t;
    }
  }
  for (int k = 0; k <= kNumTimed; ++k) cudaEventDestroy(ev[k]);
  if (rc != KT_OK) return rc;
  for (int k = 0; k < kNumTimed; ++k) ms[k] = (float)(acc[k] / n_steps);
  *n_kernels = kNumTimed;
  return finish_steps(c, n_steps);
}

int kt_get_state_event(kt_ctx* c, int event, double* tau, double* e, double* u, double* pi, double* Pi, double* q,
                       int on_device) {
  Range range_("kt_get_state");
  if (!c) return KT_ERR_ARG;
  if (event < 0 || event >= c->nev) return fail(c, KT_ERR_ARG, "kt_get_state: bad event");
  const Lattice& L = c->lat[event];
  size_t ncp = (size_t)L.nx * L.ny * L.nz;
  const long long fs = c->gs;
  std::vector<Row> rows;
  const char* Ucur = (const char*)c->U[c->cur];
  if (e) rows.push_back({c->E[0], c->mixed, e, 0});
  if (u) for (int m = 0; m < 4; ++m) rows.push_back({Ucur + (size_t)m * fs * c->esz, c->mixed, u + m * ncp, 1});
  // component n of q: FP64, or (KT_STORE_PI_FP32, n >= 4) the FP32 state
  auto qrow = [&](int n, double* dst, int array) {
    if (c->pi32 && n >= 4) rows.push_back({c->qf + (size_t)n * fs, 1, dst, array});
    else rows.push_back({c->q + (size_t)n * fs, 0, dst, array});
  };
  if (pi) for (int m = 0; m < 10; ++m) qrow(4 + m, pi + m * ncp, 2);
  if (Pi) qrow(14, Pi, 3);
  if (q) for (int n = 0; n < NQ; ++n) qrow(n, q + n * ncp, 4);
  const int rc = gather_rows(c, L, rows, on_device);
  if (rc != KT_OK) return rc;
  CK(cudaStreamSynchronize(c->stream));
  if (tau) *tau = c->tau;
  return KT_OK;
}

int kt_get_state(kt_ctx* c, double* tau, double* e, double* u, double* pi, double* Pi, double* q, int on_device) {
  return kt_get_state_event(c, 0, tau, e, u, pi, Pi, q, on_device);
}

}  // extern "C"

namespace {

// The fields of a checkpoint row by row (see KT_CHECKPOINT_ROWS in kt.h): the field array (all
// events) and its element type: 0 double, 1 the stencil precision (float in KT_MIXED), 2 float.
struct CkptRow {
  void* f;
  int is_r;
};
std::vector<CkptRow> checkpoint_rows(Ctx* c) {
  std::vector<CkptRow> rows;
  const size_t fs = (size_t)c->gs;
  for (int n = 0; n < NQ; ++n)
    rows.push_back((c->pi32 && n >= 4) ? CkptRow{c->qf + n * fs, 2} : CkptRow{c->q + n * fs, 0});
  for (int n = 0; n < NQ; ++n)
    rows.push_back(c->mixed ? CkptRow{c->qf + n * fs, 1} : CkptRow{c->q + n * fs, 0});
  rows.push_back({c->E[0], 1});
  rows.push_back({c->Pb[0], 1});
  for (int m = 0; m < 4; ++m) rows.push_back({(char*)c->U[c->cur] + m * fs * c->esz, 1});
  for (int m = 0; m < 4; ++m) rows.push_back({(char*)c->U[c->prev] + m * fs * c->esz, 1});
  rows.push_back({c->reg, 2});  // float in both modes
  return rows;
}

}  // namespace

extern "C" {

int kt_get_checkpoint(kt_ctx* c, int event, double* tau, double* buf, int on_device) {
  Range range_("kt_get_checkpoint");
  if (!c || !buf) return KT_ERR_ARG;
  if (event < 0 || event >= c->nev) return fail(c, KT_ERR_ARG, "kt_get_checkpoint: bad event");
  if (!c->ev_set[event]) return fail(c, KT_ERR_ARG, "kt_get_checkpoint: event %d has no state", event);
  const Lattice& L = c->lat[event];
  const size_t ncp = (size_t)L.nx * L.ny * L.nz;
  static_assert(KT_CHECKPOINT_ROWS == 41, "checkpoint layout");
  std::vector<Row> rows;
  for (const CkptRow& r : checkpoint_rows(c)) rows.push_back({r.f, r.is_r == 2 || (r.is_r && c->mixed), buf + rows.size() * ncp, 0});
  const int rc = gather_rows(c, L, rows, on_device);
  if (rc != KT_OK) return rc;
  CK(cudaStreamSynchronize(c->stream));
  if (tau) *tau = c->tau;
  return KT_OK;
}

int kt_set_checkpoint(kt_ctx* c, int event, double tau, const double* buf, int on_device) {
  Range range_("kt_set_checkpoint");
  if (!c || !buf) return KT_ERR_ARG;
  if (event < 0 || event >= c->nev || !(tau > 0 || !c->P.milne))
    return fail(c, KT_ERR_ARG, "kt_set_checkpoint: bad argument");
  const Lattice& L = c->lat[event];
  const size_t ncp = (size_t)L.nx * L.ny * L.nz;
  const int nb = (int)((ncp + 255) / 256);
  const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  const std::vector<CkptRow> rows = checkpoint_rows(c);
  for (size_t b = 0; b < rows.size(); b += 18) {
    const size_t nr = std::min<size_t>(18, rows.size() - b);
    CK(cudaMemcpyAsync(c->stage, buf + b * ncp, nr * ncp * 8, kind, c->stream));
    for (size_t t = 0; t < nr; ++t) {
      const CkptRow& r = rows[b + t];
      const size_t row = b + t;
      if (!c->mixed && row >= (size_t)NQ && row < (size_t)(2 * NQ)) continue;  // FP64: the stencil reads q
      if (c->pi32 && row >= (size_t)(NQ + 4) && row < (size_t)(2 * NQ)) continue;  // the state rows hold them
      const double* src = c->stage + t * ncp;
      if (r.is_r == 2 || (r.is_r && c->mixed)) scatter_kernel<float><<<nb, 256, 0, c->stream>>>(c->P, L, src, (float*)r.f);
      else scatter_kernel<double><<<nb, 256, 0, c->stream>>>(c->P, L, src, (double*)r.f);
    }
    CK(cudaGetLastError());
  }
  const TauSlot slot = tau_slot(tau, c->P.dtau, c->P.milne);
  CK(cudaMemcpyAsync(c->d_tau + c->cur, &slot, sizeof(slot), cudaMemcpyHostToDevice, c->stream));
  CK(cudaMemsetAsync(c->d_stat, 0, 256, c->stream));
  CK(cudaStreamSynchronize(c->stream));
  c->tau = tau;
  c->steps = 0;
  c->ev_set[event] = 1;
  return KT_OK;
}

int kt_selftest_wait(kt_ctx* c, unsigned polls) {
  if (!c || polls == 0) return KT_ERR_ARG;
  CK(cudaMemsetAsync(c->d_stat, 0, 4, c->stream));
  wait_selftest_kernel<<<1, 128, 0, c->stream>>>(polls, c->d_stat);
  CK(cudaGetLastError());
  unsigned st = 0;
  CK(cudaMemcpyAsync(&st, c->d_stat, 4, cudaMemcpyDeviceToHost, c->stream));
  CK(cudaStreamSynchronize(c->stream));
  if (st & ST_TIMEOUT) return fail(c, KT_ERR_TIMEOUT, "kt_selftest_wait: the wait gave up after %u polls", polls);
  return KT_OK;
}

int kt_selftest_cvt(const double* x, float* rn, float* rz, long long n, void* stream) {
  if (!x || !rn || !rz || n < 0) return KT_ERR_ARG;
  if (n == 0) return KT_OK;
  cvt_selftest_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(x, rn, rz, n);
  return cudaGetLastError() == cudaSuccess ? KT_OK : KT_ERR_CUDA;
}

int kt_selftest_div(const double* a, const double* b, double* q, long long n, void* stream) {
  if (!a || !b || !q || n < 0) return KT_ERR_ARG;
  if (n == 0) return KT_OK;
  div_selftest_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(a, b, q, n);
  return cudaGetLastError() == cudaSuccess ? KT_OK : KT_ERR_CUDA;
}

int kt_get_diagnostics(kt_ctx* c, int event, double* out, int on_device) {
  Range range_("kt_get_diagnostics");
  if (!c || !out) return KT_ERR_ARG;
  if (event < 0 || event >= c->nev) return fail(c, KT_ERR_ARG, "kt_get_diagnostics: bad event");
  if (!c->ev_set[event]) return fail(c, KT_ERR_ARG, "kt_get_diagnostics: event %d has no state", event);
  const Lattice& L = c->lat[event];
  const size_t ncp = (size_t)L.nx * L.ny * L.nz;
  const int nb = (int)((ncp + 255) / 256);
  Lattice L0 = L;  // the event's own fields
  L0.base = 0;
  if (c->mixed)
    diag_kernel<float><<<nb, 256, 0, c->stream>>>(c->P, L0, from(make_io<float>(c, 1), L.base), c->tau, c->reg + L.base,
                                                  c->stage);
  else
    diag_kernel<double><<<nb, 256, 0, c->stream>>>(c->P, L0, from(make_io<double>(c, 1), L.base), c->tau, c->reg + L.base,
                                                   c->stage);
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(out, c->stage, 7 * ncp * 8, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                     c->stream));
  CK(cudaStreamSynchronize(c->stream));
  return KT_OK;
}

int kt_mlp_features(kt_ctx* c, long long n, const long long* cells, float* x, float* y, double* e_exact) {
  if (!c || n < 0 || !cells || !x || !y || !e_exact)
    return c ? fail(c, KT_ERR_ARG, "kt_mlp_features: bad argument") : KT_ERR_ARG;
  if (!c->ev_set[0]) return fail(c, KT_ERR_ARG, "kt_mlp_features: no state set");
  if (n == 0) return KT_OK;
  CK(cudaMemsetAsync(c->d_stat, 0, 4, c->stream));
  mlp_features_kernel<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(c->P, c->lat[0], c->q, c->qf, c->pi32,
                                                                          c->tau, n, cells, x, y, e_exact, c->d_stat);
  CK(cudaGetLastError());
  unsigned st = 0;
  CK(cudaMemcpyAsync(&st, c->d_stat, 4, cudaMemcpyDeviceToHost, c->stream));
  CK(cudaStreamSynchronize(c->stream));
  if (st) return fail(c, KT_ERR_INVERSION, "kt_mlp_features: bad cell index or failed root-find");
  return KT_OK;
}

int kt_get_tuning(kt_ctx* c, int* block_xyz, int* grid_blocks, float* candidate_ms, int* n_candidates) {
  if (!c) return KT_ERR_ARG;
  if (block_xyz) {
    const Shape s = c->mixed ? kShapes[c->shape] : (c->team ? Shape{32, 4, 1} : Shape{32, 1, 1});
    block_xyz[0] = s.x;
    block_xyz[1] = s.y;
    block_xyz[2] = s.z;
  }
  if (grid_blocks) *grid_blocks = c->grid_blocks;
  if (n_candidates) {
    if (candidate_ms)
      for (int s = 0; s < std::min(*n_candidates, kNumCandidates); ++s)
        candidate_ms[s] = c->tuned ? c->tune_ms[s] : 0.f;
    *n_candidates = kNumCandidates;
  }
  return KT_OK;
}

int kt_set_tuning(kt_ctx* c, int candidate) {
  if (!c || candidate < 0 || candidate >= kNumCandidates) return KT_ERR_ARG;
  int rc = select_shape(c, candidate);
  if (rc != KT_OK) return rc;
  c->tuned = true;  // no autotuning on the next step
  return KT_OK;
}

int kt_get_stats(kt_ctx* c, kt_stats* s) {
  if (!c || !s) return KT_ERR_ARG;
  kt_stats r = c->last;
  r.tau = c->tau;
  r.steps = c->steps;
  r.e_min = r.e_max = r.reg_min = 0.0;
  bool any = false;
  for (int e = 0; e < c->nev; ++e) any |= (c->ev_set[e] != 0);
  if (any) {  // the extrema of the current state, reduced on the device (words 12-14 of the stats block)
    unsigned* ext = c->d_stat + KSTAT_WORDS;
    const unsigned init[3] = {0x7f800000u, 0u, 0x7f800000u};
    CK(cudaMemcpyAsync(ext, init, sizeof(init), cudaMemcpyHostToDevice, c->stream));
    for (int e = 0; e < c->nev; ++e) {
      if (!c->ev_set[e]) continue;
      if (c->mixed) state_extrema_kernel<float><<<152, 256, 0, c->stream>>>(c->lat[e], (const float*)c->E[0], c->reg, ext);
      else state_extrema_kernel<double><<<152, 256, 0, c->stream>>>(c->lat[e], (const double*)c->E[0], c->reg, ext);
    }
    CK(cudaGetLastError());
    unsigned h[3];
    CK(cudaMemcpyAsync(h, ext, sizeof(h), cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    float f[3];
    memcpy(f, h, sizeof(f));
    r.e_min = f[0];
    r.e_max = f[1];
    r.reg_min = f[2];
  }
  *s = r;
  return KT_OK;
}

const char* kt_last_error(const kt_ctx* c) { return c ? c->err : "null context"; }

void kt_free(kt_ctx* c) {
  if (!c) return;
  for (int p = 0; p < 3; ++p)
    if (c->graph[p]) cudaGraphExecDestroy(c->graph[p]);
  if (c->base) cudaFree(c->base);
  if (c->own_stream) cudaStreamDestroy(c->stream);
  delete c;
}

}  // extern "C"

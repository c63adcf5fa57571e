// C ABI of the MHD hot path: handle, device buffers, launches, reductions.
#include <cuda.h>   // tensor-map types; the encoder itself is fetched from the driver at run time
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>   // header-only ranges; no cost unless a profiler is attached
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <array>
#include <functional>
#include <map>
#include <new>
#include <string>
#include <vector>

#include "../../include/mhd_gb300.h"
#include "batch.cuh"

namespace mhd {
cudaError_t launch_stage_fp64(int, int, int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&,
                                const TmaMaps&);
cudaError_t launch_stage_mixed(int, int, int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&,
                                const TmaMaps&);
cudaError_t launch_stage_fp32(int, int, int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&,
                                const TmaMaps&);
cudaError_t set_smem_fp64(int, int, size_t);
cudaError_t set_smem_mixed(int, int, size_t);
cudaError_t set_smem_fp32(int, int, size_t);
size_t smem_bytes_fp64(int, int);
size_t smem_bytes_mixed(int, int);
size_t smem_bytes_fp32(int, int);
size_t smem_bytes_char_fp64();
size_t smem_bytes_learned_fp64();
size_t smem_bytes_char_mixed();
size_t smem_bytes_learned_mixed();
size_t smem_bytes_char_fp32();
size_t smem_bytes_learned_fp32();
cudaError_t launch_stage_learned_fp64(int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&);
cudaError_t launch_stage_learned_mixed(int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&);
cudaError_t launch_stage_learned_fp32(int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&);
cudaError_t launch_stage_rk3_fp64(int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&, const TmaMaps&);
cudaError_t launch_stage_rk3_mixed(int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&, const TmaMaps&);
cudaError_t launch_stage_rk3_fp32(int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&, const TmaMaps&);
cudaError_t launch_stage_2d_fp64(int, int, int, unsigned, cudaStream_t, const Geo&, const StageArgs&);
cudaError_t launch_stage_2d_mixed(int, int, int, unsigned, cudaStream_t, const Geo&, const StageArgs&);
cudaError_t launch_stage_2d_fp32(int, int, int, unsigned, cudaStream_t, const Geo&, const StageArgs&);
cudaError_t set_smem_2d_fp64(int, int, bool);
cudaError_t set_smem_2d_mixed(int, int, bool);
cudaError_t set_smem_2d_fp32(int, int, bool);
cudaError_t set_smem_rk3_fp64(size_t);
cudaError_t set_smem_rk3_mixed(size_t);
cudaError_t set_smem_rk3_fp32(size_t);
cudaError_t launch_stage_char_fp64(int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&);
cudaError_t launch_stage_char_mixed(int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&);
cudaError_t launch_stage_char_fp32(int, unsigned, size_t, cudaStream_t, const Geo&, const StageArgs&);
cudaError_t set_smem_char_fp64(size_t);
cudaError_t set_smem_char_mixed(size_t);
cudaError_t set_smem_char_fp32(size_t);
cudaError_t set_smem_learned_fp64(size_t);
cudaError_t set_smem_learned_mixed(size_t);
cudaError_t set_smem_learned_fp32(size_t);
cudaError_t launch_prims_fp64(cudaStream_t, const Geo&, const StageArgs&);
cudaError_t launch_prims_mixed(cudaStream_t, const Geo&, const StageArgs&);
cudaError_t launch_prims_fp32(cudaStream_t, const Geo&, const StageArgs&);

cudaError_t launch_stage(int prec, int stage, int tx, int ty, unsigned nb, size_t smem, cudaStream_t st,
                         const Geo& g, const StageArgs& a, const TmaMaps* tm) {
  static const TmaMaps no_tma = {};
  const TmaMaps& maps = tm ? *tm : no_tma;
  if (g.n[2] == 1 && g.bc[2] == 0 && g.recon == 0 && g.riemann != 2) {
    // a two-dimensional box of a plain form: kernels of its own
    switch (prec) {
      case P_FP64: return launch_stage_2d_fp64(stage, tx, ty, nb, st, g, a);
      case P_MIXED: return launch_stage_2d_mixed(stage, tx, ty, nb, st, g, a);
      default: return launch_stage_2d_fp32(stage, tx, ty, nb, st, g, a);
    }
  }
  if (stage >= ST_RK3_1) {
    switch (prec) {
      case P_FP64: return launch_stage_rk3_fp64(stage, nb, smem, st, g, a, maps);
      case P_MIXED: return launch_stage_rk3_mixed(stage, nb, smem, st, g, a, maps);
      default: return launch_stage_rk3_fp32(stage, nb, smem, st, g, a, maps);
    }
  }
  if (g.recon == 1) {
    switch (prec) {
      case P_FP64: return launch_stage_char_fp64(stage, nb, smem, st, g, a);
      case P_MIXED: return launch_stage_char_mixed(stage, nb, smem, st, g, a);
      default: return launch_stage_char_fp32(stage, nb, smem, st, g, a);
    }
  }
  if (g.riemann == 2) {
    // learned switch: needs the network; 16 x 8 tile only
    if (!a.mlp) return cudaErrorInvalidValue;
    switch (prec) {
      case P_FP64: return launch_stage_learned_fp64(stage, nb, smem, st, g, a);
      case P_MIXED: return launch_stage_learned_mixed(stage, nb, smem, st, g, a);
      default: return launch_stage_learned_fp32(stage, nb, smem, st, g, a);
    }
  }
  switch (prec) {
    case P_FP64: return launch_stage_fp64(stage, tx, ty, nb, smem, st, g, a, maps);
    case P_MIXED: return launch_stage_mixed(stage, tx, ty, nb, smem, st, g, a, maps);
    default: return launch_stage_fp32(stage, tx, ty, nb, smem, st, g, a, maps);
  }
}
cudaError_t launch_prims(int prec, cudaStream_t st, const Geo& g, const StageArgs& a) {
  switch (prec) {
    case P_FP64: return launch_prims_fp64(st, g, a);
    case P_MIXED: return launch_prims_mixed(st, g, a);
    default: return launch_prims_fp32(st, g, a);
  }
}
cudaError_t stage_set_smem_char(int prec, size_t bytes) {
  switch (prec) {
    case P_FP64: return set_smem_char_fp64(bytes);
    case P_MIXED: return set_smem_char_mixed(bytes);
    default: return set_smem_char_fp32(bytes);
  }
}
// the shared memory of the two-dimensional kernels, which size it themselves
static cudaError_t stage_set_smem_2d(int prec, int tx, int ty, bool rk3) {
  switch (prec) {
    case P_FP64: return set_smem_2d_fp64(tx, ty, rk3);
    case P_MIXED: return set_smem_2d_mixed(tx, ty, rk3);
    default: return set_smem_2d_fp32(tx, ty, rk3);
  }
}
cudaError_t stage_set_smem_rk3(int prec, size_t bytes) {
  const cudaError_t e = stage_set_smem_2d(prec, 16, 8, true);
  if (e != cudaSuccess) return e;
  switch (prec) {
    case P_FP64: return set_smem_rk3_fp64(bytes);
    case P_MIXED: return set_smem_rk3_mixed(bytes);
    default: return set_smem_rk3_fp32(bytes);
  }
}
cudaError_t stage_set_smem_learned(int prec, size_t bytes) {
  switch (prec) {
    case P_FP64: return set_smem_learned_fp64(bytes);
    case P_MIXED: return set_smem_learned_mixed(bytes);
    default: return set_smem_learned_fp32(bytes);
  }
}
cudaError_t stage_set_smem(int prec, int tx, int ty, size_t bytes) {
  const cudaError_t e = stage_set_smem_2d(prec, tx, ty, false);
  if (e != cudaSuccess) return e;
  switch (prec) {
    case P_FP64: return set_smem_fp64(tx, ty, bytes);
    case P_MIXED: return set_smem_mixed(tx, ty, bytes);
    default: return set_smem_fp32(tx, ty, bytes);
  }
}
size_t stage_smem_bytes(int prec, int tx, int ty) {
  switch (prec) {
    case P_FP64: return smem_bytes_fp64(tx, ty);
    case P_MIXED: return smem_bytes_mixed(tx, ty);
    default: return smem_bytes_fp32(tx, ty);
  }
}
bool stage_tile_supported(int prec, int tx, int ty) { return stage_smem_bytes(prec, tx, ty) > 0; }

// Dynamic shared memory of the kernels a configuration launches: the
// characteristic-reconstruction kernels also hold per-cell slopes, the
// learned switch its face queue (and both keep the unpadded ring).
static size_t config_smem_bytes(int prec, int recon, int riemann, int tx, int ty) {
  if (recon == MHD_RECON_CHARACTERISTIC) {
    switch (prec) {
      case P_FP64: return smem_bytes_char_fp64();
      case P_MIXED: return smem_bytes_char_mixed();
      default: return smem_bytes_char_fp32();
    }
  }
  if (riemann == MHD_LEARNED) {
    // the learned kernel and the plain one (the rhs and dump paths) share the handle's size
    size_t l;
    switch (prec) {
      case P_FP64: l = smem_bytes_learned_fp64(); break;
      case P_MIXED: l = smem_bytes_learned_mixed(); break;
      default: l = smem_bytes_learned_fp32(); break;
    }
    const size_t p = stage_smem_bytes(prec, tx, ty);
    return l > p ? l : p;
  }
  return stage_smem_bytes(prec, tx, ty);
}
}  // namespace mhd

using namespace mhd;

struct mhd_handle {
  mhd_config cfg;
  Geo geo;
  cudaStream_t stream = nullptr;
  int device = 0;
  size_t elem = 8;          // bytes per state element
  size_t kelem = 8;         // bytes per stage-1 element
  size_t welem = 8;         // bytes per primitive element
  void* U[2] = {nullptr, nullptr};
  void* K1 = nullptr;
  void* Urk[2] = {nullptr, nullptr};        // RK3: the intermediate states U1, U2
  void* W[2] = {nullptr, nullptr};
  unsigned long long* words = nullptr;     // [0,1] CFL words (step parity), [2] reductions, [3] status,
                                           // [4] scratch, [8..] counters
  unsigned int* status = nullptr;
  unsigned long long* counters = nullptr;
  void* pinned = nullptr;                  // host readback buffer
  int cur = 0;                             // U[cur], W[cur] hold the current state
  int parity = 0;                          // words[parity] = CFL max of the current state
  bool prims_valid = false;                // W[cur] and words[parity] match U[cur]
  size_t smem_bytes = 0;
  double last_dt = 0.0;
  int steps = 0;
  bool profiling = false;
  void* mlp = nullptr;                     // copy of the switch network (device)
  float mlp_zt = 0.0f;                     // logit of the switch threshold tau
  std::vector<cudaEvent_t> ev_pool;        // 3 events per recorded step
  size_t ev_used = 0;
  std::string err;
  // host streaming (mhd_stream_step): the state buffers the handle owns (the
  // U pointers rotate over them), the two input slots, the copy streams and
  // the events that order slot reuse between the three streams
  std::vector<void*> owned_states;
  static constexpr int kSlots = 3;         // device states in flight per direction
  void* slot_in[kSlots] = {};
  void* slot_out[kSlots] = {};
  cudaStream_t s_in = nullptr, s_out = nullptr;
  cudaEvent_t ev_h2d[kSlots] = {}, ev_comp[kSlots] = {}, ev_d2h[kSlots] = {};
  long long nstream = 0;                   // streamed steps since the handle was created
  unsigned long long floors_seen = 0;      // floor hits already reported (MHD_FLOOR_ERROR)
  // TMA maps of the two primitive buffers (plain kernels with 4-byte
  // primitives); the W pointers swap every step, so each map keeps its base
  TmaMaps tmaps[2] = {};
  void* tmap_base[2] = {nullptr, nullptr};
};

// error text of calls without a handle, one per host thread (calls on
// different devices may run on several threads at once)
static thread_local std::string g_create_err;

static int fail(mhd_handle* h, int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  if (h) h->err = buf; else g_create_err = buf;
  return code;
}

#define CUDA_TRY(h, call)                                                                 \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess)                                                                \
      return fail((h), MHD_ERR_CUDA, "%s failed: %s", #call, cudaGetErrorString(e_));     \
  } while (0)

extern "C" void mhd_default_config(mhd_config* c, int nx, int ny, int nz) {
  memset(c, 0, sizeof *c);
  c->nx = nx; c->ny = ny; c->nz = nz;
  int m = nx > ny ? nx : ny;
  m = m > nz ? m : nz;
  c->dx = c->dy = c->dz = 1.0 / (m > 0 ? m : 1);
  c->gamma = 5.0 / 3.0;
  c->cfl = 0.4;
  c->precision = MHD_FP64;
  c->riemann = MHD_HLLD;
  c->emf = MHD_EMF_UPWIND;
  c->rho_floor = 1e-10;
  c->p_floor = 1e-10;
}

// ---- z-chunk length ---------------------------------------------------------
// The device time of a launch whose CTAs march chunks of planes, in units of
// a lone CTA's plane.  `groups` lists (planes of a chunk, number of chunks) in
// the order they start; each of the kSMs SMs holds up to `most` CTAs and takes
// the next chunk when one of its own ends.  The CTAs of an SM do not share it
// evenly: the one that started first issues first and runs ahead, so that a
// launch of one wave ends with its SMs half empty (mixed 240^3: 240 planes a
// chunk 2237 us a stage, 32 planes 1969).  rate[n - 1] holds the planes per
// unit of an SM's n CTAs, oldest first.  A chunk costs its planes and a
// prologue.  SMs in the same state advance together.
struct ChunkGroup {
  int planes;
  long long count;
};
static constexpr int kSMs = 152;

struct MarchRates {
  int most;
  double rate[3][3];
  double prologue;
};

// FP64 CTAs share the FP64 pipe, which one of them keeps busy.  The rates of
// the others are a fit to 260 measured stages (16 sizes of 48^3 to 320^3 at all
// chunk lengths, mixed and FP32; the estimates are 2.6 % off in the mean, FP64
// 0.8 %).
static MarchRates march_rates(bool fp64, int most) {
  if (fp64) return {most, {{1.0}, {0.5, 0.5}, {1.0 / 3, 1.0 / 3, 1.0 / 3}}, 1.8};
  return {most, {{1.0}, {0.90, 0.75}, {0.825, 0.67, 0.515}}, 1.65};
}

// (`groups` is used up.  No heap: a step of mhd_step_noalloc comes here.)
static double march_time(ChunkGroup* groups, size_t ngroups, const MarchRates& m) {
  struct SMs {
    int count, n;
    double left[3];   // of the resident chunks, oldest first
  };
  SMs sms[kSMs], merged[kSMs];   // every entry stands for at least one SM
  int nsms = 1;
  sms[0] = {kSMs, 0, {}};
  double time = 0.0;
  size_t next = 0;
  for (int event = 0; event < 1 << 14; ++event) {
    for (int n = 0; n < m.most; ++n)   // waiting chunks go to the emptiest SMs first
      for (int i = 0; i < nsms; ++i) {
        while (next < ngroups && groups[next].count == 0) ++next;
        if (next == ngroups) break;
        if (sms[i].n != n) continue;
        const int take = (int)std::min<long long>(sms[i].count, groups[next].count);
        if (take < sms[i].count) {
          sms[nsms] = sms[i];
          sms[nsms++].count -= take;
          sms[i].count = take;
        }
        sms[i].left[sms[i].n++] = groups[next].planes + m.prologue;
        groups[next].count -= take;
      }
    double step = HUGE_VAL;
    for (int c = 0; c < nsms; ++c)
      for (int i = 0; i < sms[c].n; ++i) step = std::min(step, sms[c].left[i] / m.rate[sms[c].n - 1][i]);
    if (step == HUGE_VAL) return time;
    time += step;
    int nmerged = 0;
    for (int c = 0; c < nsms; ++c) {
      SMs d = {sms[c].count, 0, {}};
      for (int i = 0; i < sms[c].n; ++i) {
        const double left = sms[c].left[i] - step * m.rate[sms[c].n - 1][i];
        if (left > 1e-6) d.left[d.n++] = left;
      }
      const auto alike = [&](const SMs& e) {
        if (e.n != d.n) return false;
        for (int i = 0; i < d.n; ++i)
          if (std::fabs(e.left[i] - d.left[i]) > 1e-4) return false;
        return true;
      };
      SMs* const end = merged + nmerged;
      SMs* const it = std::find_if(merged, end, alike);
      if (it == end) merged[nmerged++] = d;
      else it->count += d.count;
    }
    std::copy(merged, merged + nmerged, sms);
    nsms = nmerged;
  }
  return HUGE_VAL;
}

// CTAs per SM of the kernel a configuration runs (the kernels' launch bounds)
static int resident_ctas(const mhd_config* c, int tx, int ty) {
  if (c->precision == MHD_FP64) return tx * ty <= 64 || c->riemann == MHD_LEARNED ? 2 : 1;
  if (c->recon == MHD_RECON_CHARACTERISTIC) return 2;
  return tx * ty >= 256 ? 1 : (tx * ty >= 192 ? 2 : 3);
}

// Default planes per z-chunk: 32, unless march_time finds a length that takes
// less than 0.98 of it.  Small boxes then have chunks enough for every SM (us a
// stage: 24^3 FP64 1 plane a chunk 109, one chunk of 24 975; 64^3 mixed 5: 66,
// 32: 181) and middle ones no nearly empty last wave (128^3 FP64 16: 4619, 32:
// 5001; 128^3 mixed 15: 362, 32: 437; 97x130x75 FP32 13: 204, 32: 236; 240^3
// mixed stays at 32: 1969, one chunk of 240: 2237).  On 17 sizes from 24^3 to
// 352^3 and all precisions the choice took at most 1.7 % more than the best length.
// Results do not depend on it, but for the learned switch in FP32 arithmetic,
// whose first pass over a chunk rounds differently: it keeps 32.
static int default_chunk(const mhd_config* c, int tx, int ty) {
  if (c->nz <= 1 || (c->riemann == MHD_LEARNED && c->precision != MHD_FP64)) return 32;
  const long long columns = (long long)((c->nx + tx - 1) / tx) * ((c->ny + ty - 1) / ty);
  const MarchRates rates = march_rates(c->precision == MHD_FP64, resident_ctas(c, tx, ty));
  const auto estimate = [&](int tz) {
    const int n = (c->nz + tz - 1) / tz, last = c->nz - (n - 1) * tz;
    ChunkGroup groups[2] = {{tz, columns * (n - 1)}, {last, columns}};
    return march_time(groups, 2, rates);
  };
  int best = 32;
  const double base = estimate(32);
  double least = 0.98 * base;
  for (int n = 1, tz = c->nz, previous = 0; n <= c->nz; ++n, previous = tz) {
    tz = (c->nz + n - 1) / n;
    if (tz == previous || tz > (1 << 20)) continue;
    if (tz < 16 && columns * n > 40LL * kSMs * rates.most) break;   // shorter chunks only add prologues to a full chip
    const double t = estimate(tz);
    if (t < least) {
      least = t;
      best = tz;
    }
  }
  return best;
}

static void resolve_tile(const mhd_config* c, int* tx, int* ty) {
  *tx = c->tile_x ? c->tile_x : 16;
  *ty = c->tile_y ? c->tile_y : 8;
}

static int validate(const mhd_config* c, mhd_handle* h) {
  if (!c) return fail(h, MHD_ERR_INVALID, "null config");
  if (c->nx < 1 || c->ny < 1 || c->nz < 1) return fail(h, MHD_ERR_INVALID, "grid must have >= 1 cell per axis");
  if ((long long)c->nx * c->ny * c->nz > (1LL << 33)) return fail(h, MHD_ERR_INVALID, "grid too large");
  int n[3] = {c->nx, c->ny, c->nz};
  double d[3] = {c->dx, c->dy, c->dz};
  for (int a = 0; a < 3; ++a) {
    if (c->bc[a] != MHD_BC_PERIODIC && c->bc[a] != MHD_BC_OUTFLOW)
      return fail(h, MHD_ERR_INVALID, "bc[%d] must be MHD_BC_PERIODIC or MHD_BC_OUTFLOW", a);
    if (c->bc[a] == MHD_BC_OUTFLOW && n[a] < 2) return fail(h, MHD_ERR_INVALID, "an outflow axis needs >= 2 cells");
    if (!(d[a] > 0.0)) return fail(h, MHD_ERR_INVALID, "cell sizes must be positive");
  }
  if (!(c->gamma > 1.0)) return fail(h, MHD_ERR_INVALID, "gamma must exceed 1");
  if (!(c->cfl > 0.0)) return fail(h, MHD_ERR_INVALID, "cfl must be positive");
  if (c->precision < MHD_FP64 || c->precision > MHD_FP32) return fail(h, MHD_ERR_INVALID, "unknown precision");
  if (c->riemann < MHD_HLLD || c->riemann > MHD_LEARNED) return fail(h, MHD_ERR_INVALID, "unknown riemann solver");
  if (c->emf != MHD_EMF_UPWIND && c->emf != MHD_EMF_MEAN) return fail(h, MHD_ERR_INVALID, "unknown emf mode");
  if (!(c->rho_floor > 0.0) || !(c->p_floor > 0.0)) return fail(h, MHD_ERR_INVALID, "floors must be positive");
  if (c->tile_x < 0 || c->tile_y < 0 || c->tile_z < 0) return fail(h, MHD_ERR_INVALID, "tile sizes must be >= 0");
  int tx, ty;
  resolve_tile(c, &tx, &ty);
  if (c->tile_z > (1 << 20)) return fail(h, MHD_ERR_INVALID, "tile_z out of range");
  if (!stage_tile_supported(c->precision, tx, ty))
    return fail(h, MHD_ERR_INVALID, "tile %dx%d is not instantiated for this precision", tx, ty);
  if (c->riemann == MHD_LEARNED && (tx != 16 || ty != 8))
    return fail(h, MHD_ERR_INVALID, "the learned switch is instantiated for the 16x8 tile only (got %dx%d)", tx, ty);
  if (c->integrator != MHD_RK2 && c->integrator != MHD_RK3) return fail(h, MHD_ERR_INVALID, "unknown integrator");
  if (c->floor_policy != MHD_FLOOR_COUNT && c->floor_policy != MHD_FLOOR_ERROR)
    return fail(h, MHD_ERR_INVALID, "unknown floor policy");
  if (c->plane_copy != MHD_COPY_AUTO && c->plane_copy != MHD_COPY_GATHER)
    return fail(h, MHD_ERR_INVALID, "unknown plane copy mode");
  if (c->integrator == MHD_RK3 && (tx != 16 || ty != 8))
    return fail(h, MHD_ERR_INVALID, "SSP-RK3 is instantiated for the 16x8 tile only (got %dx%d)", tx, ty);
  if (c->integrator == MHD_RK3 && c->riemann == MHD_LEARNED)
    return fail(h, MHD_ERR_INVALID, "the learned switch runs with the RK2 integrator");
  if (c->recon != MHD_RECON_PRIMITIVE && c->recon != MHD_RECON_CHARACTERISTIC)
    return fail(h, MHD_ERR_INVALID, "unknown reconstruction");
  if (c->recon == MHD_RECON_CHARACTERISTIC &&
      (tx != 16 || ty != 8 || c->integrator != MHD_RK2 || c->riemann == MHD_LEARNED))
    return fail(h, MHD_ERR_INVALID, "characteristic reconstruction runs on the 16x8 tile with RK2 and HLLD or HLL");
  if (config_smem_bytes(c->precision, c->recon, c->riemann, tx, ty) > 227 * 1024)
    return fail(h, MHD_ERR_INVALID, "tile %dx%d needs %zu B of shared memory (> 227 KB)", tx, ty,
                config_smem_bytes(c->precision, c->recon, c->riemann, tx, ty));
  return MHD_OK;
}

static void fill_geo(const mhd_config* c, Geo* g) {
  memset(g, 0, sizeof *g);
  g->n[0] = c->nx; g->n[1] = c->ny; g->n[2] = c->nz;
  for (int a = 0; a < 3; ++a) {
    g->bc[a] = c->bc[a];
    g->nf[a] = g->n[a] + (c->bc[a] == MHD_BC_OUTFLOW ? 1 : 0);
  }
  g->inv_d[0] = 1.0 / c->dx; g->inv_d[1] = 1.0 / c->dy; g->inv_d[2] = 1.0 / c->dz;
  for (int a = 0; a < 3; ++a) g->finv_d[a] = (float)g->inv_d[a];
  g->gamma = c->gamma; g->rho_floor = c->rho_floor; g->p_floor = c->p_floor; g->cfl = c->cfl;
  g->emf_mean = c->emf == MHD_EMF_MEAN;
  g->riemann = c->riemann == MHD_HLL ? 1 : (c->riemann == MHD_LEARNED ? 2 : 0);
  g->recon = c->recon == MHD_RECON_CHARACTERISTIC ? 1 : 0;
  g->deadband = c->precision == MHD_FP64 ? 1e-10 : 1e-6;
  if (getenv("MHD_DEADBAND")) g->deadband = atof(getenv("MHD_DEADBAND"));
  g->gm1 = g->gamma - 1.0;
  g->fgamma = (float)g->gamma;
  g->fgm1 = (float)g->gm1;
  g->frho_floor = (float)g->rho_floor;
  g->fp_floor = (float)g->p_floor;
  g->fdeadband = (float)g->deadband;
  resolve_tile(c, &g->TX, &g->TY);
  g->TZ = c->tile_z ? c->tile_z : default_chunk(c, g->TX, g->TY);
  g->ntx = (g->n[0] + g->TX - 1) / g->TX;
  g->nty = (g->n[1] + g->TY - 1) / g->TY;
  g->nchunk = (g->n[2] + g->TZ - 1) / g->TZ;
  g->ncell = (long long)g->n[0] * g->n[1] * g->n[2];
  long long o = 5 * g->ncell;
  for (int a = 0; a < 3; ++a) {
    long long cnt = (long long)(a == 0 ? g->nf[0] : g->n[0]) * (a == 1 ? g->nf[1] : g->n[1]) *
                    (a == 2 ? g->nf[2] : g->n[2]);
    g->face_off[a] = o;
    o += cnt;
  }
  g->total = o;
}

// ---- TMA maps -----------------------------------------------------------------

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn tensor_map_encoder() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    cudaGetLastError();
    return (EncodeTiledFn)p;
  }();
  return fn;
}

// Maps of one primitive buffer: 4D (x, y, z, array) over 11 arrays of n0 x
// n1 x n2 floats; the 8-primitive plane box and the 3-field lower-face box
// of a tile's ring (ring x-offset 4).  Left off (on = 0) where the form has
// no TMA path or the layout breaks a tensor-copy rule (rows of n0 floats
// must be multiples of 16 bytes).
static void build_tma_maps(const mhd_handle* h, void* wbuf, TmaMaps* out) {
  memset(out, 0, sizeof *out);
  const Geo& g = h->geo;
  const mhd_config& c = h->cfg;
  if (c.plane_copy != MHD_COPY_AUTO || c.precision == MHD_FP64 || c.recon != MHD_RECON_PRIMITIVE ||
      c.riemann == MHD_LEARNED)
    return;
  if (g.n[2] < 2 || g.n[0] % 4 != 0 || ((uintptr_t)wbuf & 15u)) return;
  const EncodeTiledFn encode = tensor_map_encoder();
  if (!encode) return;
  const cuuint32_t W = (cuuint32_t)(g.TX + 8), H = (cuuint32_t)(g.TY + 4);
  const cuuint64_t dims[4] = {(cuuint64_t)g.n[0], (cuuint64_t)g.n[1], (cuuint64_t)g.n[2], (cuuint64_t)NW};
  const cuuint64_t strides[3] = {(cuuint64_t)g.n[0] * 4, (cuuint64_t)g.n[0] * g.n[1] * 4, (cuuint64_t)g.ncell * 4};
  const cuuint32_t box_p[4] = {W, H, 1, 8}, box_b[4] = {W, H - 2, 1, 3}, es[4] = {1, 1, 1, 1};
  const CUresult r1 = encode(reinterpret_cast<CUtensorMap*>(&out->p), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, wbuf, dims,
                             strides, box_p, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  const CUresult r2 = encode(reinterpret_cast<CUtensorMap*>(&out->bn), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, wbuf, dims,
                             strides, box_b, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  out->on = r1 == CUDA_SUCCESS && r2 == CUDA_SUCCESS;
}

// the maps of the buffer a stage reads its primitives from, or null
static const TmaMaps* tma_for(const mhd_handle* h, const void* win) {
  for (int i = 0; i < 2; ++i)
    if (h->tmaps[i].on && h->tmap_base[i] == win) return &h->tmaps[i];
  return nullptr;
}

// NVTX range over one host entry point (seen by Nsight Systems as the call's
// span on the host timeline; the kernels it enqueues appear beneath it)
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
};

static long long face_count(const Geo& g, int d) {
  long long n[3] = {g.n[0], g.n[1], g.n[2]};
  n[d] = g.nf[d];
  return n[0] * n[1] * n[2];
}

extern "C" int mhd_create(const mhd_config* cfg, void* cuda_stream, mhd_handle** out) {
  if (!out) return fail(nullptr, MHD_ERR_INVALID, "null output pointer");
  int rc = validate(cfg, nullptr);
  if (rc) return rc;
  mhd_handle* h = new (std::nothrow) mhd_handle();
  if (!h) return fail(nullptr, MHD_ERR_NOMEM, "host allocation failed");
  h->cfg = *cfg;
  fill_geo(cfg, &h->geo);
  h->stream = (cudaStream_t)cuda_stream;
  h->elem = cfg->precision == MHD_FP32 ? 4 : 8;
  h->kelem = cfg->precision == MHD_FP64 ? 8 : 4;
  h->welem = cfg->precision == MHD_FP64 ? 8 : 4;
  h->smem_bytes = config_smem_bytes(cfg->precision, cfg->recon, cfg->riemann, h->geo.TX, h->geo.TY);
  cudaError_t e = cudaGetDevice(&h->device);
  const size_t bytes = (size_t)h->geo.total * h->elem;
  const size_t kbytes = (size_t)h->geo.total * h->kelem;
  const size_t wbytes = (size_t)h->geo.ncell * NW * h->welem;
  if (e == cudaSuccess) e = cudaMalloc(&h->U[0], bytes);
  if (e == cudaSuccess) e = cudaMalloc(&h->U[1], bytes);
  h->owned_states = {h->U[0], h->U[1]};
  if (e == cudaSuccess) e = cudaMalloc(&h->K1, kbytes);
  if (e == cudaSuccess && cfg->integrator == MHD_RK3) e = cudaMalloc(&h->Urk[0], bytes);
  if (e == cudaSuccess && cfg->integrator == MHD_RK3) e = cudaMalloc(&h->Urk[1], bytes);
  if (e == cudaSuccess) e = cudaMalloc(&h->W[0], wbytes);
  if (e == cudaSuccess) e = cudaMalloc(&h->W[1], wbytes);
  if (e == cudaSuccess) e = cudaMalloc(&h->words, 64 * sizeof(unsigned long long));
  if (e == cudaSuccess) e = cudaMallocHost(&h->pinned, 256);
  if (e != cudaSuccess) {
    int code = e == cudaErrorMemoryAllocation ? MHD_ERR_NOMEM : MHD_ERR_CUDA;
    fail(nullptr, code, "device allocation of %zu B failed: %s", 2 * bytes + kbytes + 2 * wbytes,
         cudaGetErrorString(e));
    cudaGetLastError();
    mhd_destroy(h);
    return code;
  }
  h->status = (unsigned int*)(h->words + 3);
  h->counters = h->words + 8;
  for (int i = 0; i < 2; ++i) {
    h->tmap_base[i] = h->W[i];
    build_tma_maps(h, h->W[i], &h->tmaps[i]);
  }
  e = cudaMemsetAsync(h->words, 0, 64 * sizeof(unsigned long long), h->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(h->U[0], 0, bytes, h->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(h->K1, 0, kbytes, h->stream);
  if (e == cudaSuccess) e = stage_set_smem(cfg->precision, h->geo.TX, h->geo.TY, h->smem_bytes);
  if (e == cudaSuccess && cfg->riemann == MHD_LEARNED) e = stage_set_smem_learned(cfg->precision, h->smem_bytes);
  if (e == cudaSuccess && cfg->integrator == MHD_RK3) e = stage_set_smem_rk3(cfg->precision, h->smem_bytes);
  if (e == cudaSuccess && cfg->recon == MHD_RECON_CHARACTERISTIC)
    e = stage_set_smem_char(cfg->precision, h->smem_bytes);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) {
    fail(nullptr, MHD_ERR_CUDA, "initialisation failed: %s", cudaGetErrorString(e));
    cudaGetLastError();
    mhd_destroy(h);
    return MHD_ERR_CUDA;
  }
  *out = h;
  return MHD_OK;
}

extern "C" void mhd_destroy(mhd_handle* h) {
  if (!h) return;
  if (h->stream) cudaStreamSynchronize(h->stream); else cudaDeviceSynchronize();
  if (h->s_in) cudaStreamSynchronize(h->s_in);
  if (h->s_out) cudaStreamSynchronize(h->s_out);
  for (void* p : h->owned_states) cudaFree(p);
  for (int p = 0; p < mhd_handle::kSlots; ++p) {
    if (h->ev_h2d[p]) cudaEventDestroy(h->ev_h2d[p]);
    if (h->ev_comp[p]) cudaEventDestroy(h->ev_comp[p]);
    if (h->ev_d2h[p]) cudaEventDestroy(h->ev_d2h[p]);
  }
  if (h->s_in) cudaStreamDestroy(h->s_in);
  if (h->s_out) cudaStreamDestroy(h->s_out);
  cudaFree(h->K1);
  cudaFree(h->Urk[0]);
  cudaFree(h->Urk[1]);
  cudaFree(h->W[0]);
  cudaFree(h->W[1]);
  cudaFree(h->words);
  cudaFree(h->mlp);
  if (h->pinned) cudaFreeHost(h->pinned);
  for (cudaEvent_t e : h->ev_pool) cudaEventDestroy(e);
  delete h;
}

extern "C" const char* mhd_last_error(const mhd_handle* h) {
  return h ? h->err.c_str() : g_create_err.c_str();
}

// ---- state copies -------------------------------------------------------------
// The eight arrays of a state between the caller's device arrays and a packed
// buffer, in one launch: blockIdx.y is the array.  16 bytes a thread and access
// where both ends are aligned to 16, else 8, else 4 (the element sizes).  Eight
// copies of a small box are eight launches of ~2 us each, on the host and on
// the device (measured, set / get: 128^2 FP64 51 / 45 -> 29 / 20 us,
// 64 boxes 3449 / 3938 -> 1131 / 1712, 256^3 375 / 362 -> 367 / 355).
struct StateCopy {
  const void* src[8];
  void* dst[8];
  unsigned long long bytes[8];
};

template <typename V>
__device__ __forceinline__ void copy_as(const void* src, void* dst, unsigned long long bytes) {
  const unsigned long long n = bytes / sizeof(V), step = (unsigned long long)gridDim.x * blockDim.x;
  unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  const V* s = (const V*)src;
  V* d = (V*)dst;
  for (; i + 3 * step < n; i += 4 * step) {   // four loads in flight
    const V a = s[i], b = s[i + step], c = s[i + 2 * step], e = s[i + 3 * step];
    d[i] = a;
    d[i + step] = b;
    d[i + 2 * step] = c;
    d[i + 3 * step] = e;
  }
  for (; i < n; i += step) d[i] = s[i];
  const unsigned long long done = n * sizeof(V);   // the rest, fewer than 16 bytes
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < (unsigned)((bytes - done) / 4))
    ((unsigned*)((char*)dst + done))[t] = ((const unsigned*)((const char*)src + done))[t];
}

__global__ void __launch_bounds__(256) state_copy_kernel(StateCopy c) {
  const int q = blockIdx.y;
  const uintptr_t both = (uintptr_t)c.src[q] | (uintptr_t)c.dst[q];
  if ((both & 15) == 0) copy_as<uint4>(c.src[q], c.dst[q], c.bytes[q]);
  else if ((both & 7) == 0) copy_as<uint2>(c.src[q], c.dst[q], c.bytes[q]);
  else copy_as<unsigned>(c.src[q], c.dst[q], c.bytes[q]);
}

// How the bytes from p on may be copied: by the kernel where they are plain
// memory of the current device, by the runtime's copy where they are anything
// else (a host pointer passed for a device one among it); not at all where they
// run past the end of the cudaMalloc allocation that p lies in, which the
// runtime's copy refuses and a kernel would not notice.  (Of memory mapped
// piecewise the driver knows the piece; the runtime's copy judges that.)
enum CopyKind { COPY_KERNEL, COPY_RUNTIME, COPY_REFUSED };
static CopyKind copy_kind(const void* p, unsigned long long bytes, int current) {
  static const auto attributes = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    cudaGetLastError();
    return (CUresult(*)(unsigned, CUpointer_attribute*, void**, CUdeviceptr))f;
  }();
  unsigned type = 0, managed = 0, whole = 0;
  int device = -1;
  CUdeviceptr start = 0;
  size_t size = 0;
  CUpointer_attribute ask[6] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE,     CU_POINTER_ATTRIBUTE_IS_MANAGED,
                                CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL,  CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                CU_POINTER_ATTRIBUTE_RANGE_SIZE,      CU_POINTER_ATTRIBUTE_IS_LEGACY_CUDA_IPC_CAPABLE};
  void* out[6] = {&type, &managed, &device, &start, &size, &whole};
  const CUdeviceptr at = (CUdeviceptr)(uintptr_t)p;
  if (!attributes || attributes(6, ask, out, at) != CUDA_SUCCESS || type != CU_MEMORYTYPE_DEVICE || managed)
    return COPY_RUNTIME;
  if (at < start || at - start > size || bytes > size - (at - start)) return whole ? COPY_REFUSED : COPY_RUNTIME;
  return device == current && (at & 3) == 0 ? COPY_KERNEL : COPY_RUNTIME;
}

namespace mhd {
// Copy the arrays of a packed state (in: to it, else from it), device to device.
cudaError_t copy_state_on_device(const Geo& g, bool in, char* base, size_t elem, void* const* cell, void* const* face,
                                 cudaStream_t st) {
  StateCopy c;
  int current = -1;
  cudaError_t e = cudaGetDevice(&current);
  if (e != cudaSuccess) return e;
  bool plain = copy_kind(base, 0, current) == COPY_KERNEL;   // (a handle of another device than the current one)
  unsigned long long most = 0;
  for (int q = 0; q < 8; ++q) {
    void* user = q < 5 ? cell[q] : face[q - 5];
    char* own = base + (size_t)(q < 5 ? q * g.ncell : g.face_off[q - 5]) * elem;
    c.src[q] = in ? user : own;
    c.dst[q] = in ? own : user;
    c.bytes[q] = (unsigned long long)(q < 5 ? g.ncell : face_count(g, q - 5)) * elem;
    most = std::max(most, c.bytes[q]);
    const CopyKind kind = copy_kind(user, c.bytes[q], current);
    if (kind == COPY_REFUSED) return cudaErrorInvalidValue;
    plain = plain && kind == COPY_KERNEL;
  }
  if (plain) {
    const unsigned blocks = (unsigned)std::min<unsigned long long>((most + 4095) / 4096, 152ull * 4);
    state_copy_kernel<<<dim3(blocks, 8), 256, 0, st>>>(c);
    return cudaGetLastError();
  }
  for (int q = 0; q < 8 && e == cudaSuccess; ++q)
    e = cudaMemcpyAsync(c.dst[q], c.src[q], c.bytes[q], cudaMemcpyDeviceToDevice, st);
  return e;
}
}  // namespace mhd

static int copy_arrays(mhd_handle* h, bool in, char* base, size_t elem, void* const* cell, void* const* face,
                       int on_device) {
  if (!cell || !face) return fail(h, MHD_ERR_INVALID, "null state pointer array");
  for (int v = 0; v < 5; ++v)
    if (!cell[v]) return fail(h, MHD_ERR_INVALID, "null cell array %d", v);
  for (int d = 0; d < 3; ++d)
    if (!face[d]) return fail(h, MHD_ERR_INVALID, "null face array %d", d);
  if (on_device) {
    CUDA_TRY(h, copy_state_on_device(h->geo, in, base, elem, cell, face, h->stream));
    if (!in) CUDA_TRY(h, cudaStreamSynchronize(h->stream));
    return MHD_OK;
  }
  const cudaMemcpyKind kind = in ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost;
  for (int v = 0; v < 5; ++v) {
    char* dev = base + (size_t)v * h->geo.ncell * elem;
    size_t n = (size_t)h->geo.ncell * elem;
    CUDA_TRY(h, in ? cudaMemcpyAsync(dev, cell[v], n, kind, h->stream) : cudaMemcpyAsync(cell[v], dev, n, kind, h->stream));
  }
  for (int d = 0; d < 3; ++d) {
    char* dev = base + (size_t)h->geo.face_off[d] * elem;
    size_t n = (size_t)face_count(h->geo, d) * elem;
    CUDA_TRY(h, in ? cudaMemcpyAsync(dev, face[d], n, kind, h->stream) : cudaMemcpyAsync(face[d], dev, n, kind, h->stream));
  }
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  return MHD_OK;
}

extern "C" int mhd_set_state(mhd_handle* h, const void* const cell[5], const void* const face[3], int on_device) {
  if (!h) return MHD_ERR_INVALID;
  int rc = copy_arrays(h, true, (char*)h->U[h->cur], h->elem, (void* const*)cell, (void* const*)face, on_device);
  if (!rc) h->prims_valid = false;
  return rc;
}

extern "C" int mhd_get_state(mhd_handle* h, void* cell[5], void* face[3], int on_device) {
  if (!h) return MHD_ERR_INVALID;
  return copy_arrays(h, false, (char*)h->U[h->cur], h->elem, cell, face, on_device);
}

static cudaError_t record_event(mhd_handle* h) {
  if (h->ev_used == h->ev_pool.size()) {
    cudaEvent_t e;
    cudaError_t err = cudaEventCreate(&e);
    if (err) return err;
    h->ev_pool.push_back(e);
  }
  return cudaEventRecord(h->ev_pool[h->ev_used++], h->stream);
}

static StageArgs base_args(mhd_handle* h) {
  StageArgs a;
  memset(&a, 0, sizeof a);
  a.status = h->status;
  a.counters = h->counters;
  a.mlp = (const float*)h->mlp;
  a.mlp_zt = h->mlp_zt;
  return a;
}

// Primitives and CFL max of the current state (after set_state).
static cudaError_t ensure_prims(mhd_handle* h) {
  if (h->prims_valid) return cudaSuccess;
  StageArgs a = base_args(h);
  a.U = h->U[h->cur];
  a.Wout = h->W[h->cur];
  a.nextword = h->words + h->parity;
  cudaError_t e = cudaMemsetAsync(h->words + h->parity, 0, sizeof(unsigned long long), h->stream);
  if (e) return e;
  e = launch_prims(h->cfg.precision, h->stream, h->geo, a);
  if (e) return e;
  h->prims_valid = true;
  return cudaSuccess;
}

// One SSP-RK3 step: three stage launches, U^n -> U1 -> U2 -> U^{n+1}.  The
// primitives alternate W[cur] -> W[cur^1] -> W[cur] -> W[cur^1], so W[cur^1]
// holds those of U^{n+1} when cur flips.
static cudaError_t launch_step_rk3(mhd_handle* h, double dt) {
  const Geo& g = h->geo;
  const unsigned nblocks = (unsigned)(g.ntx * g.nty * g.nchunk);
  const int prec = h->cfg.precision;
  StageArgs a = base_args(h);
  a.dt = dt;
  a.dtword = h->words + h->parity;
  a.nextword = h->words + (h->parity ^ 1);
  a.U = h->U[h->cur];
  void* in[3] = {h->U[h->cur], h->Urk[0], h->Urk[1]};
  void* outs[3] = {h->Urk[0], h->Urk[1], h->U[h->cur ^ 1]};
  void* win[3] = {h->W[h->cur], h->W[h->cur ^ 1], h->W[h->cur]};
  void* wout[3] = {h->W[h->cur ^ 1], h->W[h->cur], h->W[h->cur ^ 1]};
  cudaError_t e = cudaSuccess;
  for (int s = 0; s < 3; ++s) {
    a.Uin = in[s];
    a.Uout = outs[s];
    a.Win = win[s];
    a.Wout = wout[s];
    if (h->profiling && (e = record_event(h))) return e;
    e = launch_stage(prec, ST_RK3_1 + s, g.TX, g.TY, nblocks, h->smem_bytes, h->stream, g, a, tma_for(h, a.Win));
    if (e) return e;
  }
  if (h->profiling && (e = record_event(h))) return e;
  h->cur ^= 1;
  h->parity ^= 1;
  return cudaSuccess;
}

static cudaError_t launch_step(mhd_handle* h, double dt) {
  const Geo& g = h->geo;
  const unsigned nblocks = (unsigned)(g.ntx * g.nty * g.nchunk);
  const int prec = h->cfg.precision;
  cudaError_t e = ensure_prims(h);
  if (e) return e;
  if (h->cfg.integrator == MHD_RK3) return launch_step_rk3(h, dt);
  StageArgs a = base_args(h);
  a.dt = dt;
  a.dtword = h->words + h->parity;
  a.nextword = h->words + (h->parity ^ 1);
  a.U = h->U[h->cur];
  a.Win = h->W[h->cur];
  a.K1out = h->K1;
  a.Wout = h->W[h->cur ^ 1];
  if (h->profiling && (e = record_event(h))) return e;
  e = launch_stage(prec, 1, g.TX, g.TY, nblocks, h->smem_bytes, h->stream, g, a, tma_for(h, a.Win));
  if (e) return e;
  if (h->profiling && (e = record_event(h))) return e;
  a.K1 = h->K1;
  a.K1out = nullptr;
  a.Win = h->W[h->cur ^ 1];
  a.Wout = h->W[h->cur];     // W(U^n) is dead once stage 1 has read it
  a.Uout = h->U[h->cur ^ 1];
  e = launch_stage(prec, 2, g.TX, g.TY, nblocks, h->smem_bytes, h->stream, g, a, tma_for(h, a.Win));
  if (e) return e;
  if (h->profiling && (e = record_event(h))) return e;
  // U^{n+1} is in U[cur^1] and its primitives in W[cur]: swap the W buffers
  // so that W[new cur] holds them
  void* t = h->W[0];
  h->W[0] = h->W[1];
  h->W[1] = t;
  h->cur ^= 1;
  h->parity ^= 1;
  return cudaSuccess;
}

static int need_switch(mhd_handle* h) {
  if (h->cfg.riemann == MHD_LEARNED && !h->mlp)
    return fail(h, MHD_ERR_INVALID, "riemann is MHD_LEARNED but no network was set (mhd_set_switch)");
  return MHD_OK;
}

static int enqueue_steps(mhd_handle* h, double dt, int nsteps) {
  if (int rc = need_switch(h)) return rc;
  for (int s = 0; s < nsteps; ++s) {
    cudaError_t e = launch_step(h, dt);
    if (e != cudaSuccess) return fail(h, MHD_ERR_CUDA, "stage launch failed: %s", cudaGetErrorString(e));
    h->steps++;
  }
  return MHD_OK;
}

static int read_words(mhd_handle* h) {
  unsigned long long* hp = (unsigned long long*)h->pinned;
  CUDA_TRY(h, cudaMemcpyAsync(hp, h->words, 16 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, h->stream));
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  return MHD_OK;
}

static int check_status(mhd_handle* h) {
  int rc = read_words(h);
  if (rc) return rc;
  unsigned st = *(unsigned*)((unsigned long long*)h->pinned + 3);
  if (st & ST_NONFINITE) return fail(h, MHD_ERR_NONFINITE, "non-finite state value met on the device");
  if (st & ST_TIMEOUT) return fail(h, MHD_ERR_TIMEOUT, "a device wait timed out (barrier or plane copy)");
  if (st & ST_BOUNDS) return fail(h, MHD_ERR_BOUNDS, "a kernel index left its array (bounds-checked build)");
  if (h->cfg.floor_policy == MHD_FLOOR_ERROR) {
    const unsigned long long* hp = (const unsigned long long*)h->pinned;
    unsigned long long hits = hp[8 + C_RHO_FLOOR] + hp[8 + C_P_FLOOR];
    if (hits > h->floors_seen) {
      unsigned long long rho = hp[8 + C_RHO_FLOOR], p = hp[8 + C_P_FLOOR];
      h->floors_seen = hits;
      return fail(h, MHD_ERR_FLOOR, "floors applied: %llu density and %llu pressure hits so far", rho, p);
    }
  }
  return MHD_OK;
}

// ---- host streaming ---------------------------------------------------------

static int stream_setup(mhd_handle* h) {
  if (h->s_in) return MHD_OK;
  const size_t bytes = (size_t)h->geo.total * h->elem;
  cudaError_t e = cudaSuccess;
  constexpr int NS = mhd_handle::kSlots;
  for (int p = 0; p < NS && e == cudaSuccess; ++p) {
    e = cudaMalloc(&h->slot_in[p], bytes);
    if (e == cudaSuccess) h->owned_states.push_back(h->slot_in[p]);
  }
  // the output slots: the handle's own two state buffers and further ones
  for (int p = 0; p < NS && e == cudaSuccess; ++p) {
    if (p < 2) {
      h->slot_out[p] = h->owned_states[p];
    } else {
      e = cudaMalloc(&h->slot_out[p], bytes);
      if (e == cudaSuccess) h->owned_states.push_back(h->slot_out[p]);
    }
  }
  for (int p = 0; p < NS && e == cudaSuccess; ++p) {
    e = cudaEventCreateWithFlags(&h->ev_h2d[p], cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_comp[p], cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_d2h[p], cudaEventDisableTiming);
  }
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&h->s_out, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&h->s_in, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    // undo this call's allocations, so that a later call starts afresh
    int code = e == cudaErrorMemoryAllocation ? MHD_ERR_NOMEM : MHD_ERR_CUDA;
    cudaGetLastError();
    for (int p = 0; p < NS; ++p) {
      if (h->ev_h2d[p]) cudaEventDestroy(h->ev_h2d[p]);
      if (h->ev_comp[p]) cudaEventDestroy(h->ev_comp[p]);
      if (h->ev_d2h[p]) cudaEventDestroy(h->ev_d2h[p]);
      h->ev_h2d[p] = h->ev_comp[p] = h->ev_d2h[p] = nullptr;
      h->slot_in[p] = h->slot_out[p] = nullptr;
    }
    if (h->s_out) cudaStreamDestroy(h->s_out);
    if (h->s_in) cudaStreamDestroy(h->s_in);
    h->s_out = h->s_in = nullptr;
    while (h->owned_states.size() > 2) {   // the first two are the handle's own state buffers
      cudaFree(h->owned_states.back());
      h->owned_states.pop_back();
    }
    return fail(h, code, "streaming setup failed: %s", cudaGetErrorString(e));
  }
  return MHD_OK;
}

static cudaError_t copy_state_async(const mhd_handle* h, bool in, char* dev, void* const* cell, void* const* face,
                                    cudaStream_t st) {
  const cudaMemcpyKind kind = in ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost;
  cudaError_t e = cudaSuccess;
  for (int v = 0; v < 5 && e == cudaSuccess; ++v) {
    char* d = dev + (size_t)v * h->geo.ncell * h->elem;
    const size_t n = (size_t)h->geo.ncell * h->elem;
    e = in ? cudaMemcpyAsync(d, cell[v], n, kind, st) : cudaMemcpyAsync(cell[v], d, n, kind, st);
  }
  for (int k = 0; k < 3 && e == cudaSuccess; ++k) {
    char* d = dev + (size_t)h->geo.face_off[k] * h->elem;
    const size_t n = (size_t)face_count(h->geo, k) * h->elem;
    e = in ? cudaMemcpyAsync(d, face[k], n, kind, st) : cudaMemcpyAsync(face[k], d, n, kind, st);
  }
  return e;
}

extern "C" int mhd_stream_step(mhd_handle* h, const void* const cell_in[5], const void* const face_in[3],
                               void* cell_out[5], void* face_out[3], double dt) {
  NvtxRange nvtx_range("mhd_stream_step");
  if (!h) return MHD_ERR_INVALID;
  if (!cell_in || !face_in || !cell_out || !face_out) return fail(h, MHD_ERR_INVALID, "null state pointer array");
  for (int v = 0; v < 5; ++v)
    if (!cell_in[v] || !cell_out[v]) return fail(h, MHD_ERR_INVALID, "null cell array %d", v);
  for (int k = 0; k < 3; ++k)
    if (!face_in[k] || !face_out[k]) return fail(h, MHD_ERR_INVALID, "null face array %d", k);
  if (dt != dt) return fail(h, MHD_ERR_INVALID, "dt is NaN");
  if (int rc = need_switch(h)) return rc;
  if (int rc = stream_setup(h)) return rc;
  const int p = (int)(h->nstream % mhd_handle::kSlots);
  // input: slot p is free once the step that read it (two back) has run
  CUDA_TRY(h, cudaStreamWaitEvent(h->s_in, h->ev_comp[p], 0));
  CUDA_TRY(h, copy_state_async(h, true, (char*)h->slot_in[p], (void* const*)cell_in, (void* const*)face_in, h->s_in));
  CUDA_TRY(h, cudaEventRecord(h->ev_h2d[p], h->s_in));
  // compute: after the input arrived and the output slot's previous copy-out
  CUDA_TRY(h, cudaStreamWaitEvent(h->stream, h->ev_h2d[p], 0));
  CUDA_TRY(h, cudaStreamWaitEvent(h->stream, h->ev_d2h[p], 0));
  h->U[h->cur] = h->slot_in[p];
  h->U[h->cur ^ 1] = h->slot_out[p];
  h->prims_valid = false;
  if (int rc = enqueue_steps(h, dt, 1)) return rc;
  if (dt > 0.0) h->last_dt = dt;
  CUDA_TRY(h, cudaEventRecord(h->ev_comp[p], h->stream));
  // output: the new state, now U[cur] = slot_out[p]
  CUDA_TRY(h, cudaStreamWaitEvent(h->s_out, h->ev_comp[p], 0));
  CUDA_TRY(h, copy_state_async(h, false, (char*)h->U[h->cur], cell_out, face_out, h->s_out));
  CUDA_TRY(h, cudaEventRecord(h->ev_d2h[p], h->s_out));
  h->nstream++;
  return MHD_OK;
}

extern "C" int mhd_stream_sync(mhd_handle* h) {
  if (!h) return MHD_ERR_INVALID;
  if (h->s_in) CUDA_TRY(h, cudaStreamSynchronize(h->s_in));
  if (h->s_out) CUDA_TRY(h, cudaStreamSynchronize(h->s_out));
  return check_status(h);
}

extern "C" int mhd_step_async(mhd_handle* h, double dt, int nsteps) {
  NvtxRange nvtx_range("mhd_step_async");
  if (!h) return MHD_ERR_INVALID;
  if (nsteps < 0) return fail(h, MHD_ERR_INVALID, "nsteps must be >= 0");
  if (dt != dt) return fail(h, MHD_ERR_INVALID, "dt is NaN");
  int rc = enqueue_steps(h, dt, nsteps);
  if (!rc && nsteps && dt > 0.0) h->last_dt = dt;
  return rc;
}

extern "C" int mhd_step(mhd_handle* h, double dt, int nsteps) {
  NvtxRange nvtx_range("mhd_step");
  if (!h) return MHD_ERR_INVALID;
  if (nsteps < 0) return fail(h, MHD_ERR_INVALID, "nsteps must be >= 0");
  if (dt != dt) return fail(h, MHD_ERR_INVALID, "dt is NaN");
  int rc = enqueue_steps(h, dt, nsteps);
  if (rc) return rc;
  rc = check_status(h);
  if (nsteps) {
    if (dt > 0.0) {
      h->last_dt = dt;
    } else {
      // the last step used the word of its starting state: parity ^ 1 now
      double m;
      unsigned long long bits = ((unsigned long long*)h->pinned)[h->parity ^ 1];
      memcpy(&m, &bits, sizeof m);
      h->last_dt = m > 0.0 ? h->cfg.cfl / m : 0.0;
    }
  }
  return rc;
}

extern "C" int mhd_rhs(mhd_handle* h, void* cell[5], void* face[3], int on_device) {
  NvtxRange nvtx_range("mhd_rhs");
  if (!h) return MHD_ERR_INVALID;
  if (int rc = need_switch(h)) return rc;
  cudaError_t e = ensure_prims(h);
  if (e) return fail(h, MHD_ERR_CUDA, "primitive recovery failed: %s", cudaGetErrorString(e));
  const Geo& g = h->geo;
  StageArgs a = base_args(h);
  a.dt = 1.0;                               // any dt > 0: only K1 = L(U) is kept
  a.dtword = h->words + h->parity;
  a.nextword = h->words + 4;                // scratch word, not the next step's
  a.U = h->U[h->cur];
  a.Win = h->W[h->cur];
  a.K1out = h->K1;
  a.Wout = nullptr;                         // no primitives of U + dt L
  e = launch_stage(h->cfg.precision, 1, g.TX, g.TY, (unsigned)(g.ntx * g.nty * g.nchunk), h->smem_bytes,
                   h->stream, g, a, tma_for(h, a.Win));
  if (e) return fail(h, MHD_ERR_CUDA, "stage launch failed: %s", cudaGetErrorString(e));
  int rc = copy_arrays(h, false, (char*)h->K1, h->kelem, cell, face, on_device);
  if (rc) return rc;
  return check_status(h);
}

extern "C" int mhd_set_profiling(mhd_handle* h, int on) {
  if (!h) return MHD_ERR_INVALID;
  h->profiling = on != 0;
  return MHD_OK;
}

extern "C" int mhd_get_profile(mhd_handle* h, double ms[3], long long launches[3]) {
  if (!h) return MHD_ERR_INVALID;
  if (!ms || !launches) return fail(h, MHD_ERR_INVALID, "null output pointer");
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  const size_t nst = h->cfg.integrator == MHD_RK3 ? 3 : 2;   // events per step: nst + 1
  for (int s = 0; s < 3; ++s) {
    ms[s] = 0.0;
    launches[s] = 0;
  }
  for (size_t i = 0; i + nst + 1 <= h->ev_used; i += nst + 1) {
    for (size_t s = 0; s < nst; ++s) {
      float t = 0.f;
      CUDA_TRY(h, cudaEventElapsedTime(&t, h->ev_pool[i + s], h->ev_pool[i + s + 1]));
      ms[s] += t;
      launches[s]++;
    }
  }
  h->ev_used = 0;
  return MHD_OK;
}

// ------------------------------------------------------------ reductions
// CFL dt of the current state and max |div B|, both in FP64.

__device__ __forceinline__ float mag32(float x) { return fabsf(x); }
__device__ __forceinline__ float mag32(double x) { return cut32(fabs(x)); }
__device__ __forceinline__ float signed32(float x) { return x; }
__device__ __forceinline__ float signed32(double x) { return copysignf(cut32(fabs(x)), __int_as_float(__double2hiint(x))); }

// FP32 upper bound of a cell's CFL speed sum, from its conserved values and
// faces: the sum grows with p and with every |B_d|, so both are raised by
// more than their rounding (1e-6 of the terms they are formed from; p
// subtracts the field at its lower end), and the rest is a few roundings (the
// factor at the end).  Infinity where FP32's exponent range does not hold the
// terms: energies near its end (a pressure formed from infinities could drop
// to its floor), densities and pressures near its ends, sound speeds below
// 1e-8 (whose fourth powers underflow), sums near its lower end (cells of 1e38
// across).  Fields that overflow make the sum infinite or NaN by themselves.
__device__ __forceinline__ float cfl_bound(const Geo& g, float rho, const float (&m)[3], float e, const float (&lo)[3],
                                           const float (&hi)[3]) {
  const float inf = __int_as_float(0x7f800000);
  rho = fmaxf(rho, g.frho_floor);
  const float ir = 1.0f / rho;
  float v[3], b2[3], mm = 0.f, bl = 0.f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float c = 0.5f * fabsf(lo[d] + hi[d]), err = 1e-6f * (fabsf(lo[d]) + fabsf(hi[d]));
    const float low = fmaxf(c - err, 0.f), high = c + err;
    v[d] = m[d] * ir;
    b2[d] = high * high * ir;
    mm += m[d] * m[d];
    bl += low * low;
  }
  const float kin = 0.5f * mm * ir, mag = 0.5f * bl, terms = fabsf(e) + kin + mag;
  float p = g.fgm1 * (fabsf(e) * 1.000001f - kin - mag + 4e-6f * terms);
  p = fmaxf(p, g.fp_floor * 1.000001f);
  const float a2 = g.fgamma * p * ir;
  if (!(terms < 1e37f && rho > 1e-30f && rho < 1e30f && p > 1e-30f && p < 1e30f && a2 > 1e-16f)) return inf;
  const float sum = signal_sum(g, v, a2, b2);
  return sum > 1e-30f ? sum * 1.00001f : inf;
}

// The speed sum in FP64 (signal_sum from conserved values, with the division
// by rho taken out of the roots): the three fast speeds share a^2, b^2 and their
// difference, c_f,d^2 = (a^2 + b^2 + sqrt((a^2 - b^2)^2 + 4 a^2 b_t,d^2)) / 2.
__device__ __forceinline__ double cfl_sum(const Geo& g, double rho, const double (&m)[3], double e,
                                          const double (&b)[3]) {
  if (rho < g.rho_floor) rho = g.rho_floor;   // (not lt_: a cell with a NaN of either sign stays out of the maximum)
  const double ir = qrcp_(rho);
  const double b2[3] = {b[0] * b[0], b[1] * b[1], b[2] * b[2]};
  const double bb = b2[0] + b2[1] + b2[2];
  double p = g.gm1 * (e - 0.5 * (m[0] * m[0] + m[1] * m[1] + m[2] * m[2]) * ir - 0.5 * bb);
  if (p < g.p_floor) p = g.p_floor;
  const double gp = g.gamma * p, a2 = gp * ir, q = bb * ir, x = a2 - q, s = a2 + q, xx = x * x, a4r = 4.0 * a2 * ir;
  double sum = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (g.n[d] > 1) {
      const double root = qroot_(xx + a4r * (b2[(d + 1) % 3] + b2[(d + 2) % 3]));
      sum += (fabs(m[d]) * ir + qroot_(0.5 * (s + root))) * g.inv_d[d];
    }
  }
  return sum;
}

// CFL maximum.  The FP64 sum (~70 operations of a pipe that takes ~17 cycles
// for each) is formed only by warps with a cell whose FP32 bound is not below
// the largest sum found so far, which every warp reads before a run.
// Measured (GB300), a call with its synchronisation: 256^3 mixed 480 us (4742 with
// every sum in FP64 and IEEE divides), 97x130x75 FP32 68 (424).
template <typename S>
__global__ void __launch_bounds__(256) cfl_kernel(Geo g, const S* U, unsigned long long* word, int run) {
  const int lane = threadIdx.x & 31;
  const int per_row = (g.n[0] + run - 1) / run;
  const long long items = (long long)g.n[1] * g.n[2] * per_row;
  const long long nwarps = (long long)gridDim.x * (blockDim.x / 32);
  for (long long item = blockIdx.x * (long long)(blockDim.x / 32) + threadIdx.x / 32; item < items; item += nwarps) {
    const RowRun r = row_run(g, item, per_row, run);
    double top = __longlong_as_double((long long)*(volatile unsigned long long*)word);
    for (int base = r.i0; base < r.i1; base += 32) {
      const int i = base + lane;
      const bool valid = i < r.i1;
      S u[5], lo[3], hi[3];
      float bound = 0.0f;
      if (valid) {
#pragma unroll
        for (int v = 0; v < 5; ++v) u[v] = U[v * g.ncell + r.cell + i];
        lo[0] = U[r.x + i];
        hi[0] = U[r.x + (i + 1 < g.nf[0] ? i + 1 : 0)];
        lo[1] = U[r.ylo + i];
        hi[1] = U[r.yhi + i];
        lo[2] = U[r.zlo + i];
        hi[2] = U[r.zhi + i];
        const float m[3] = {mag32(u[1]), mag32(u[2]), mag32(u[3])};
        const float l[3] = {signed32(lo[0]), signed32(lo[1]), signed32(lo[2])};
        const float h[3] = {signed32(hi[0]), signed32(hi[1]), signed32(hi[2])};
        bound = cfl_bound(g, signed32(u[0]), m, signed32(u[4]), l, h);
      }
      // (cut32 rounds top down; a bound or sum that is not a number is formed in FP64)
      const bool need = valid && !(bound < cut32(top));
      if (!__any_sync(0xffffffffu, need)) continue;
      double sum = 0.0;
      if (need) {
        const double m[3] = {to_f64(u[1]), to_f64(u[2]), to_f64(u[3])};
        const double b[3] = {0.5 * (to_f64(lo[0]) + to_f64(hi[0])), 0.5 * (to_f64(lo[1]) + to_f64(hi[1])),
                             0.5 * (to_f64(lo[2]) + to_f64(hi[2]))};
        sum = cfl_sum(g, to_f64(u[0]), m, to_f64(u[4]), b);
      }
      double w = sum > 0.0 ? sum : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) w = fmax(w, __shfl_xor_sync(0xffffffffu, w, o));
      if (w > top) {
        top = w;
        if (lane == 0) atomicMax(word, (unsigned long long)__double_as_longlong(w));
      }
    }
  }
}

template <typename S>
__global__ void __launch_bounds__(256) divb_kernel(Geo g, const S* U, unsigned long long* word, int run) {
  const int lane = threadIdx.x & 31;
  const int per_row = (g.n[0] + run - 1) / run;
  const long long items = (long long)g.n[1] * g.n[2] * per_row;
  const long long nwarps = (long long)gridDim.x * (blockDim.x / 32);
  long long m = 0;   // bits of the largest |div B|; non-negative doubles order as integers
  for (long long item = blockIdx.x * (long long)(blockDim.x / 32) + threadIdx.x / 32; item < items; item += nwarps) {
    const RowRun r = row_run(g, item, per_row, run);
    for (int i = r.i0 + lane; i < r.i1; i += 32) {
      const double div = (to_f64(U[r.x + (i + 1 < g.nf[0] ? i + 1 : 0)]) - to_f64(U[r.x + i])) * g.inv_d[0] +
                         (to_f64(U[r.yhi + i]) - to_f64(U[r.ylo + i])) * g.inv_d[1] +
                         (to_f64(U[r.zhi + i]) - to_f64(U[r.zlo + i])) * g.inv_d[2];
      const long long v = __double_as_longlong(fabs(div));
      if (v <= 0x7ff0000000000000LL && v > m) m = v;   // cells that hold a NaN stay out
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0 && m > 0) atomicMax(word, (unsigned long long)m);
}

static int reduce_word(mhd_handle* h, bool cfl, double* out) {
  if (!h) return MHD_ERR_INVALID;
  if (!out) return fail(h, MHD_ERR_INVALID, "null output pointer");
  unsigned long long* word = h->words + 2;
  CUDA_TRY(h, cudaMemsetAsync(word, 0, sizeof(unsigned long long), h->stream));
  const int run = row_run_length(h->geo);
  const unsigned blocks = row_run_blocks(h->geo, run);
  if (h->elem == 8) {
    const double* U = (const double*)h->U[h->cur];
    if (cfl) cfl_kernel<double><<<blocks, 256, 0, h->stream>>>(h->geo, U, word, run);
    else divb_kernel<double><<<blocks, 256, 0, h->stream>>>(h->geo, U, word, run);
  } else {
    const float* U = (const float*)h->U[h->cur];
    if (cfl) cfl_kernel<float><<<blocks, 256, 0, h->stream>>>(h->geo, U, word, run);
    else divb_kernel<float><<<blocks, 256, 0, h->stream>>>(h->geo, U, word, run);
  }
  CUDA_TRY(h, cudaGetLastError());
  unsigned long long* hp = (unsigned long long*)h->pinned;
  CUDA_TRY(h, cudaMemcpyAsync(hp, word, sizeof(unsigned long long), cudaMemcpyDeviceToHost, h->stream));
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  double m;
  memcpy(&m, hp, sizeof m);
  *out = cfl ? (m > 0.0 ? h->cfg.cfl / m : 0.0) : m;
  return MHD_OK;
}

extern "C" int mhd_cfl_dt(mhd_handle* h, double* dt_out) { return reduce_word(h, true, dt_out); }
extern "C" int mhd_divb_max(mhd_handle* h, double* out) { return reduce_word(h, false, out); }

extern "C" int mhd_get_stats(mhd_handle* h, mhd_stats* out) {
  if (!h) return MHD_ERR_INVALID;
  if (!out) return fail(h, MHD_ERR_INVALID, "null output pointer");
  int rc = read_words(h);
  if (rc) return rc;
  unsigned long long* hp = (unsigned long long*)h->pinned;
  memset(out, 0, sizeof *out);
  out->status = (int)*(unsigned*)(hp + 3);
  out->rho_floor_hits = (long long)hp[8 + C_RHO_FLOOR];
  out->p_floor_hits = (long long)hp[8 + C_P_FLOOR];
  out->faces_hll = (long long)hp[8 + C_HLL];
  out->faces_hlld = (long long)hp[8 + C_HLLD];
  out->last_dt = h->last_dt;
  out->steps = h->steps;
  out->tma_planes = (long long)hp[8 + C_TMA];
  return MHD_OK;
}

// =====================================================================
// Batched persistent launch
// =====================================================================

namespace mhd {
cudaError_t batch_launch_fp64(int, int, unsigned, size_t, cudaStream_t, const BatchArgs&);
cudaError_t batch_launch_mixed(int, int, unsigned, size_t, cudaStream_t, const BatchArgs&);
cudaError_t batch_launch_fp32(int, int, unsigned, size_t, cudaStream_t, const BatchArgs&);
cudaError_t batch_set_smem_fp64(int, int, size_t);
cudaError_t batch_set_smem_mixed(int, int, size_t);
cudaError_t batch_set_smem_fp32(int, int, size_t);
int batch_max_blocks_fp64(int, int, size_t);
size_t batch_smem_bytes_fp64(int, int);
size_t batch_smem_bytes_mixed(int, int);
size_t batch_smem_bytes_fp32(int, int);
int batch_max_blocks_mixed(int, int, size_t);
int batch_max_blocks_fp32(int, int, size_t);
cudaError_t batch_prims_fp64(unsigned, cudaStream_t, BoxDesc*, const BoxSet&, int, unsigned*, unsigned long long*);
cudaError_t batch_prims_mixed(unsigned, cudaStream_t, BoxDesc*, const BoxSet&, int, unsigned*, unsigned long long*);
cudaError_t batch_prims_fp32(unsigned, cudaStream_t, BoxDesc*, const BoxSet&, int, unsigned*, unsigned long long*);
static cudaError_t batch_prims(int prec, unsigned blocks, cudaStream_t st, BoxDesc* boxes, const BoxSet& set, int run,
                               unsigned* status, unsigned long long* counters) {
  switch (prec) {
    case P_FP64: return batch_prims_fp64(blocks, st, boxes, set, run, status, counters);
    case P_MIXED: return batch_prims_mixed(blocks, st, boxes, set, run, status, counters);
    default: return batch_prims_fp32(blocks, st, boxes, set, run, status, counters);
  }
}

cudaError_t batch_launch(int prec, int tx, int ty, unsigned grid, size_t smem, cudaStream_t st, const BatchArgs& ba) {
  switch (prec) {
    case P_FP64: return batch_launch_fp64(tx, ty, grid, smem, st, ba);
    case P_MIXED: return batch_launch_mixed(tx, ty, grid, smem, st, ba);
    default: return batch_launch_fp32(tx, ty, grid, smem, st, ba);
  }
}
cudaError_t batch_set_smem(int prec, int tx, int ty, size_t bytes) {
  switch (prec) {
    case P_FP64: return batch_set_smem_fp64(tx, ty, bytes);
    case P_MIXED: return batch_set_smem_mixed(tx, ty, bytes);
    default: return batch_set_smem_fp32(tx, ty, bytes);
  }
}
static size_t batch_smem_bytes(int prec, int tx, int ty) {
  switch (prec) {
    case P_FP64: return batch_smem_bytes_fp64(tx, ty);
    case P_MIXED: return batch_smem_bytes_mixed(tx, ty);
    default: return batch_smem_bytes_fp32(tx, ty);
  }
}
int batch_max_blocks_per_sm(int prec, int tx, int ty, size_t smem) {
  switch (prec) {
    case P_FP64: return batch_max_blocks_fp64(tx, ty, smem);
    case P_MIXED: return batch_max_blocks_mixed(tx, ty, smem);
    default: return batch_max_blocks_fp32(tx, ty, smem);
  }
}
}  // namespace mhd

struct mhd_batch {
  int nbox = 0;
  int prec = 0;
  std::vector<mhd_config> cfg;
  std::vector<BoxDesc> box;          // host mirror
  BoxDesc* dbox = nullptr;           // device copy
  ItemRef* dorder = nullptr;         // device item list, longest first
  size_t dorder_cap = 0;             // its capacity in entries
  std::vector<size_t> ubytes, kbytes, wbytes;
  std::vector<bool> prims_valid;
  void* pool = nullptr;              // all per-box buffers
  unsigned long long* words = nullptr;   // [0..63] general, then 2 per box
  unsigned* bar_count = nullptr;
  unsigned long long* work = nullptr;    // item draws of one launch
  unsigned* status = nullptr;
  unsigned long long* counters = nullptr;
  void* pinned = nullptr;
  cudaStream_t stream = nullptr;     // caller's stream
  cudaStream_t cap = nullptr;        // private stream for graph capture
  int tx = 16, ty = 8, tz = 32;
  size_t smem = 0;
  unsigned grid = 0;
  long long total_items = 0;
  double timeout_s = 2.0;
  int skip_arrival = 0;
  bool use_graph = true;
  cudaGraphExec_t gexec = nullptr;
  double g_dt = 0.0;
  int g_nsteps = -1;
  int steps = 0;
  std::string err;
};

static thread_local std::string g_batch_err;   // error text of batch calls without a handle, per host thread

static int bfail(mhd_batch* b, int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  if (b) b->err = buf; else g_batch_err = buf;
  return code;
}

#define BCUDA_TRY(b, call)                                                                \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess)                                                                \
      return bfail((b), MHD_ERR_CUDA, "%s failed: %s", #call, cudaGetErrorString(e_));    \
  } while (0)

static void drop_graph(mhd_batch* b) {
  if (b->gexec) cudaGraphExecDestroy(b->gexec);
  b->gexec = nullptr;
  b->g_nsteps = -1;
}

// Default planes per z-chunk of a batch: the length whose items, started
// longest first, take the least estimated time, if that is under 0.98 of 32's
// (measured, FP32, us a stage: 64 boxes of 32-128 cells an axis 4690 at 32,
// 4598 at 96; 4 boxes of 32-112 365 at 32, 198 at 8).  An item's prologue also
// draws its ticket and gathers its planes without TMA: 2.5 planes.
static int batch_default_chunk(const mhd_batch* b, int tx, int ty) {
  static const int lengths[] = {32, 2, 4, 6, 8, 12, 16, 24, 48, 64, 96, 128};
  MarchRates rates = march_rates(b->prec == MHD_FP64, resident_ctas(&b->cfg[0], tx, ty));
  if (b->prec != MHD_FP64) rates.prologue = 2.5;
  int best = 32;
  double least = HUGE_VAL;
  for (int tz : lengths) {
    std::map<int, long long, std::greater<int>> count;   // chunks by planes, longest first
    long long items = 0;
    for (const mhd_config& c : b->cfg) {
      const long long columns = (long long)((c.nx + tx - 1) / tx) * ((c.ny + ty - 1) / ty);
      const int n = (c.nz + tz - 1) / tz;
      if (n > 1) count[tz] += columns * (n - 1);
      count[c.nz - (n - 1) * tz] += columns;
      items += columns * n;
    }
    if (tz < 16 && items > 40LL * kSMs * rates.most) continue;
    std::vector<ChunkGroup> groups;
    for (const auto& q : count) groups.push_back({q.first, q.second});
    const double t = march_time(groups.data(), groups.size(), rates);
    if (tz == 32) least = 0.98 * t;
    else if (t < least) {
      least = t;
      best = tz;
    }
  }
  return best;
}

// Recompute per-box geometry, work items, shared memory and the persistent
// grid for tile (tx, ty, tz), and upload the box table.
static int batch_apply_tile(mhd_batch* b, int tx, int ty, int tz) {
  if (!stage_tile_supported(b->prec, tx, ty) || batch_max_blocks_per_sm(b->prec, tx, ty, 0) < 0)
    return bfail(b, MHD_ERR_INVALID, "tile %dx%d not available for the batch kernel", tx, ty);
  const size_t smem = batch_smem_bytes(b->prec, tx, ty);
  if (smem == 0 || smem > 227 * 1024) return bfail(b, MHD_ERR_INVALID, "tile %dx%d not available", tx, ty);
  cudaError_t e = batch_set_smem(b->prec, tx, ty, smem);
  if (e) return bfail(b, MHD_ERR_INVALID, "tile %dx%d is not instantiated for the batch kernel: %s", tx, ty,
                      cudaGetErrorString(e));
  int per_sm = batch_max_blocks_per_sm(b->prec, tx, ty, smem);
  if (per_sm < 1) return bfail(b, MHD_ERR_INVALID, "tile %dx%d cannot be resident", tx, ty);
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  long long item = 0;
  for (int i = 0; i < b->nbox; ++i) {
    mhd_config c = b->cfg[i];
    c.tile_x = tx; c.tile_y = ty; c.tile_z = tz;
    fill_geo(&c, &b->box[i].g);
    b->box[i].item_begin = item;
    b->box[i].nitems = b->box[i].g.ntx * b->box[i].g.nty * b->box[i].g.nchunk;
    item += b->box[i].nitems;
  }
  b->total_items = item;
  // the item list, longest first: a chunk's cost grows with its planes plus
  // the three-plane prologue of its z-march (ties keep box order)
  std::vector<std::pair<int, ItemRef>> items;
  items.reserve((size_t)item);
  for (int i = 0; i < b->nbox; ++i) {
    const Geo& g = b->box[i].g;
    const int per_chunk = g.ntx * g.nty;
    for (int l = 0; l < b->box[i].nitems; ++l) {
      const int kb = (l / per_chunk) * g.TZ;
      const int ke = kb + g.TZ < g.n[2] ? kb + g.TZ : g.n[2];
      items.push_back({ke - kb + 3, ItemRef{i, l}});
    }
  }
  std::stable_sort(items.begin(), items.end(),
                   [](const std::pair<int, ItemRef>& x, const std::pair<int, ItemRef>& y) { return x.first > y.first; });
  std::vector<ItemRef> order(items.size());
  for (size_t q = 0; q < items.size(); ++q) order[q] = items[q].second;
  if (order.size() > b->dorder_cap) {
    drop_graph(b);
    cudaFree(b->dorder);
    b->dorder = nullptr;
    b->dorder_cap = 0;
    BCUDA_TRY(b, cudaMalloc(&b->dorder, order.size() * sizeof(ItemRef)));
    b->dorder_cap = order.size();
  }
  BCUDA_TRY(b, cudaMemcpyAsync(b->dorder, order.data(), order.size() * sizeof(ItemRef), cudaMemcpyHostToDevice,
                               b->stream));
  b->tx = tx; b->ty = ty; b->tz = tz;
  b->smem = smem;
  b->grid = (unsigned)(per_sm * nsm);
  BCUDA_TRY(b, cudaMemcpyAsync(b->dbox, b->box.data(), sizeof(BoxDesc) * b->nbox, cudaMemcpyHostToDevice, b->stream));
  BCUDA_TRY(b, cudaStreamSynchronize(b->stream));
  drop_graph(b);
  return MHD_OK;
}

extern "C" void mhd_batch_destroy(mhd_batch* b) {
  if (!b) return;
  if (b->stream) cudaStreamSynchronize(b->stream); else cudaDeviceSynchronize();
  drop_graph(b);
  if (b->cap) cudaStreamDestroy(b->cap);
  cudaFree(b->pool);
  cudaFree(b->words);
  cudaFree(b->dbox);
  cudaFree(b->dorder);
  if (b->pinned) cudaFreeHost(b->pinned);
  delete b;
}

extern "C" const char* mhd_batch_last_error(const mhd_batch* b) { return b ? b->err.c_str() : g_batch_err.c_str(); }

extern "C" int mhd_batch_create(int nbox, const mhd_config* cfgs, void* cuda_stream, mhd_batch** out) {
  if (!out || !cfgs || nbox < 1) return bfail(nullptr, MHD_ERR_INVALID, "need nbox >= 1, configs and an output pointer");
  for (int i = 0; i < nbox; ++i) {
    int rc = validate(&cfgs[i], nullptr);
    if (rc) return bfail(nullptr, rc, "box %d: %s", i, g_create_err.c_str());
    if (cfgs[i].precision != cfgs[0].precision || cfgs[i].riemann != cfgs[0].riemann || cfgs[i].emf != cfgs[0].emf)
      return bfail(nullptr, MHD_ERR_INVALID, "all boxes of a batch share precision, Riemann solver and EMF mode");
    if (cfgs[i].riemann == MHD_LEARNED)
      return bfail(nullptr, MHD_ERR_INVALID, "batches solve with HLLD or HLL; the learned switch is single-box only");
    if (cfgs[i].integrator != MHD_RK2)
      return bfail(nullptr, MHD_ERR_INVALID, "batches step with the RK2 integrator; SSP-RK3 is single-box only");
    if (cfgs[i].recon != MHD_RECON_PRIMITIVE)
      return bfail(nullptr, MHD_ERR_INVALID, "batches reconstruct the primitives; characteristic PLM is single-box only");
  }
  mhd_batch* b = new (std::nothrow) mhd_batch();
  if (!b) return bfail(nullptr, MHD_ERR_NOMEM, "host allocation failed");
  b->nbox = nbox;
  b->prec = cfgs[0].precision;
  b->cfg.assign(cfgs, cfgs + nbox);
  b->box.resize(nbox);
  b->prims_valid.assign(nbox, false);
  b->stream = (cudaStream_t)cuda_stream;
  const size_t elem = b->prec == MHD_FP32 ? 4 : 8, kelem = b->prec == MHD_FP64 ? 8 : 4, welem = kelem;
  size_t total = 0;
  auto take = [&](size_t n) { size_t o = total; total += (n + 255) / 256 * 256; return o; };
  std::vector<size_t> off(5 * nbox);
  for (int i = 0; i < nbox; ++i) {
    Geo g;
    fill_geo(&cfgs[i], &g);
    off[5 * i + 0] = take((size_t)g.total * elem);
    off[5 * i + 1] = take((size_t)g.total * elem);
    off[5 * i + 2] = take((size_t)g.total * kelem);
    off[5 * i + 3] = take((size_t)g.ncell * NW * welem);
    off[5 * i + 4] = take((size_t)g.ncell * NW * welem);
    b->ubytes.push_back((size_t)g.total * elem);
    b->kbytes.push_back((size_t)g.total * kelem);
    b->wbytes.push_back((size_t)g.ncell * NW * welem);
  }
  cudaError_t e = cudaMalloc(&b->pool, total);
  if (e == cudaSuccess) e = cudaMalloc(&b->words, (64 + 2 * (size_t)nbox) * sizeof(unsigned long long));
  if (e == cudaSuccess) e = cudaMalloc(&b->dbox, sizeof(BoxDesc) * nbox);
  if (e == cudaSuccess) e = cudaMallocHost(&b->pinned, 64 * sizeof(unsigned long long) + 8 * (size_t)nbox * 2);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    int code = e == cudaErrorMemoryAllocation ? MHD_ERR_NOMEM : MHD_ERR_CUDA;
    bfail(nullptr, code, "batch allocation of %zu B failed: %s", total, cudaGetErrorString(e));
    cudaGetLastError();
    mhd_batch_destroy(b);
    return code;
  }
  b->bar_count = (unsigned*)(b->words + 0);
  b->work = b->words + 1;
  b->status = (unsigned*)(b->words + 3);
  b->counters = b->words + 8;
  char* pool = (char*)b->pool;
  for (int i = 0; i < nbox; ++i) {
    BoxDesc& d = b->box[i];
    memset(&d, 0, sizeof d);
    d.U[0] = pool + off[5 * i + 0];
    d.U[1] = pool + off[5 * i + 1];
    d.K1 = pool + off[5 * i + 2];
    d.W[0] = pool + off[5 * i + 3];
    d.W[1] = pool + off[5 * i + 4];
    d.words = b->words + 64 + 2 * i;
  }
  e = cudaMemsetAsync(b->words, 0, (64 + 2 * (size_t)nbox) * sizeof(unsigned long long), b->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(b->pool, 0, total, b->stream);
  if (e != cudaSuccess) {
    bfail(nullptr, MHD_ERR_CUDA, "batch initialisation failed: %s", cudaGetErrorString(e));
    mhd_batch_destroy(b);
    return MHD_ERR_CUDA;
  }
  int tx, ty;
  resolve_tile(&cfgs[0], &tx, &ty);
  int rc = batch_apply_tile(b, tx, ty, cfgs[0].tile_z ? cfgs[0].tile_z : batch_default_chunk(b, tx, ty));
  if (rc) {
    g_batch_err = b->err;
    mhd_batch_destroy(b);
    return rc;
  }
  *out = b;
  return MHD_OK;
}

static int batch_copy(mhd_batch* b, int i, bool in, void* const* cell, void* const* face, int on_device) {
  if (!b) return MHD_ERR_INVALID;
  if (i < 0 || i >= b->nbox) return bfail(b, MHD_ERR_INVALID, "box index %d out of range", i);
  if (!cell || !face) return bfail(b, MHD_ERR_INVALID, "null state pointer array");
  const Geo& g = b->box[i].g;
  const size_t elem = b->prec == MHD_FP32 ? 4 : 8;
  char* base = (char*)b->box[i].U[b->box[i].cur];
  for (int v = 0; v < 5; ++v)
    if (!cell[v]) return bfail(b, MHD_ERR_INVALID, "null cell array %d", v);
  for (int d = 0; d < 3; ++d)
    if (!face[d]) return bfail(b, MHD_ERR_INVALID, "null face array %d", d);
  if (on_device) {
    BCUDA_TRY(b, copy_state_on_device(g, in, base, elem, cell, face, b->stream));
    if (!in) BCUDA_TRY(b, cudaStreamSynchronize(b->stream));
  } else {
    const cudaMemcpyKind kind = in ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost;
    for (int q = 0; q < 8; ++q) {
      char* dev = base + (size_t)(q < 5 ? q * g.ncell : g.face_off[q - 5]) * elem;
      const size_t n = (size_t)(q < 5 ? g.ncell : face_count(g, q - 5)) * elem;
      void* user = q < 5 ? cell[q] : face[q - 5];
      BCUDA_TRY(b, in ? cudaMemcpyAsync(dev, user, n, kind, b->stream) : cudaMemcpyAsync(user, dev, n, kind, b->stream));
    }
    BCUDA_TRY(b, cudaStreamSynchronize(b->stream));
  }
  if (in) b->prims_valid[i] = false;
  return MHD_OK;
}

extern "C" int mhd_batch_set_state(mhd_batch* b, int box, const void* const cell[5], const void* const face[3],
                                   int on_device) {
  return batch_copy(b, box, true, (void* const*)cell, (void* const*)face, on_device);
}

extern "C" int mhd_batch_get_state(mhd_batch* b, int box, void* cell[5], void* face[3], int on_device) {
  return batch_copy(b, box, false, cell, face, on_device);
}

// Primitives and CFL maxima of the boxes whose state was set from outside: one
// launch for up to 1024 boxes (and one that clears their CFL words).
static int batch_ensure_prims(mhd_batch* b) {
  for (int first = 0; first < b->nbox; first += BoxSet::kMost) {
    BoxSet set = {};
    set.first = first;
    set.count = std::min(b->nbox - first, (int)BoxSet::kMost);
    long long runs = 0, widest = 0;
    for (int i = 0; i < set.count; ++i) {
      if (b->prims_valid[first + i]) continue;
      const Geo& g = b->box[first + i].g;
      set.bits[i / 32] |= 1u << (i % 32);
      const long long n = (long long)g.n[1] * g.n[2] * ((g.n[0] + 127) / 128);
      runs += n;
      widest = std::max(widest, n);
    }
    if (!runs) continue;
    const int run = runs >= 152LL * 64 ? 128 : 32;   // as row_run_length for one box
    if (run == 32) widest *= 4;
    // enough blocks a box for its runs, no more in all than a few per SM
    const long long most = std::max(1LL, 152LL * 16 / set.count);
    const unsigned blocks = (unsigned)std::min(most, (widest + 7) / 8);
    BCUDA_TRY(b, batch_prims(b->prec, blocks, b->stream, b->dbox, set, run, b->status, b->counters));
    for (int i = 0; i < set.count; ++i) b->prims_valid[first + i] = true;
  }
  return MHD_OK;
}

static BatchArgs batch_args(mhd_batch* b, double dt, int nsteps) {
  BatchArgs ba;
  memset(&ba, 0, sizeof ba);
  ba.boxes = b->dbox;
  ba.nbox = b->nbox;
  ba.total_items = b->total_items;
  ba.order = b->dorder;
  ba.work = b->work;
  ba.nsteps = nsteps;
  ba.dt = dt;
  ba.bar_count = b->bar_count;
  ba.status = b->status;
  ba.counters = b->counters;
  ba.timeout_ns = (unsigned long long)(b->timeout_s * 1e9);
  ba.skip_arrival = b->skip_arrival;
  return ba;
}

// One persistent launch of nsteps steps for every box (enqueue only).
static int batch_enqueue(mhd_batch* b, double dt, int nsteps) {
  int rc = batch_ensure_prims(b);
  if (rc) return rc;
  const BatchArgs ba = batch_args(b, dt, nsteps);
  const bool graph = b->use_graph && !b->skip_arrival;
  if (graph && !(b->gexec && b->g_dt == dt && b->g_nsteps == nsteps)) {
    drop_graph(b);
    cudaGraph_t gr = nullptr;
    BCUDA_TRY(b, cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal));
    cudaError_t e = cudaMemsetAsync(b->words, 0, 2 * sizeof(unsigned long long), b->cap);   // barrier, draws
    if (e == cudaSuccess) e = batch_launch(b->prec, b->tx, b->ty, b->grid, b->smem, b->cap, ba);
    if (e == cudaSuccess) {
      batch_advance<<<(b->nbox + 127) / 128, 128, 0, b->cap>>>(b->dbox, b->nbox, nsteps);
      e = cudaGetLastError();
    }
    cudaError_t e2 = cudaStreamEndCapture(b->cap, &gr);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->gexec, gr, 0);
    if (gr) cudaGraphDestroy(gr);
    if (e != cudaSuccess) {
      drop_graph(b);
      cudaGetLastError();
      return bfail(b, MHD_ERR_CUDA, "graph capture of the persistent launch failed: %s", cudaGetErrorString(e));
    }
    b->g_dt = dt;
    b->g_nsteps = nsteps;
  }
  if (graph) {
    BCUDA_TRY(b, cudaGraphLaunch(b->gexec, b->stream));
  } else {
    BCUDA_TRY(b, cudaMemsetAsync(b->words, 0, 2 * sizeof(unsigned long long), b->stream));   // barrier, draws
    BCUDA_TRY(b, batch_launch(b->prec, b->tx, b->ty, b->grid, b->smem, b->stream, ba));
    batch_advance<<<(b->nbox + 127) / 128, 128, 0, b->stream>>>(b->dbox, b->nbox, nsteps);
    BCUDA_TRY(b, cudaGetLastError());
  }
  for (int i = 0; i < b->nbox; ++i) {
    b->box[i].cur = (b->box[i].cur + nsteps) & 1;
    b->box[i].parity = (b->box[i].parity + nsteps) & 1;
  }
  b->steps += nsteps;
  return MHD_OK;
}

static int batch_check(mhd_batch* b) {
  unsigned long long* hp = (unsigned long long*)b->pinned;
  BCUDA_TRY(b, cudaMemcpyAsync(hp, b->words, 16 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, b->stream));
  BCUDA_TRY(b, cudaStreamSynchronize(b->stream));
  const unsigned st = *(unsigned*)(hp + 3);
  if (st & (ST_TIMEOUT | ST_NONFINITE | ST_BOUNDS)) {
    // report once, then clear so that the handle can be reused
    BCUDA_TRY(b, cudaMemsetAsync(b->status, 0, sizeof(unsigned), b->stream));
    BCUDA_TRY(b, cudaStreamSynchronize(b->stream));
    if (st & ST_TIMEOUT) return bfail(b, MHD_ERR_TIMEOUT, "device-wide barrier of the persistent launch timed out");
    if (st & ST_BOUNDS) return bfail(b, MHD_ERR_BOUNDS, "a kernel index left its array (bounds-checked build)");
    return bfail(b, MHD_ERR_NONFINITE, "non-finite state value met on the device");
  }
  return MHD_OK;
}

extern "C" int mhd_batch_step_async(mhd_batch* b, double dt, int nsteps) {
  NvtxRange nvtx_range("mhd_batch_step_async");
  if (!b) return MHD_ERR_INVALID;
  if (nsteps < 1) return bfail(b, MHD_ERR_INVALID, "nsteps must be >= 1");
  if (dt != dt) return bfail(b, MHD_ERR_INVALID, "dt is NaN");
  return batch_enqueue(b, dt, nsteps);
}

extern "C" int mhd_batch_step(mhd_batch* b, double dt, int nsteps) {
  NvtxRange nvtx_range("mhd_batch_step");
  int rc = mhd_batch_step_async(b, dt, nsteps);
  if (rc) return rc;
  return batch_check(b);
}

extern "C" int mhd_batch_set_tile(mhd_batch* b, int tx, int ty, int tz) {
  if (!b) return MHD_ERR_INVALID;
  if (tz < 1) return bfail(b, MHD_ERR_INVALID, "tile_z must be >= 1");
  BCUDA_TRY(b, cudaStreamSynchronize(b->stream));
  return batch_apply_tile(b, tx, ty, tz);
}

extern "C" int mhd_batch_get_tile(mhd_batch* b, int tile[3], long long* items, int* grid) {
  if (!b || !tile) return MHD_ERR_INVALID;
  tile[0] = b->tx; tile[1] = b->ty; tile[2] = b->tz;
  if (items) *items = b->total_items;
  if (grid) *grid = (int)b->grid;
  return MHD_OK;
}

extern "C" int mhd_batch_set_barrier_timeout(mhd_batch* b, double seconds) {
  if (!b) return MHD_ERR_INVALID;
  if (!(seconds > 0.0)) return bfail(b, MHD_ERR_INVALID, "timeout must be positive");
  b->timeout_s = seconds;
  drop_graph(b);
  return MHD_OK;
}

extern "C" int mhd_batch_inject_missed_arrival(mhd_batch* b, int on) {
  if (!b) return MHD_ERR_INVALID;
  b->skip_arrival = on != 0;
  drop_graph(b);
  return MHD_OK;
}

extern "C" int mhd_batch_box_dt(mhd_batch* b, int box, double* dt_out) {
  if (!b || !dt_out) return MHD_ERR_INVALID;
  if (box < 0 || box >= b->nbox) return bfail(b, MHD_ERR_INVALID, "box index %d out of range", box);
  int rc = batch_ensure_prims(b);
  if (rc) return rc;
  unsigned long long* hp = (unsigned long long*)b->pinned + 32;
  const BoxDesc& d = b->box[box];
  BCUDA_TRY(b, cudaMemcpyAsync(hp, d.words + d.parity, sizeof(unsigned long long), cudaMemcpyDeviceToHost, b->stream));
  BCUDA_TRY(b, cudaStreamSynchronize(b->stream));
  double m;
  memcpy(&m, hp, sizeof m);
  *dt_out = m > 0.0 ? b->cfg[box].cfl / m : 0.0;
  return MHD_OK;
}

extern "C" int mhd_batch_get_stats(mhd_batch* b, mhd_stats* out) {
  if (!b || !out) return MHD_ERR_INVALID;
  unsigned long long* hp = (unsigned long long*)b->pinned;
  BCUDA_TRY(b, cudaMemcpyAsync(hp, b->words, 16 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, b->stream));
  BCUDA_TRY(b, cudaStreamSynchronize(b->stream));
  memset(out, 0, sizeof *out);
  out->status = (int)*(unsigned*)(hp + 3);
  out->rho_floor_hits = (long long)hp[8 + C_RHO_FLOOR];
  out->p_floor_hits = (long long)hp[8 + C_P_FLOOR];
  out->faces_hll = (long long)hp[8 + C_HLL];
  out->faces_hlld = (long long)hp[8 + C_HLLD];
  out->steps = b->steps;
  return MHD_OK;
}

// ---------------------------------------------------------------- autotuner
// Times the tile the batch has and every instantiated tile shape (at its
// default z-chunk length and a few fixed ones) on the batch itself for
// `trial_steps` steps, keeps the fastest, and records it in a JSON-lines cache
// keyed by device, precision, Riemann solver, the box sizes and the set of
// lengths tried, so later runs on the same batch skip the trials.

static std::string batch_key(mhd_batch* b) {
  int dev = 0, maj = 0, min = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&maj, cudaDevAttrComputeCapabilityMajor, dev);
  cudaDeviceGetAttribute(&min, cudaDevAttrComputeCapabilityMinor, dev);
  unsigned long long h = 1469598103934665603ull;
  long long cells = 0;
  for (int i = 0; i < b->nbox; ++i) {
    const int n[3] = {b->cfg[i].nx, b->cfg[i].ny, b->cfg[i].nz};
    for (int d = 0; d < 3; ++d) h = (h ^ (unsigned long long)(n[d] * 2 + b->cfg[i].bc[d])) * 1099511628211ull;
    cells += (long long)n[0] * n[1] * n[2];
  }
  char buf[256];
  snprintf(buf, sizeof buf, "sm_%d%d|prec%d|riemann%d|nbox%d|cells%lld|dims%016llx|z2", maj, min, b->prec,
           b->cfg[0].riemann, b->nbox, cells, h);
  return buf;
}

static bool cache_lookup(const char* path, const std::string& key, int tile[3], double* ms) {
  if (!path) return false;
  FILE* f = fopen(path, "r");
  if (!f) return false;
  char line[1024];
  bool found = false;
  while (fgets(line, sizeof line, f)) {
    char k[512];
    int tx, ty, tz;
    double m;
    if (sscanf(line, "{\"key\": \"%511[^\"]\", \"tile\": [%d, %d, %d], \"ms_per_step\": %lf", k, &tx, &ty, &tz, &m) == 5 &&
        key == k) {
      tile[0] = tx; tile[1] = ty; tile[2] = tz;
      *ms = m;
      found = true;  // the last matching line wins
    }
  }
  fclose(f);
  return found;
}

extern "C" int mhd_batch_autotune(mhd_batch* b, int trial_steps, const char* cache_path, int tile_out[3],
                                  double* ms_out) {
  if (!b) return MHD_ERR_INVALID;
  if (trial_steps < 1) return bfail(b, MHD_ERR_INVALID, "trial_steps must be >= 1");
  const std::string key = batch_key(b);
  int best[3] = {b->tx, b->ty, b->tz};
  double best_ms = -1.0;
  if (cache_lookup(cache_path, key, best, &best_ms)) {
    int rc = batch_apply_tile(b, best[0], best[1], best[2]);
    if (rc == MHD_OK) {
      if (tile_out) { tile_out[0] = best[0]; tile_out[1] = best[1]; tile_out[2] = best[2]; }
      if (ms_out) *ms_out = best_ms;
      return MHD_OK;
    }
  }
  // keep the states: trials advance them
  int rc = batch_ensure_prims(b);
  if (rc) return rc;
  std::vector<void*> save(b->nbox, nullptr);
  for (int i = 0; i < b->nbox; ++i) {
    cudaError_t e = cudaMalloc(&save[i], b->ubytes[i]);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(save[i], b->box[i].U[b->box[i].cur], b->ubytes[i], cudaMemcpyDeviceToDevice, b->stream);
    if (e != cudaSuccess) {
      for (void* p : save) cudaFree(p);
      return bfail(b, MHD_ERR_NOMEM, "autotune state copy failed: %s", cudaGetErrorString(e));
    }
  }
  static const int cand_xy[][2] = {{16, 8}, {16, 16}, {32, 8}, {24, 8}, {8, 8}};
  static const int cand_z[] = {16, 32, 64, 128};
  int maxnz = 1;
  for (int i = 0; i < b->nbox; ++i) maxnz = b->cfg[i].nz > maxnz ? b->cfg[i].nz : maxnz;
  // the batch's own tile first; a shape's default length only where it is none of the fixed ones
  std::vector<std::array<int, 3>> cand = {{b->tx, b->ty, b->tz}};
  const auto propose = [&](int tx, int ty, int tz) {
    const std::array<int, 3> t = {tx, ty, tz};
    if (std::find(cand.begin(), cand.end(), t) == cand.end()) cand.push_back(t);
  };
  for (const auto& xy : cand_xy) {
    for (int zi = 0; zi < 4 && (zi == 0 || cand_z[zi - 1] < maxnz); ++zi) propose(xy[0], xy[1], cand_z[zi]);
    propose(xy[0], xy[1], batch_default_chunk(b, xy[0], xy[1]));
  }
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  best_ms = -1.0;
  for (const auto& t : cand) {
    if (batch_apply_tile(b, t[0], t[1], t[2]) != MHD_OK) continue;   // tile not instantiated
    if (batch_enqueue(b, -1.0, 1) != MHD_OK) continue;
    cudaEventRecord(e0, b->stream);
    if (batch_enqueue(b, -1.0, trial_steps) != MHD_OK) continue;
    cudaEventRecord(e1, b->stream);
    if (batch_check(b) != MHD_OK) continue;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    const double per = ms / trial_steps;
    if (best_ms < 0.0 || per < best_ms) {
      best_ms = per;
      best[0] = t[0]; best[1] = t[1]; best[2] = t[2];
    }
    // restore the states for the next candidate
    for (int i = 0; i < b->nbox; ++i) {
      cudaMemcpyAsync(b->box[i].U[b->box[i].cur], save[i], b->ubytes[i], cudaMemcpyDeviceToDevice, b->stream);
      b->prims_valid[i] = false;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  for (int i = 0; i < b->nbox; ++i) {
    cudaMemcpyAsync(b->box[i].U[b->box[i].cur], save[i], b->ubytes[i], cudaMemcpyDeviceToDevice, b->stream);
    b->prims_valid[i] = false;
  }
  cudaStreamSynchronize(b->stream);
  for (void* p : save) cudaFree(p);
  if (best_ms < 0.0) return bfail(b, MHD_ERR_CUDA, "no tile candidate ran");
  rc = batch_apply_tile(b, best[0], best[1], best[2]);
  if (rc) return rc;
  if (cache_path) {
    FILE* f = fopen(cache_path, "a");
    if (f) {
      fprintf(f, "{\"key\": \"%s\", \"tile\": [%d, %d, %d], \"ms_per_step\": %.6f}\n", key.c_str(), best[0], best[1],
              best[2], best_ms);
      fclose(f);
    }
  }
  if (tile_out) { tile_out[0] = best[0]; tile_out[1] = best[1]; tile_out[2] = best[2]; }
  if (ms_out) *ms_out = best_ms;
  return MHD_OK;
}

// Helpers shared with the allocation-free entry point (noalloc.cu).
namespace mhd {
int internal_validate(const mhd_config* c) { return validate(c, nullptr); }
void internal_fill_geo(const mhd_config* c, Geo* g) { fill_geo(c, g); }
void internal_set_error(const char* msg) { g_create_err = msg; }
}  // namespace mhd

// ---------------------------------------------------------------- learned switch
namespace mhd {
int dump_faces_launch(int prec, const Geo& g, const void* W, const long long* ids, long long n, float* X, float* y,
                      float* score, cudaStream_t st);
}
extern "C" size_t mlp_param_bytes(void);

extern "C" int mhd_dump_faces(mhd_handle* h, const long long* face_ids, long long n, float* features, float* labels,
                              float* scores) {
  if (!h) return MHD_ERR_INVALID;
  if (!face_ids || !features || !labels || n < 0) return fail(h, MHD_ERR_INVALID, "bad arguments");
  for (int d = 0; d < 3; ++d)
    if (h->geo.bc[d] != 0) return fail(h, MHD_ERR_INVALID, "mhd_dump_faces samples periodic boxes only");
  cudaError_t e = ensure_prims(h);
  if (e) return fail(h, MHD_ERR_CUDA, "primitive recovery failed: %s", cudaGetErrorString(e));
  if (n == 0) return MHD_OK;
  int rc = dump_faces_launch(h->cfg.precision, h->geo, h->W[h->cur], face_ids, n, features, labels, scores,
                             h->stream);
  if (rc) return fail(h, rc, "face sampler launch failed");
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  return MHD_OK;
}

extern "C" int mhd_set_switch(mhd_handle* h, const void* block, double tau) {
  if (!h) return MHD_ERR_INVALID;
  if (!block) return fail(h, MHD_ERR_INVALID, "null parameter block");
  if (!(tau > 0.0 && tau < 1.0)) return fail(h, MHD_ERR_INVALID, "tau must lie in (0, 1)");
  if (!h->mlp) CUDA_TRY(h, cudaMalloc(&h->mlp, mlp_param_bytes()));
  CUDA_TRY(h, cudaMemcpyAsync(h->mlp, block, mlp_param_bytes(), cudaMemcpyDeviceToDevice, h->stream));
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  h->mlp_zt = (float)log(tau / (1.0 - tau));
  return MHD_OK;
}

extern "C" int mhd_switch_choices(mhd_handle* h, unsigned char* choices, float* logits) {
  if (!h) return MHD_ERR_INVALID;
  if (h->cfg.riemann != MHD_LEARNED) return fail(h, MHD_ERR_INVALID, "the handle's riemann is not MHD_LEARNED");
  if (!choices) return fail(h, MHD_ERR_INVALID, "null choices pointer");
  if (int rc = need_switch(h)) return rc;
  cudaError_t e = ensure_prims(h);
  if (e) return fail(h, MHD_ERR_CUDA, "primitive recovery failed: %s", cudaGetErrorString(e));
  const Geo& g = h->geo;
  StageArgs a = base_args(h);
  a.dt = 1.0;
  a.dtword = h->words + h->parity;
  a.nextword = h->words + 4;
  a.U = h->U[h->cur];
  a.Win = h->W[h->cur];
  a.K1out = h->K1;                          // scratch: the operator's value is discarded
  a.Wout = nullptr;
  a.choices = choices;
  a.logits = logits;
  e = launch_stage(h->cfg.precision, 1, g.TX, g.TY, (unsigned)(g.ntx * g.nty * g.nchunk), h->smem_bytes,
                   h->stream, g, a);
  if (e) return fail(h, MHD_ERR_CUDA, "stage launch failed: %s", cudaGetErrorString(e));
  return check_status(h);
}

// batch.cu -- batches of independent D2Q9 lattices (the C ABI's
// mlswlbm_batch_*): one arena of states, per-instance device descriptors,
// one unit table in which the instances that share layer count, kernel mode
// and nominal tile height (a group) have a contiguous range, one launch per step
// over the whole table (batch_kernels.cu), and a timing autotuner for the
// nominal height of every layer count and mode.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <new>
#include <tuple>
#include <vector>

#include "../../include/mlswlbm.h"
#include "host.h"
#include "kernels.h"
#include "physics.cuh"
#include "unit_rows.h"

using mlsw::BatchInst;
using mlsw::KParams;

namespace {

constexpr int kQ = 9;

struct Group {
  int n, mode, variant;
  int offset, nunits;  // slice of the unit table
};

}  // namespace

struct mlsw_batch {
  int count;
  std::vector<BatchInst> hinst;  // host copies of the descriptors
  std::vector<int> variant;      // nominal-height variant of every instance
  std::vector<char> solo;        // its maps and strips are those of one column a lane
  // instances the step advances (mlswlbm_batch_select; all at create) and,
  // for one left out, the buffer index that holds its state
  std::vector<char> selected;
  std::vector<int> home;
  std::vector<Group> groups;
  BatchInst* dinst;
  int2* dtable;  // the unit table, sorted by kind
  int nunits;          // its length
  unsigned kinds;      // kinds in it
  int same_params;     // its instances' parameters differ in H and Hsum only
  KParams params;         // of the first instance in it
  std::vector<int> tiny;  // selected instances whose ghosts need a pass of their own
  float* arena;
  int* dstatus;  // error bits
  float* hbuf;   // heights of the largest instance (upload, read-out)
  int* dk;       // 2 count mode numbers
  double* dmode; // 2 kMaxLayers count doubles
  int cur;
  cudaStream_t stream;   // the caller's stream
  long launches;
  int num_sms;
};

namespace {

#define CUB(call)                                    \
  do {                                               \
    if ((call) != cudaSuccess) return MLSW_ERR_CUDA; \
  } while (0)

// planes per layer of an instance's buffers
int planes_of(const KParams& P) { return mlsw::step_moments(P) ? mlsw::kMomPlanes : kQ; }

int units_of(const BatchInst& b, int rows) { return b.strips * ((b.P.ny + rows - 1) / rows); }

// Rows of an instance's units at scale r: four and five layers half of r, the
// others r, or half of it too where the variant is 8 (half).
int scaled_rows(const BatchInst& b, int r, bool half) {
  const int rows = b.P.n <= 3 ? r : (r + 1) / 2;
  return std::min(64, b.P.n <= 3 && half ? mlsw::half_rows(rows) : rows);
}

double weight_of(const BatchInst& b) {
  return mlsw::batch_weight(b.P.n, b.kind % 3, b.P.sub_amp != 0.f);
}

unsigned kinds_of(const mlsw_batch* b, const std::vector<int>& members) {
  unsigned kinds = 0;
  for (int j : members) kinds |= 1u << b->hinst[j].kind;
  return kinds;
}

bool one_kind(unsigned kinds) { return (kinds & (kinds - 1)) == 0; }

// Tables whose units have one height, scaled: those of one kind, of the kernel
// for at most three layers, or without an instance whose cells have many terms
// (whose rows take up to four times the others').
bool scaled_table(const mlsw_batch* b, const std::vector<int>& members, unsigned kinds) {
  if (one_kind(kinds) || mlsw::batch_small(kinds)) return true;
  for (int j : members)
    if (mlsw::step_dear(b->hinst[j].P)) return false;
  return true;
}

// Scale r of the units of such a table, by a model of a step's time in units of
// a row's issue time on one of an SM's four schedulers. A unit costs its rows
// plus about five rows of warm-up; a warp alone on a scheduler needs 1.75 times
// that time for a row's latencies.
// Instances of one layer count finish together, in whole waves, and as the
// schedulers' fullest; uneven ones (work in proportion to n) overlap, and the
// longest unit may come last. Beside four or five layers the variants shift the
// proportion of the heights, and the scale follows; without them the scale is that
// of the nominal 16, so that 8 are half of it (a scale for them would give the same
// heights again). 16 films of 256^2: r = 12 instead of 16 brings a step from 47 to
// 44 us.
int scale_for(const mlsw_batch* b, const std::vector<int>& members, unsigned kinds) {
  int nmax = 0, nmin = mlsw::kMaxLayers;
  for (int j : members) {
    nmax = std::max(nmax, b->hinst[j].P.n);
    nmin = std::min(nmin, b->hinst[j].P.n);
  }
  const int per_sm = mlsw::batch_warps_per_sm(kinds);
  const double schedulers = 4.0 * b->num_sms, slots = (double)per_sm * b->num_sms;
  int best_r = 1;
  double best = 0.0;
  for (int r = 1; r <= 128; ++r) {
    double units = 0.0, work = 0.0, longest = 0.0;
    for (int j : members) {
      const int rows = scaled_rows(b->hinst[j], r, nmax > 3 && b->variant[j] == 1);
      const double u = units_of(b->hinst[j], rows), w = (double)(rows + 5) * b->hinst[j].P.n;
      units += u;
      work += u * w;
      longest = std::max(longest, w);
    }
    double cost;
    if (nmin == nmax) {
      const double full = per_sm / 4.0;
      const double q = units <= slots ? std::min(std::ceil(units / schedulers), full)
                                      : std::ceil(units / slots) * full;
      cost = longest * std::max(1.75, q);
    } else {
      cost = work / schedulers + 1.75 * longest;
    }
    if (r == 1 || cost < best) {
      best = cost;
      best_r = r;
    }
  }
  return best_r;
}

// Duration t (us) of the units of other tables: the same for all kinds, so that
// none is left running alone (32 lattices of 2 to 5 layers, all modes: 294 us a
// step with one scaled height, 226). *one_wave: they fit the chip at once.
double unit_time(const mlsw_batch* b, const std::vector<int>& members, unsigned kinds,
                 bool* one_wave) {
  const int slots = b->num_sms * mlsw::batch_warps_per_sm(kinds);
  double best_t = 0.0, best = 0.0;
  for (int c = 0; c < 128; ++c) {
    const double t = 3.0 * std::pow(1.035, c);
    double units = 0.0, work = 0.0, longest = 0.0;
    for (int j : members) {
      const double w = weight_of(b->hinst[j]);
      const int rows = mlsw::batch_rows(w, t);
      const double u = units_of(b->hinst[j], rows);
      units += u;
      work += u * (rows + 5) * w;
      longest = std::max(longest, (rows + 5) * w);
    }
    const double cost = mlsw::batch_cost(units, work, longest, b->num_sms, slots);
    if (c == 0 || cost < best) {
      best = cost;
      best_t = t;
      *one_wave = units <= slots;
    }
  }
  return best_t;
}

bool any_general(unsigned kinds) {
  for (int k = mlsw::kGeneral; k < mlsw::kBatchKinds; k += 3)
    if ((kinds >> k) & 1u) return true;
  return false;
}

// Rows of the members' units: all of the model's for the nominal 16, half for 8.
// Returns whether the table is one wave of units of equal duration. Tables at
// tau = 1 in several waves keep one height (71 lattices of the fast mode and on a
// substrate: 274 us a step, 299 with equal durations).
bool choose_rows(mlsw_batch* b, const std::vector<int>& members, unsigned kinds) {
  bool scaled = scaled_table(b, members, kinds), one_wave = false;
  const double t = scaled ? 0.0 : unit_time(b, members, kinds, &one_wave);
  scaled = scaled || (!one_wave && !any_general(kinds));
  const int r = scaled ? scale_for(b, members, kinds) : 1;
  for (int j : members) {
    BatchInst& bi = b->hinst[j];
    const bool half = b->variant[j] == 1;
    if (scaled) {
      bi.rows = scaled_rows(bi, r, half);
    } else {
      const int rows = mlsw::batch_rows(weight_of(bi), t);
      bi.rows = bi.P.n <= 3 && half ? mlsw::half_rows(rows) : rows;
    }
  }
  return !scaled && one_wave;
}

// The order of a table of units of equal duration that is sorted by kind and
// runs as one wave: neighbouring CTAs start on different SMs, so neighbouring
// entries go num_sms apart, and the warps of an SM share few kinds' instructions
// (9 lattices of 2 to 5 layers, all modes: 56 us a step in the sorted order, 28; in
// several waves the sorted order does it, and spreads the work better).
void order_one_wave(std::vector<int2>& table, int num_sms) {
  std::vector<int2> out(table.size());
  size_t u = 0;
  for (int s = 0; s < num_sms; ++s)
    for (size_t p = s; p < table.size(); p += num_sms) out[p] = table[u++];
  table.swap(out);
}

// the buffer that holds instance j's state now
int state_buffer(const mlsw_batch* b, int j) { return b->selected[j] ? b->cur : b->home[j]; }

// Moves every left-out instance whose state sits in the other buffer to the
// current one by swapping its two buffers (and their tensor maps) in its
// descriptor, so that every instance's state is in buffer cur.
int align_buffers(mlsw_batch* b) {
  bool changed = false;
  for (int j = 0; j < b->count; ++j) {
    if (b->selected[j] || b->home[j] == b->cur) continue;
    BatchInst& bi = b->hinst[j];
    std::swap(bi.f[0], bi.f[1]);
    std::swap(bi.map[0], bi.map[1]);
    b->home[j] = b->cur;
    changed = true;
  }
  // pageable source: the copy is staged before the call returns
  if (changed)
    CUB(cudaMemcpyAsync(b->dinst, b->hinst.data(), (size_t)b->count * sizeof(BatchInst),
                        cudaMemcpyHostToDevice, b->stream));
  return MLSW_OK;
}

// the row maps of instance j's two buffers, in the form it marches in
bool map_rows(mlsw_batch* b, int j) {
  BatchInst& bi = b->hinst[j];
  bool ok = true;
  for (int k = 0; k < 2; ++k)
    ok = ok && mlsw_host::make_row_map(&bi.map[k], bi.f[k], bi.P.L, bi.P.n * planes_of(bi.P),
                                       b->solo[j]);
  return ok;
}

// (re)initialise every instance from its heights: f = f_eq(h, U = 0)
int init_all(mlsw_batch* b, const float* const* h_init) {
  for (int j = 0; j < b->count; ++j) {
    const KParams& P = b->hinst[j].P;
    const size_t bytes = (size_t)P.n * P.nx * P.ny * sizeof(float);
    mlsw::KShift sh;
    for (int i = 0; i < mlsw::kMaxLayers; ++i) sh.H[i] = P.H[i];
    CUB(cudaMemcpyAsync(b->hbuf, h_init[j], bytes, cudaMemcpyHostToDevice, b->stream));
    CUB(mlsw::launch_init(planes_of(P), P.n, P.L, b->hbuf, b->hinst[j].f[0], sh, b->dstatus,
                          b->stream));
    b->launches += 1;
    b->home[j] = 0;
  }
  b->cur = 0;
  return MLSW_OK;
}

// whether the parameters of the members differ in H and Hsum only
int same_params(const mlsw_batch* b, const std::vector<int>& members) {
  for (int j : members) {
    KParams q = b->hinst[j].P;
    const KParams& p = b->hinst[members[0]].P;
    std::memcpy(q.H, p.H, sizeof(q.H));
    std::memcpy(q.Hsum, p.Hsum, sizeof(q.Hsum));
    if (std::memcmp(&q, &p, sizeof(q)) != 0) return 0;
  }
  return 1;
}

// the unit table of the groups for the current variant choice, sorted by
// kind (layer count descending: the dearest units first, so that the last
// ones to run are short), and the unit rows in the descriptors
int build_groups(mlsw_batch* b) {
  std::map<std::tuple<int, int, int>, std::vector<int>> members;
  std::vector<int> all;
  b->kinds = 0;
  b->tiny.clear();
  for (int j = 0; j < b->count; ++j) {
    if (!b->selected[j]) continue;
    const BatchInst& bi = b->hinst[j];
    members[std::make_tuple(-bi.P.n, mlsw::step_mode(bi.P), b->variant[j])].push_back(j);
    all.push_back(j);
    b->kinds |= 1u << bi.kind;
    if (bi.P.tiny) b->tiny.push_back(j);
  }
  // the strips of the kernel that these instances will run, and its row maps
  for (int j : all) {
    BatchInst& bi = b->hinst[j];
    const bool solo = mlsw::batch_solo(b->kinds, bi.kind);
    if (solo == b->solo[j]) continue;
    b->solo[j] = solo;
    bi.strips = mlsw::march_strips(bi.P.nx, solo);
    if (!map_rows(b, j)) return MLSW_ERR_CUDA;
  }
  const bool one_wave = !all.empty() && choose_rows(b, all, b->kinds);
  b->same_params = same_params(b, all);
  if (!all.empty()) b->params = b->hinst[all[0]].P;
  std::vector<int2> table;
  b->groups.clear();
  for (auto& kv : members) {
    Group g;
    g.n = -std::get<0>(kv.first);
    g.mode = std::get<1>(kv.first);
    g.variant = std::get<2>(kv.first);
    g.offset = (int)table.size();
    for (int j : kv.second) {
      const int nu = units_of(b->hinst[j], b->hinst[j].rows);
      for (int t = 0; t < nu; ++t) table.push_back(make_int2(j, t));
    }
    g.nunits = (int)table.size() - g.offset;
    b->groups.push_back(g);
  }
  b->nunits = (int)table.size();
  if (one_wave && b->nunits <= b->num_sms * mlsw::batch_warps_per_sm(b->kinds))
    order_one_wave(table, b->num_sms);
  if (b->dtable) cudaFree(b->dtable);
  b->dtable = nullptr;
  if (cudaMalloc(&b->dtable, std::max<size_t>(1, table.size()) * sizeof(int2)) != cudaSuccess)
    return MLSW_ERR_NOMEM;
  // on the stream of the steps that read them (pageable sources: staged before
  // the calls return)
  CUB(cudaMemcpyAsync(b->dtable, table.data(), table.size() * sizeof(int2), cudaMemcpyHostToDevice,
                      b->stream));
  CUB(cudaMemcpyAsync(b->dinst, b->hinst.data(), (size_t)b->count * sizeof(BatchInst),
                      cudaMemcpyHostToDevice, b->stream));
  return MLSW_OK;
}

// the launch of a step over the groups' table, from buffer cur
mlsw::BatchLaunch step_launch(const mlsw_batch* b) {
  mlsw::BatchLaunch a;
  a.inst = b->dinst;
  a.table = b->dtable;
  a.nunits = b->nunits;
  a.kinds = b->kinds;
  a.same_params = b->same_params;
  a.P = b->params;
  a.cur = b->cur;
  a.status = b->dstatus;
  return a;
}

// us of a step over the present table, from kTimed steps after a few
int time_steps(mlsw_batch* b, cudaEvent_t e0, cudaEvent_t e1, float* ms) {
  constexpr int kWarm = 2, kTimed = 8;
  for (int s = 0; s < kWarm + kTimed; ++s) {
    if (s == kWarm) CUB(cudaEventRecord(e0, b->stream));
    mlsw::BatchLaunch a = step_launch(b);
    a.cur = s & 1;
    CUB(mlsw::launch_batch_step(a, b->stream));
    b->launches += 1;
  }
  CUB(cudaEventRecord(e1, b->stream));
  CUB(cudaEventSynchronize(e1));
  CUB(cudaEventElapsedTime(ms, e0, e1));
  return MLSW_OK;
}

// Timing autotuner: for every layer count (<= 3) and mode of the batch in turn,
// the whole batch is stepped with that class's units at the nominal 16 and 8
// rows, in the kernel it will run; 8 is kept where it is 0.5 % faster (the spread
// of the timings; the sweep of 512 lattices: 1097 us a step with 16, 1085 with 8). The steps change the states, which the caller
// resets afterwards, and leave the table to be built.
int autotune(mlsw_batch* b) {
  std::map<int, std::vector<int>> classes;
  for (int j = 0; j < b->count; ++j)
    if (b->hinst[j].P.n <= 3) classes[b->hinst[j].kind].push_back(j);
  cudaEvent_t e0, e1;
  CUB(cudaEventCreate(&e0));
  if (cudaEventCreate(&e1) != cudaSuccess) {
    cudaEventDestroy(e0);
    return MLSW_ERR_CUDA;
  }
  float best = 0.f;
  int rc = build_groups(b);
  if (rc == MLSW_OK) rc = time_steps(b, e0, e1, &best);
  for (auto& kv : classes) {
    if (rc != MLSW_OK) break;
    for (int j : kv.second) b->variant[j] = 1;
    float ms = 0.f;
    rc = build_groups(b);
    if (rc == MLSW_OK) rc = time_steps(b, e0, e1, &ms);
    if (rc == MLSW_OK && ms < 0.995f * best)
      best = ms;
    else
      for (int j : kv.second) b->variant[j] = 0;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return rc;
}

}  // namespace

extern "C" {

void mlswlbm_batch_destroy(mlsw_batch* b) {
  if (!b) return;
  cudaStreamSynchronize(b->stream);
  cudaFree(b->dinst);
  cudaFree(b->dtable);
  cudaFree(b->arena);
  cudaFree(b->dstatus);
  cudaFree(b->hbuf);
  cudaFree(b->dk);
  cudaFree(b->dmode);
  delete b;
}

int mlswlbm_batch_create(int count, const mlsw_params* params, const float* const* h_init,
                         int flags, void* stream, mlsw_batch** out) {
  if (!out) return MLSW_ERR_ARG;
  *out = nullptr;
  if (count < 1 || !params || !h_init) return MLSW_ERR_ARG;
  mlsw_batch* b = new (std::nothrow) mlsw_batch();
  if (!b) return MLSW_ERR_NOMEM;
  b->count = count;
  b->stream = (cudaStream_t)stream;
  int rc = MLSW_OK;
  size_t arena_floats = 0, max_heights = 0;
  std::vector<size_t> off(count);
  try {
    b->hinst.resize(count);
    b->variant.resize(count);
    b->solo.assign(count, 0);
    b->selected.assign(count, 1);
    b->home.assign(count, 0);
  } catch (...) {
    delete b;
    return MLSW_ERR_NOMEM;
  }
  for (int j = 0; j < count && rc == MLSW_OK; ++j) {
    if (params[j].lattice != MLSW_D2Q9) {
      rc = MLSW_ERR_UNSUPPORTED;
      break;
    }
    BatchInst& bi = b->hinst[j];
    std::memset(&bi, 0, sizeof(bi));
    mlsw::KShift sh;
    rc = mlsw_host::prepare_instance(params[j], h_init[j], bi.P, sh);
    if (rc != MLSW_OK) break;
    bi.kind = mlsw::batch_kind(bi.P.n, mlsw::step_mode(bi.P));
    bi.strips = mlsw::march_strips(bi.P.nx, false);
    const size_t flen = (size_t)bi.P.n * planes_of(bi.P) * bi.P.L.plane;
    off[j] = arena_floats;
    arena_floats += 2 * ((flen + 63) / 64 * 64);  // two buffers, 256-byte aligned
    max_heights = std::max(max_heights, (size_t)bi.P.n * bi.P.nx * bi.P.ny);
    b->variant[j] = (flags & MLSW_BATCH_TILE8) || bi.P.n > 3 ? 1 : 0;
  }
  if (rc != MLSW_OK) {
    delete b;
    return rc;
  }
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    delete b;
    return MLSW_ERR_CUDA;
  }
  b->num_sms = sms > 0 ? sms : 1;
  bool ok = cudaMalloc(&b->arena, arena_floats * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&b->dinst, (size_t)count * sizeof(BatchInst)) == cudaSuccess &&
            cudaMalloc(&b->dstatus, sizeof(int)) == cudaSuccess &&
            cudaMalloc(&b->hbuf, max_heights * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&b->dk, 2 * (size_t)count * sizeof(int)) == cudaSuccess &&
            cudaMalloc(&b->dmode, 2 * (size_t)mlsw::kMaxLayers * count * sizeof(double)) ==
                cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    mlswlbm_batch_destroy(b);
    return MLSW_ERR_NOMEM;
  }
  // zero padding (columns outside the real domains and their ghosts are
  // read by edge strips but feed no real cell) and the status word
  ok = cudaMemsetAsync(b->dstatus, 0, sizeof(int), b->stream) == cudaSuccess &&
       cudaMemsetAsync(b->arena, 0, arena_floats * sizeof(float), b->stream) == cudaSuccess;
  for (int j = 0; j < count && ok; ++j) {
    BatchInst& bi = b->hinst[j];
    const size_t flen = (size_t)bi.P.n * planes_of(bi.P) * bi.P.L.plane;
    bi.f[0] = b->arena + off[j];
    bi.f[1] = b->arena + off[j] + (flen + 63) / 64 * 64;
    ok = map_rows(b, j);
  }
  ok = ok && cudaMemcpy(b->dinst, b->hinst.data(), (size_t)count * sizeof(BatchInst),
                        cudaMemcpyHostToDevice) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    mlswlbm_batch_destroy(b);
    return MLSW_ERR_CUDA;
  }
  rc = init_all(b, h_init);
  if (rc == MLSW_OK && (flags & MLSW_BATCH_AUTOTUNE) && !(flags & MLSW_BATCH_TILE8)) {
    rc = autotune(b);
    if (rc == MLSW_OK) rc = init_all(b, h_init);
  }
  if (rc == MLSW_OK) rc = build_groups(b);
  if (rc == MLSW_OK && cudaStreamSynchronize(b->stream) != cudaSuccess) rc = MLSW_ERR_CUDA;
  if (rc == MLSW_OK) {
    // a non-finite or non-positive height in h_init was flagged by init
    int flag = 0;
    if (cudaMemcpy(&flag, b->dstatus, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
      rc = MLSW_ERR_CUDA;
    else if (flag)
      rc = MLSW_ERR_ARG;
  }
  if (rc != MLSW_OK) {
    mlswlbm_batch_destroy(b);
    return rc;
  }
  *out = b;
  return MLSW_OK;
}

int mlswlbm_batch_step(mlsw_batch* b, long nsteps) {
  if (!b || nsteps < 0) return MLSW_ERR_ARG;
  if (b->groups.empty()) return MLSW_OK;  // no instance selected
  for (long s = 0; s < nsteps; ++s) {
    CUB(mlsw::launch_batch_step(step_launch(b), b->stream));
    b->launches += 1;
    b->cur ^= 1;
    for (int j : b->tiny) {
      const BatchInst& bi = b->hinst[j];
      CUB(mlsw::launch_fill_ghosts(bi.P.n * kQ, bi.P.L, bi.f[b->cur], b->stream));
      b->launches += 1;
    }
  }
  return MLSW_OK;
}

int mlswlbm_batch_status(mlsw_batch* b) {
  if (!b) return MLSW_ERR_ARG;
  int flag = 0;
  CUB(cudaMemcpyAsync(&flag, b->dstatus, sizeof(int), cudaMemcpyDeviceToHost, b->stream));
  CUB(cudaStreamSynchronize(b->stream));
  if (flag) {
    CUB(cudaMemsetAsync(b->dstatus, 0, sizeof(int), b->stream));
    return (flag & mlsw::kStatusTimeout) ? MLSW_ERR_TIMEOUT : MLSW_ERR_NONFINITE;
  }
  return MLSW_OK;
}

int mlswlbm_batch_get_heights(mlsw_batch* b, int index, float* out) {
  if (!b || !out || index < 0 || index >= b->count) return MLSW_ERR_ARG;
  const KParams& P = b->hinst[index].P;
  CUB(mlsw::launch_batch_heights(&b->hinst[index], state_buffer(b, index), b->hbuf, b->stream));
  b->launches += 1;
  CUB(cudaMemcpyAsync(out, b->hbuf, (size_t)P.n * P.nx * P.ny * sizeof(float),
                      cudaMemcpyDeviceToHost, b->stream));
  return mlswlbm_batch_status(b);
}

int mlswlbm_batch_get_heights_device(mlsw_batch* b, int index, float* dev_out) {
  if (!b || !dev_out || index < 0 || index >= b->count) return MLSW_ERR_ARG;
  CUB(mlsw::launch_batch_heights(&b->hinst[index], state_buffer(b, index), dev_out, b->stream));
  b->launches += 1;
  return MLSW_OK;
}

int mlswlbm_batch_set_heights_device(mlsw_batch* b, int index, const float* dev_in) {
  if (!b || !dev_in || index < 0 || index >= b->count) return MLSW_ERR_ARG;
  const KParams& P = b->hinst[index].P;
  mlsw::KShift sh;
  for (int i = 0; i < mlsw::kMaxLayers; ++i) sh.H[i] = P.H[i];
  CUB(mlsw::launch_init(planes_of(P), P.n, P.L, dev_in, b->hinst[index].f[state_buffer(b, index)],
                        sh, b->dstatus, b->stream));
  b->launches += 1;
  return MLSW_OK;
}

int mlswlbm_batch_get_heights_device_many(mlsw_batch* b, int count, const int* indices,
                                          float* dev_out) {
  if (!b || count < 0 || (count > 0 && (!indices || !dev_out))) return MLSW_ERR_ARG;
  for (int k = 0; k < count; ++k)
    if (indices[k] < 0 || indices[k] >= b->count) return MLSW_ERR_ARG;
  size_t off = 0;
  for (int k = 0; k < count; ++k) {
    const int j = indices[k];
    const KParams& P = b->hinst[j].P;
    CUB(mlsw::launch_batch_heights(&b->hinst[j], state_buffer(b, j), dev_out + off, b->stream));
    b->launches += 1;
    off += (size_t)P.n * P.nx * P.ny;
  }
  return MLSW_OK;
}

int mlswlbm_batch_set_heights_device_many(mlsw_batch* b, int count, const int* indices,
                                          const float* dev_in) {
  if (!b || count < 0 || (count > 0 && (!indices || !dev_in))) return MLSW_ERR_ARG;
  for (int k = 0; k < count; ++k)
    if (indices[k] < 0 || indices[k] >= b->count) return MLSW_ERR_ARG;
  size_t off = 0;
  for (int k = 0; k < count; ++k) {
    const int j = indices[k];
    const KParams& P = b->hinst[j].P;
    mlsw::KShift sh;
    for (int i = 0; i < mlsw::kMaxLayers; ++i) sh.H[i] = P.H[i];
    CUB(mlsw::launch_init(planes_of(P), P.n, P.L, dev_in + off, b->hinst[j].f[state_buffer(b, j)],
                          sh, b->dstatus, b->stream));
    b->launches += 1;
    off += (size_t)P.n * P.nx * P.ny;
  }
  return MLSW_OK;
}

int mlswlbm_batch_modes(mlsw_batch* b, const int* kx, const int* ky, double* out) {
  if (!b || !kx || !ky || !out) return MLSW_ERR_ARG;
  const int rc = align_buffers(b);
  if (rc != MLSW_OK) return rc;
  const size_t nk = (size_t)b->count * sizeof(int);
  CUB(cudaMemcpyAsync(b->dk, kx, nk, cudaMemcpyHostToDevice, b->stream));
  CUB(cudaMemcpyAsync(b->dk + b->count, ky, nk, cudaMemcpyHostToDevice, b->stream));
  CUB(mlsw::launch_batch_modes(b->dinst, b->count, b->cur, b->dk, b->dk + b->count, b->dmode,
                               b->stream));
  b->launches += 1;
  CUB(cudaMemcpyAsync(out, b->dmode, 2 * (size_t)mlsw::kMaxLayers * b->count * sizeof(double),
                      cudaMemcpyDeviceToHost, b->stream));
  return mlswlbm_batch_status(b);
}

int mlswlbm_batch_select(mlsw_batch* b, int nsel, const int* indices) {
  if (!b || nsel < 0 || nsel > b->count || (nsel > 0 && !indices)) return MLSW_ERR_ARG;
  std::vector<char> want(b->count, 0);
  for (int k = 0; k < nsel; ++k) {
    const int j = indices[k];
    if (j < 0 || j >= b->count || want[j]) return MLSW_ERR_ARG;
    want[j] = 1;
  }
  // every state into buffer cur first: then leaving out or taking back an
  // instance moves no data
  int rc = align_buffers(b);
  if (rc != MLSW_OK) return rc;
  for (int j = 0; j < b->count; ++j) {
    b->selected[j] = want[j];
    b->home[j] = b->cur;
  }
  // steps in flight read the unit table being replaced
  CUB(cudaStreamSynchronize(b->stream));
  return build_groups(b);
}

int mlswlbm_batch_tile_rows(const mlsw_batch* b, int index) {
  if (!b || index < 0 || index >= b->count) return MLSW_ERR_ARG;
  return mlsw::batch_tile_rows(b->variant[index]);
}

long mlswlbm_batch_launch_count(const mlsw_batch* b) { return b ? b->launches : -1; }

int mlswlbm_batch_groups(const mlsw_batch* b) { return b ? (int)b->groups.size() : -1; }

}  // extern "C"

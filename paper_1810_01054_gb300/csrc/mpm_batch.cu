// Batched execution of many scenes (include/mpm.h, mpm_batch_*).
//
// Scenes of one dimension advance together: every launch of a batched step covers all scenes of
// a sub-batch through one scene table (one record per scene, selected on the device from that
// scene's own tables and step counter, with the scene's tile and particle offsets in the batch).
// Scenes whose next work is a forward step (rollout or segment recompute) form the forward
// sub-batch; scenes in their reverse pass form the reverse sub-batch.  Both run every tick, the
// reverse one on the context's second stream beside the forward one (disjoint scenes, each with
// its own tile arrays and node blocks), joined before the tick's bookkeeping.  Tiles
// never span scenes and every sum inside a tile has a fixed order, so a scene's results are the
// same bits alone or in any mix.
//
// Per-scene life cycle of a request: rollout of n_steps (every state kept, or a checkpoint every
// ceil(sqrt(n_steps)) steps: request_interval); with want_grad, the reverse pass seeded by loss = mean of the final x_0, segment by
// segment (recompute, then reverse steps).  Results stay in the scene (mpm_get_state,
// mpm_get_gradients).
#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "mpm_scene.h"

using namespace gbmpm;

namespace {

enum SlotState { S_FREE = 0, S_FWD, S_RCM, S_REV, S_CLOSING, S_DONE };

struct Slot {
  mpm_scene* s = nullptr;
  int state = S_FREE;
  int T = 0, want_grad = 0, done_steps = 0, seg = 0, left = 0;
  int tiles = 0;  // most tiles its particles were seen in (a share of the composition's)
  size_t mem = 0;  // checkpoint bytes charged to the budget
  mpm_status status = MPM_OK;
};

struct SubBatch {
  std::vector<int> members;  // slot indices
  BatchDev b{};
  // what a composition uploads, in one device block: selections, controllers, particle offsets and
  // the tiles' scenes.  Written on the host into one of two pinned blocks in turn and copied on the
  // stream, so that a change of composition waits for nothing (16 requests of 0.5k-3k particles and
  // up to 41 steps, 11 with their gradient: 9.7 ms with a wait and eight copies at each of ~100
  // changes; 4.9 ms with this, every state kept and finished requests closed once a tick).
  char* meta = nullptr;
  char* staging[2] = {nullptr, nullptr};
  cudaEvent_t copied[2] = {nullptr, nullptr};
  int turn = 0;
  size_t off_ctrl = 0, off_pbase = 0, off_tiles = 0, meta_bytes = 0;
  SelectPar* dsel = nullptr;
  ScenePar* cur = nullptr;
  CtrlPar* dctrl = nullptr;
  int* pbase = nullptr;
  int cap_scenes = 0, cap_tiles = 0, cap_particles = 0;
  bool need_keys = true;  // composition changed: bin keys and histogram from the selected states
  // launch shapes: the cache entry of the composition's key, else trials during its steps
  TuneState tune;
  long long key_particles = -1, key_tiles = -1;
  unsigned key_kernels = 0;  // kernels of the key whose launch shapes are tuned
  int trial_wait = 0;  // steps of this key left before its trials start (0: none pending)
  BinSet bins;        // tile bins, for compositions of at most bin_tiles tiles (none: they sort)
  int bin_tiles = 0;
  // 3D compositions of few tiles: the active tiles of the last step of a tick, copied to `seen` (pinned)
  // without waiting and looked at by a later tick if the composition is still the same
  long long composed = 0, seen_composed = -1;  // compositions so far; the one `seen` is of (-1: none)
  int* seen = nullptr;
  cudaEvent_t seen_at = nullptr;
  uint32_t* sorted = nullptr;
  float4 *partial = nullptr, *partial_b = nullptr;  // node blocks (each half its own: they run at once)
  int cap_edge = 0;  // tile edge the node-block arrays are sized for
};

// Steps a composition key must run before its launch-shape trials start: a serving mix changes
// composition every few ticks, and trials that never finish would only cost time.
constexpr int kTrialWait = 32;

#define CK(expr)                                                                   \
  do {                                                                             \
    cudaError_t e_ = (expr);                                                       \
    if (e_ != cudaSuccess) return out_of_memory(e_) ? MPM_ERR_OOM : MPM_ERR_CUDA;       \
  } while (0)
#define CKS(expr)                \
  do {                           \
    mpm_status s_ = (expr);      \
    if (s_ != MPM_OK) return s_; \
  } while (0)

template <class T>
void dfree(T*& p) {
  if (p) cudaFree(p);
  p = nullptr;
}

void free_sub(mpm_ctx* ctx, SubBatch& sb) {
  batch_tune_release(sb.tune);
  sb.key_particles = sb.key_tiles = -1;
  dfree(sb.meta);
  for (int i = 0; i < 2; ++i) {
    if (sb.staging[i]) cudaFreeHost(sb.staging[i]);
    sb.staging[i] = nullptr;
    if (sb.copied[i]) cudaEventDestroy(sb.copied[i]);
    sb.copied[i] = nullptr;
  }
  if (sb.seen) cudaFreeHost(sb.seen);
  if (sb.seen_at) cudaEventDestroy(sb.seen_at);
  sb.seen = nullptr;
  sb.seen_at = nullptr;
  sb.seen_composed = -1;
  dfree(sb.cur);
  dfree(sb.b.tile_count);
  dfree(sb.b.tile_fill);
  dfree(sb.b.tile_start);
  dfree(sb.b.tile_slot);
  dfree(sb.b.active);
  dfree(sb.b.n_active);
  dfree(sb.b.block_sums);
  dfree(sb.b.work);
  dfree(sb.sorted);
  drop_bins(ctx, sb.bins);
  sb.bin_tiles = 0;
  dfree(sb.b.gpartial);
  dfree(sb.partial);
  dfree(sb.partial_b);
  sb.cap_scenes = sb.cap_tiles = sb.cap_particles = 0;
}

// Nodes of a tile's node block ((edge + 2)^dim).
int block_nodes(int dim, int edge) {
  const int bn = edge + 2;
  return dim == 2 ? bn * bn : bn * bn * bn;
}

}  // namespace

struct mpm_batch {
  mpm_ctx* ctx = nullptr;
  int dim = 0;
  int edge = 0;  // tile edge of the admitted scenes (set by the first admission into an empty batch)
  size_t budget = 0, used = 0;
  std::vector<Slot> slots;
  SubBatch fwd, rev;
  bool dirty = true;
  cudaEvent_t fork = nullptr, join = nullptr;  // the reverse half runs on the second stream
  // per-tick bookkeeping: counter writes of the scenes changing phase (one launch), the slots whose
  // request finished (one status gather), device array of the gathered status words
  std::vector<std::pair<int*, int>> pend_ctr;
  std::vector<int> finishing;
  int* d_status = nullptr;
  int status_cap = 0;
};

namespace {

mpm_status grow(mpm_batch* B, SubBatch& sb, int n_scenes, int tiles, int particles) {
  const int sc = std::max(1, n_scenes), tl = std::max(1, tiles), pc = std::max(64, particles);
  if (sc <= sb.cap_scenes && tl <= sb.cap_tiles && pc <= sb.cap_particles && sb.cap_edge == B->edge)
    return MPM_OK;
  CK(cudaStreamSynchronize(B->ctx->stream));
  free_sub(B->ctx, sb);
  auto round = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
  sb.off_ctrl = round(sizeof(SelectPar) * sc);
  sb.off_pbase = sb.off_ctrl + round(sizeof(CtrlPar) * sc);
  sb.off_tiles = sb.off_pbase + round(sizeof(int) * (size_t(sc) + 1));
  sb.meta_bytes = sb.off_tiles + round(sizeof(int) * size_t(tl));
  CK(cudaMalloc(&sb.meta, sb.meta_bytes));
  for (int i = 0; i < 2; ++i) {
    CK(cudaMallocHost(&sb.staging[i], sb.meta_bytes));
    CK(cudaEventCreateWithFlags(&sb.copied[i], cudaEventDisableTiming));
  }
  sb.dsel = reinterpret_cast<SelectPar*>(sb.meta);
  sb.dctrl = reinterpret_cast<CtrlPar*>(sb.meta + sb.off_ctrl);
  sb.pbase = reinterpret_cast<int*>(sb.meta + sb.off_pbase);
  sb.b.tile_scene = reinterpret_cast<int*>(sb.meta + sb.off_tiles);
  CK(cudaMalloc(&sb.cur, sizeof(ScenePar) * sc));
  CK(cudaMalloc(&sb.b.tile_count, sizeof(uint32_t) * tl));
  CK(cudaMalloc(&sb.b.tile_fill, sizeof(uint32_t) * tl));
  CK(cudaMalloc(&sb.b.tile_start, sizeof(uint32_t) * (tl + 1)));
  CK(cudaMalloc(&sb.b.tile_slot, sizeof(int) * tl));
  CK(cudaMalloc(&sb.b.active, sizeof(int) * tl));
  CK(cudaMalloc(&sb.b.n_active, sizeof(int)));
  CK(cudaMalloc(&sb.b.block_sums, sizeof(uint32_t) * (2 * ((tl + 2047) / 2048) + 2)));
  CK(cudaMalloc(&sb.b.work, sizeof(uint32_t) * 4));
  CK(cudaMemsetAsync(sb.b.work, 0, sizeof(uint32_t) * 4, B->ctx->stream));
  CK(cudaMalloc(&sb.sorted, sizeof(uint32_t) * pc));
  // the bins are what the batch can do without: they yield to what follows
  CKS(take_bins(B->ctx, sb.bins, bin_set_bytes(B->dim, B->edge, std::min(tl, BIN_TILES))));
  auto get = [&](auto** p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes);
    if (sb.bins.mem && out_of_memory(e)) {
      drop_bins(B->ctx, sb.bins);
      e = cudaMalloc(p, bytes);
    }
    return e;
  };
  CK(get(&sb.b.gpartial, sizeof(float) * size_t(tl) * MAX_GROUPS));
  CK(cudaMemsetAsync(sb.b.tile_count, 0, sizeof(uint32_t) * tl, B->ctx->stream));
  CK(cudaMemsetAsync(sb.b.tile_fill, 0, sizeof(uint32_t) * tl, B->ctx->stream));
  CK(get(&sb.partial, sizeof(float4) * size_t(tl) * block_nodes(B->dim, B->edge)));
  CK(get(&sb.partial_b, sizeof(float4) * size_t(tl) * block_nodes(B->dim, B->edge)));
  sb.bin_tiles = sb.bins.mem ? std::min(tl, BIN_TILES) : 0;
  sb.cap_scenes = sc;  // only now: after a failed allocation the next call starts over
  sb.cap_tiles = tl;
  sb.cap_particles = pc;
  sb.cap_edge = B->edge;
  return MPM_OK;
}

// Tile kernels a half of the batch runs: forward steps P2G and G2P, reverse steps the adjoint
// scatter and gather.
unsigned half_kernels(const mpm_batch* B, const SubBatch& sb) {
  return &sb == &B->fwd ? (1u << TK_P2G) | (1u << TK_G2P) : (1u << TK_P2G_ADJ) | (1u << TK_ADJ_GATHER);
}

int phase_of(int state) { return state == S_FWD ? PH_ROLL : state == S_RCM ? PH_RCM : PH_REV; }

// Lays the members of a sub-batch out in the batch's tile and particle spaces and uploads the
// scene table sources (selections, controllers, offsets).
mpm_status compose(mpm_batch* B, SubBatch& sb) {
  int tiles = 0, particles = 0;
  for (int i : sb.members) {
    tiles += B->slots[i].s->hp.n_tiles;
    particles += B->slots[i].s->N;
  }
  CKS(grow(B, sb, int(sb.members.size()), tiles, particles));
  sb.b.partial = sb.partial;
  sb.b.partial_b = sb.partial_b;
  cudaStream_t st = B->ctx->stream;
  if (!sb.members.empty()) {
    char* host = sb.staging[sb.turn];
    CK(cudaEventSynchronize(sb.copied[sb.turn]));  // the copy that last read this block (long done)
    SelectPar* sel = reinterpret_cast<SelectPar*>(host);
    CtrlPar* ctl = reinterpret_cast<CtrlPar*>(host + sb.off_ctrl);
    int* pb = reinterpret_cast<int*>(host + sb.off_pbase);
    int* tscene = reinterpret_cast<int*>(host + sb.off_tiles);
    int tb = 0, p0 = 0;
    pb[0] = 0;
    for (size_t m = 0; m < sb.members.size(); ++m) {
      mpm_scene* s = B->slots[sb.members[m]].s;
      sel[m] = s->hsel[phase_of(B->slots[sb.members[m]].state)];
      sel[m].tile_base = tb;
      sel[m].pbase = p0;
      ctl[m] = s->ctrl;
      ctl[m].gpart = sb.b.gpartial;
      ctl[m].active = sb.b.active;
      ctl[m].n_active = sb.b.n_active;
      ctl[m].whole = sb.members.size() == 1 ? 1 : 0;  // others' tiles share the active list otherwise
      std::fill(tscene + tb, tscene + tb + s->hp.n_tiles, int(m));
      tb += s->hp.n_tiles;
      p0 += s->N;
      pb[m + 1] = p0;
    }
    CK(cudaMemcpyAsync(sb.meta, host, sb.off_tiles + sizeof(int) * size_t(tb), cudaMemcpyHostToDevice, st));
    CK(cudaEventRecord(sb.copied[sb.turn], st));
    sb.turn ^= 1;
  }
  use_bins(sb.b, tiles <= sb.bin_tiles ? sb.bins : BinSet(), B->dim, B->edge, sb.bin_tiles, sb.sorted);
  sb.b.scenes = sb.cur;
  sb.b.tile_edge = B->edge;
  sb.b.n_scenes = int(sb.members.size());
  sb.b.scene_pbase = sb.pbase;
  sb.b.total_particles = particles;
  sb.b.total_tiles = tiles;
  sb.b.has_material = sb.b.occupied = 0;
  for (int m : sb.members) {
    sb.b.has_material |= B->slots[m].s->hp.gmat ? 1 : 0;
    sb.b.occupied += B->slots[m].tiles;
  }
  sb.composed += 1;
  sb.b.sm_count = B->ctx->sm_count;
  // a new workload key takes its shapes anew; an empty composition keeps the last key's shapes
  // and trials (a lockstep batch alternates each half between its members and nothing)
  const unsigned kernels = tunable(B->dim, sb.b, half_kernels(B, sb));
  if (!sb.members.empty() && (particles != sb.key_particles || tiles != sb.key_tiles || kernels != sb.key_kernels)) {
    default_launch(sb.b, B->ctx->sm_count);
    CKS(batch_tune_init(sb.tune, sb.b, B->dim, 0u));  // cached shapes, no trials yet
    sb.trial_wait = (kernels == 0 || batch_tune_cached(sb.b, B->dim, kernels)) ? 0 : kTrialWait;
    sb.key_particles = particles;
    sb.key_tiles = tiles;
    sb.key_kernels = kernels;
  }
  sb.need_keys = true;
  return MPM_OK;
}

// Asks for the active tiles of the half's last step, while they decide its CTA sizes.
mpm_status ask_tiles(mpm_batch* B, SubBatch& sb) {
  if (B->dim != 3 || sb.members.empty() || sb.seen_composed >= 0 || !few_tiles(3, sb.b, 2)) return MPM_OK;
  if (!sb.seen) {
    CK(cudaMallocHost(&sb.seen, sizeof(int)));
    CK(cudaEventCreateWithFlags(&sb.seen_at, cudaEventDisableTiming));
  }
  CK(cudaMemcpyAsync(sb.seen, sb.b.n_active, sizeof(int), cudaMemcpyDeviceToHost, B->ctx->stream));
  CK(cudaEventRecord(sb.seen_at, B->ctx->stream));
  sb.seen_composed = sb.composed;
  return MPM_OK;
}

// Looks at them, if they have arrived: a body that spread over more tiles leaves the wide CTAs.  Its
// composition's tiles are known only together, so its scenes' shares grow alike.
void look_at_tiles(mpm_batch* B, SubBatch& sb) {
  if (sb.seen_composed < 0) return;
  if (cudaEventQuery(sb.seen_at) != cudaSuccess) {
    cudaGetLastError();  // not ready is no failure
    return;
  }
  const bool same = sb.seen_composed == sb.composed;
  sb.seen_composed = -1;
  if (!same || *sb.seen <= sb.b.occupied) return;
  const unsigned before = tunable(B->dim, sb.b, ~0u);
  int sum = 0;
  for (int m : sb.members) {
    int& o = B->slots[m].tiles;
    o = int((long long)(o) * *sb.seen / sb.b.occupied) + 1;
    sum += o;
  }
  sb.b.occupied = sum;
  if (tunable(B->dim, sb.b, ~0u) != before) B->dirty = true;  // composed anew with other launch shapes
}

// Counts a step of the half's key; its trials start once the key has run kTrialWait steps.
mpm_status trial_clock(mpm_batch* B, SubBatch& sb) {
  if (sb.trial_wait > 0 && --sb.trial_wait == 0) CKS(batch_tune_init(sb.tune, sb.b, B->dim, sb.key_kernels));
  return MPM_OK;
}

mpm_status recompose(mpm_batch* B) {
  B->fwd.members.clear();
  B->rev.members.clear();
  for (int i = 0; i < int(B->slots.size()); ++i) {
    const int st = B->slots[i].state;
    if (st == S_FWD || st == S_RCM) B->fwd.members.push_back(i);
    if (st == S_REV) B->rev.members.push_back(i);
  }
  CKS(compose(B, B->fwd));
  CKS(compose(B, B->rev));
  B->dirty = false;
  return MPM_OK;
}

template <int D>
mpm_status forward_step(mpm_batch* B, cudaStream_t st) {
  SubBatch& sb = B->fwd;
  const int n = int(sb.members.size());
  if (n == 0) return MPM_OK;
  CK(launch_select(sb.dsel, n, sb.cur, st));
  for (int m = 0; m < n; ++m) {
    mpm_scene* s = B->slots[sb.members[m]].s;
    if (ctrl_reads_state(s->ctrl)) CK(ctrl_step_forward(s->hp, sb.cur + m, s->ctrl, st));
  }
  if (sb.need_keys) {
    CK(launch_keys<D>(sb.b, st));
    sb.need_keys = false;
  }
  CK(launch_sort<D>(sb.b, st));
  CKS(trial_clock(B, sb));
  batch_tune_begin(sb.tune, sb.b, D);
  {
    TuneScope ts(sb.tune, TK_P2G, st);
    CK(launch_p2g<D>(sb.b, false, st));
  }
  {
    TuneScope ts(sb.tune, TK_G2P, st);
    CK(launch_g2p<D>(sb.b, st));  // advances every member's forward counter, bins state n+1
  }
  return batch_tune_end(sb.tune, sb.b, D);
}

template <int D>
mpm_status reverse_step(mpm_batch* B, cudaStream_t st) {
  SubBatch& sb = B->rev;
  const int n = int(sb.members.size());
  if (n == 0) return MPM_OK;
  CK(launch_select(sb.dsel, n, sb.cur, st));
  CK(launch_keys<D>(sb.b, st, nullptr, sb.need_keys));
  sb.need_keys = false;
  for (int m = 0; m < n; ++m) {
    mpm_scene* s = B->slots[sb.members[m]].s;
    if (ctrl_reads_state(s->ctrl)) CK(ctrl_step_forward(s->hp, sb.cur + m, s->ctrl, st));
  }
  CK(launch_sort<D>(sb.b, st));
  CKS(trial_clock(B, sb));
  batch_tune_begin(sb.tune, sb.b, D);
  {
    TuneScope ts(sb.tune, TK_P2G_ADJ, st);
    CK(launch_p2g<D>(sb.b, true, st));
  }
  {
    TuneScope ts(sb.tune, TK_ADJ_GATHER, st);
    CK(launch_adj_gather<D>(sb.b, st));
  }
  CKS(batch_tune_end(sb.tune, sb.b, D));
  CK(ctrl_backward_batched(sb.cur, sb.dctrl, n, st));  // rewinds every member's reverse counter
  for (int m = 0; m < n; ++m) {
    mpm_scene* s = B->slots[sb.members[m]].s;
    if (ctrl_reads_state(s->ctrl)) CK(ctrl_scatter_x(s->hp, sb.cur + m, s->ctrl, st));
  }
  return MPM_OK;
}

// Start of the reverse work of segment sg (recompute from its checkpoint, then reverse steps).
mpm_status begin_segment(mpm_batch* B, Slot& sl) {
  mpm_scene* s = sl.s;
  const int L = std::min(s->roll_k, s->roll_T - sl.seg * s->roll_k);
  if (L > 1) {
    CKS(set_counter(s, s->d_step, s->roll_start + sl.seg * s->roll_k));
    sl.state = S_RCM;
    sl.left = L - 1;
  } else {
    sl.state = S_REV;
    sl.left = L;
  }
  B->dirty = true;
  return MPM_OK;
}

// Writes the counters the scenes' phase changes asked for (set_counter through the sink), in
// order, with as few launches as the list needs.
mpm_status flush_counters(mpm_batch* B) {
  cudaStream_t st = B->ctx->stream;
  for (size_t i0 = 0; i0 < B->pend_ctr.size(); i0 += INT_LIST_MAX) {
    IntPtrList l;
    l.n = int(std::min<size_t>(INT_LIST_MAX, B->pend_ctr.size() - i0));
    for (int i = 0; i < l.n; ++i) {
      l.ptr[i] = B->pend_ctr[i0 + i].first;
      l.val[i] = B->pend_ctr[i0 + i].second;
    }
    CK(launch_set_int_list(l, st));
  }
  B->pend_ctr.clear();
  return MPM_OK;
}

// Finished requests, closed together at the end of a tick: the reverse passes' scenes get the bin keys of their current state back, then
// one gather and one copy read every finished scene's status word.
mpm_status finish_requests(mpm_batch* B) {
  if (B->finishing.empty()) return MPM_OK;
  cudaStream_t st = B->ctx->stream;
  for (int idx : B->finishing)
    if (B->slots[idx].want_grad) CKS(restore_keys(B->slots[idx].s));
  const int n = int(B->finishing.size());
  if (n > B->status_cap) {
    CK(cudaStreamSynchronize(st));
    dfree(B->d_status);
    B->status_cap = 0;
    CK(cudaMalloc(&B->d_status, sizeof(int) * n));
    B->status_cap = n;
  }
  for (int i0 = 0; i0 < n; i0 += INT_LIST_MAX) {
    IntPtrList l;
    l.n = std::min(INT_LIST_MAX, n - i0);
    for (int i = 0; i < l.n; ++i) l.ptr[i] = B->slots[B->finishing[i0 + i]].s->d_status;
    CK(launch_gather_ints(l, B->d_status + i0, st));
  }
  std::vector<int> h(n);
  CK(cudaMemcpyAsync(h.data(), B->d_status, sizeof(int) * n, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  for (int i = 0; i < n; ++i) {
    Slot& sl = B->slots[B->finishing[i]];
    sl.status = mpm_status(h[i]);
    sl.state = S_DONE;
  }
  B->finishing.clear();
  return MPM_OK;
}

// Slot bookkeeping after one batched step.  Counter writes are collected (one launch for all
// scenes), finished requests are closed together.
mpm_status advance(mpm_batch* B) {
  for (int idx = 0; idx < int(B->slots.size()); ++idx) {
    Slot& sl = B->slots[idx];
    if (sl.state != S_FWD && sl.state != S_RCM && sl.state != S_REV) continue;
    mpm_scene* s = sl.s;
    s->ctr_sink = &B->pend_ctr;
    mpm_status st = MPM_OK;
    if (sl.state == S_FWD) {
      if (++sl.done_steps >= sl.T) {
        s->step += sl.T;
        s->have_rollout = true;
        if (sl.want_grad) {
          st = seed_mean_x0(s);
          sl.seg = s->roll_nseg - 1;
          if (st == MPM_OK) st = begin_segment(B, sl);
        } else {
          sl.state = S_CLOSING;  // status read in finish_requests
          B->finishing.push_back(idx);
          B->dirty = true;
        }
      }
    } else if (sl.state == S_RCM) {
      if (--sl.left <= 0) {
        const int L = std::min(s->roll_k, s->roll_T - sl.seg * s->roll_k);
        sl.state = S_REV;
        sl.left = L;
        B->dirty = true;
      }
    } else if (--sl.left <= 0) {  // S_REV
      if (--sl.seg >= 0) {
        st = begin_segment(B, sl);
      } else {
        finish_backward_quiet(s);
        sl.state = S_CLOSING;
        B->finishing.push_back(idx);
        B->dirty = true;
      }
    }
    s->ctr_sink = nullptr;
    if (st != MPM_OK) return st;
  }
  return flush_counters(B);
}

size_t request_bytes(const mpm_scene* s, int T, int k) {
  const int nseg = (T + k - 1) / k;
  return (size_t(nseg) + size_t(k - 1)) * s->state_bytes;
}

int sqrt_interval(int T) { return T <= 16 ? 1 : int(std::ceil(std::sqrt(double(T)))); }

// Checkpoint interval of a request.  Without a memory budget a gradient request keeps every state,
// as mpm_rollout does, while its states are at most KEEP_ONE bytes and those of the context's scenes
// whose requests did so KEEP_ALL (a scene holds its states until its next rollout of another shape or
// its end): nothing is recomputed, and its scene changes sub-batch once instead of twice a segment.
// That takes 8-20 % less time at every size tried (batches of 16 x 3 MB to 2 x 522 MB of states:
// 3721 -> 3426 us to 11523 -> 9300 us), so the bounds are not where it stops paying: they keep what
// scenes hold between requests, unasked, to a sixty-fourth of the device's memory, and one request
// to a sixteenth of that.  With a budget the admission counts checkpoints, and the interval stays
// ceil(sqrt(T)).
constexpr size_t KEEP_ONE = size_t(256) << 20, KEEP_ALL = size_t(4) << 30;
int request_interval(const mpm_batch* B, const mpm_scene* s, int T, int want_grad) {
  if (!want_grad || B->budget != 0) return sqrt_interval(T);
  const size_t need = request_bytes(s, T, 1);
  return need <= KEEP_ONE && B->ctx->kept_bytes - s->kept_bytes + need <= KEEP_ALL ? 1 : sqrt_interval(T);
}

// Up to max_steps batched steps.
mpm_status run_steps(mpm_batch* B, int max_steps) {
  look_at_tiles(B, B->fwd);
  look_at_tiles(B, B->rev);
  for (int it = 0; it < max_steps; ++it) {
    bool busy = false;
    for (const Slot& sl : B->slots) busy = busy || sl.state == S_FWD || sl.state == S_RCM || sl.state == S_REV;
    if (!busy) break;
    if (B->dirty) CKS(recompose(B));
    // the two halves touch disjoint scenes and buffers: the reverse half runs on the second
    // stream beside the forward half, joined before the bookkeeping
    cudaStream_t ms = B->ctx->stream, as = B->ctx->aux;
    CK(cudaEventRecord(B->fork, ms));
    CK(cudaStreamWaitEvent(as, B->fork, 0));
    if (B->dim == 2) {
      CKS(forward_step<2>(B, ms));
      CKS(reverse_step<2>(B, as));
    } else {
      CKS(forward_step<3>(B, ms));
      CKS(reverse_step<3>(B, as));
    }
    CK(cudaEventRecord(B->join, as));
    CK(cudaStreamWaitEvent(ms, B->join, 0));
    CKS(advance(B));
  }
  CKS(ask_tiles(B, B->fwd));
  return ask_tiles(B, B->rev);
}

}  // namespace

extern "C" {

mpm_status mpm_batch_create(mpm_ctx* ctx, int dim, size_t mem_budget, mpm_batch** out) {
  if (!ctx || !out || (dim != 2 && dim != 3)) return MPM_ERR_ARG;
  mpm_batch* B = new (std::nothrow) mpm_batch();
  if (!B) return MPM_ERR_OOM;
  B->ctx = ctx;
  B->dim = dim;
  B->budget = mem_budget;
  if (cudaEventCreateWithFlags(&B->fork, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&B->join, cudaEventDisableTiming) != cudaSuccess) {
    if (B->fork) cudaEventDestroy(B->fork);
    delete B;
    return MPM_ERR_CUDA;
  }
  ctx->live.fetch_add(1);
  *out = B;
  return MPM_OK;
}

mpm_status mpm_batch_destroy(mpm_batch* B) {
  if (!B) return MPM_ERR_ARG;
  cudaStreamSynchronize(B->ctx->stream);
  cudaStreamSynchronize(B->ctx->aux);
  for (Slot& sl : B->slots)  // the scenes of unreleased slots are the caller's again
    if (sl.state != S_FREE && sl.s) sl.s->batch_refs -= 1;
  free_sub(B->ctx, B->fwd);
  free_sub(B->ctx, B->rev);
  dfree(B->d_status);
  cudaEventDestroy(B->fork);
  cudaEventDestroy(B->join);
  B->ctx->live.fetch_sub(1);
  delete B;
  return MPM_OK;
}

mpm_status mpm_batch_admit(mpm_batch* B, mpm_scene* s, int n_steps, int want_grad, int* slot) {
  if (!B || !s || !slot || n_steps < 1) return MPM_ERR_ARG;
  *slot = -1;
  if (s->dim != B->dim || s->impl != MPM_IMPL_TILED || s->ctx != B->ctx) return MPM_ERR_ARG;
  bool empty = true;
  for (const Slot& sl : B->slots) {
    if (sl.s == s && sl.state != S_FREE) return MPM_ERR_STATE;  // a scene runs in one slot at a time
    empty = empty && sl.state == S_FREE;
  }
  // one tile edge per batch: the tile kernels of a launch are instantiated for one edge
  if (!empty && s->b.tile_edge != B->edge) return MPM_ERR_ARG;
  int k = request_interval(B, s, n_steps, want_grad);
  const size_t need = request_bytes(s, n_steps, k);
  if (B->budget != 0 && B->used + need > B->budget) return MPM_OK;  // no room now: *slot stays -1
  int idx = -1;
  for (int i = 0; i < int(B->slots.size()); ++i)
    if (B->slots[i].state == S_FREE) {
      idx = i;
      break;
    }
  if (idx < 0) {
    B->slots.push_back(Slot());
    idx = int(B->slots.size()) - 1;
  }
  mpm_status st = prepare_rollout(s, n_steps, k, 0);
  if (st == MPM_ERR_OOM && k != sqrt_interval(n_steps)) {
    k = sqrt_interval(n_steps);  // the smaller store
    st = prepare_rollout(s, n_steps, k, 0);
  }
  if (st != MPM_OK) return st;
  if (k != sqrt_interval(n_steps)) {  // every state kept, uncalled for: counted until they are freed
    B->ctx->kept_bytes += request_bytes(s, n_steps, k) - s->kept_bytes;
    s->kept_bytes = request_bytes(s, n_steps, k);
  }
  Slot& sl = B->slots[idx];
  sl = Slot();
  if (empty) B->edge = s->b.tile_edge;
  sl.s = s;
  sl.state = S_FWD;
  sl.T = n_steps;
  sl.want_grad = want_grad;
  sl.tiles = s->b.occupied;
  sl.mem = request_bytes(s, n_steps, k);
  B->used += sl.mem;
  B->dirty = true;
  s->batch_refs += 1;
  s->keys_stale = true;
  *slot = idx;
  return MPM_OK;
}

mpm_status mpm_batch_tick(mpm_batch* B, int max_steps) {
  if (!B || max_steps < 1) return MPM_ERR_ARG;
  const mpm_status ran = run_steps(B, max_steps);
  // the requests that finished are closed even if a later step could not run (the arrays of a new
  // composition that do not fit): their release may be what makes room
  const mpm_status closed = finish_requests(B);
  CKS(ran);
  CKS(closed);
  CK(cudaGetLastError());
  return MPM_OK;
}

mpm_status mpm_batch_poll(mpm_batch* B, int slot, int* done) {
  if (!B || !done || slot < 0 || slot >= int(B->slots.size()) || B->slots[slot].state == S_FREE) return MPM_ERR_ARG;
  const Slot& sl = B->slots[slot];
  *done = sl.state == S_DONE ? 1 : 0;
  if (sl.state == S_DONE && sl.status != MPM_OK) return sl.status;
  return MPM_OK;
}

mpm_status mpm_batch_release(mpm_batch* B, int slot) {
  if (!B || slot < 0 || slot >= int(B->slots.size()) || B->slots[slot].state == S_FREE) return MPM_ERR_ARG;
  Slot& sl = B->slots[slot];
  if (sl.state != S_DONE) return MPM_ERR_STATE;
  B->used -= sl.mem;
  sl.s->batch_refs -= 1;
  sl = Slot();
  B->dirty = true;
  return MPM_OK;
}

}  // extern "C"

// Several small levels in one launch. Included by kernels_s32.cu / kernels_s64.cu.
//
// A level of up to some 10^5 candidates is a few microseconds of work; what it
// cost was eight or nine launches and a round trip to the host (55-110 us). Here
// a cooperative launch (every block resident, so that they may wait for one
// another) runs the levels one after another: the blocks build a level with the
// code of the ordinary kernels (lanes_run for path A, group_run otherwise) and
// meet at a barrier, where block 0 closes the level - it records its counters,
// plans the next one from the level sizes, which it keeps in shared memory (the listing of paragraph "A
// generic program synthesiser": unary operators on level k - 1, binary operators
// on every split of k - 1) or stops. Ids are reserved exactly, so a level has no
// holes to close. Candidates that met an unpublished slot (rare, see the kernels)
// are settled by further steps over the deferred list.
//
// It stops before a level that is too large (its own launches then pay for
// themselves), at the first solution, when the arena is full or a check fails;
// the host commits the levels from their records and goes on from there. The
// wait at the barrier is bounded; should it run out, the launch ends without a
// record and the context has to be reset.
//
// Measured (one GB300): a level of 10^1 to 10^4 candidates in 10-15 us inside a
// solve, 28-45 us as a call of its own, against 55-110 us (up to 1 ms on wide
// matrices, before the group kernels); a tiny problem's reset and solve 135 us
// instead of 170 or 168 instead of 319, by the problem (about 100 are the
// caller's Python), levels 1-10 of 250 traces 4.44 ms instead of 4.66. Two blocks per SM (up to 128 registers, three
// kinds of step in one kernel): beyond kSmallCandidates a level's own launches
// are faster.
#pragma once

#include "lsyn_group.cuh"
#include "lsyn_lanes.cuh"
#include "lsyn_text.cuh"

namespace lsyn {

constexpr unsigned kBarrierPolls = 1u << 22;  // seconds; a level's step takes microseconds
enum : int { kStepStop = 0, kStepLevel = 1, kStepList = 2 };
constexpr int kMaxListSteps = 48;

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// What every block needs for a step: block 0 makes it in shared memory and
// copies it to the state, the others copy it from there.
struct SmallStep {
  int step, k;
  uint32_t u_first, u_count, u_warps, u_batch, b_warps, b_batch, list_from, list_to;
  unsigned long long b_items;
  BinaryPlan plan;
};
static_assert(sizeof(SmallStep) <= sizeof(SmallState::words), "a step fits the state");

// Block 0's own: the levels so far.
struct SmallLocal {
  int list_steps, n_done;
  uint32_t start;
  unsigned long long t0;
  uint32_t level_start[kSmallLevels + 1], level_n[kSmallLevels + 1];
};

// Plans level s->k; false (and nothing planned) if it is too large.
template <bool kGroups>
__device__ bool small_plan(const CacheView& cv, const SmallArgs& a, const SmallLocal* o, SmallStep* s) {
  const int k = s->k;
  s->u_count = 0;
  s->b_items = 0;
  if (k == 1) return true;
  unsigned long long cand = 0, pairs = 0;
  BinaryPlan& plan = s->plan;
  plan.n_splits = 0;
  plan.ops = a.b_ops;
  if (a.u_ops) {
    s->u_first = o->level_start[k - 1];
    s->u_count = o->level_n[k - 1];
    cand += (unsigned long long)s->u_count * unsigned(__popc(a.u_ops));
  }
  if (a.b_ops && k >= 3)
    for (int i = 1; 2 * i <= k - 1; ++i) {
      const int j = k - 1 - i;
      const uint32_t ni = o->level_n[i], nj = o->level_n[j];
      if (!ni || !nj || (i == j && ni < 2)) continue;
      Split& S = plan.s[plan.n_splits++];
      const bool ij = i == j || ni <= nj;  // the smaller level on the left
      S.left_start = o->level_start[ij ? i : j];
      S.left_n = ij ? ni : nj;
      S.right_start = o->level_start[ij ? j : i];
      S.right_n = ij ? nj : ni;
      S.tri = i == j ? 1u : 0u;
      S.pairs_begin = pairs;
      S.pairs = S.tri ? (unsigned long long)ni * (ni - 1) / 2 : (unsigned long long)ni * nj;
      pairs += S.pairs;
    }
  plan.total_pairs = pairs;
  cand += pairs * unsigned(__popc(a.b_ops));
  if (cand > a.max_candidates || o->start + cand > a.max_total) return false;
  if constexpr (kGroups) {
    GroupWork g;
    group_shape(cv, kGroupUnary, s->u_count, gridDim.x * unsigned(kGroupMaxWarps), &g);
    s->u_warps = g.warps;
    s->u_batch = g.batch;
    group_shape(cv, kGroupBinary, pairs, gridDim.x * unsigned(kGroupMaxWarps), &g);
    s->b_warps = g.warps;
    s->b_batch = g.batch;
    s->b_items = group_items(&plan, unsigned(g.batch));
  } else {
    s->b_items = pairs;
  }
  return true;
}

// Closes the step that every block has finished and decides on the next one
// (thread 0 of block 0, while all others wait).
template <bool kGroups>
__device__ void small_close(const CacheView& cv, const SmallArgs& a, SmallState* st, SmallLocal* o, SmallStep* s,
                            bool begin) {
  DevCounters* c = cv.ctr;
  if (begin) {
    for (int i = 1; i < a.first_level; ++i) {
      o->level_start[i] = a.level_start[i];
      o->level_n[i] = a.level_n[i];
    }
    s->k = a.first_level;
    o->start = a.start;
    o->n_done = 0;
    st->text_status = -1;
  } else {
    SmallLevel r;
    r.sol = __ldcg(&c->sol);
    r.full = __ldcg(&c->full);
    r.solved = __ldcg(&c->solved);
    r.error = __ldcg(&c->error);
    r.defer_overflow = __ldcg(&c->defer_overflow);
    r.holes = __ldcg(&c->holes_n);
    r.deferred = min(__ldcg(&c->defer_n[0]), cv.defer_cap);
    r.total = min(__ldcg(&c->n_entries), cv.max_entries);
#pragma unroll
    for (int i = 0; i < kLaunchKinds; ++i) {
      r.built_k[i] = __ldcg(&c->built_k[i]);
      r.inserted_k[i] = __ldcg(&c->inserted_k[i]);
    }
    const bool bad = r.error != 0u || r.defer_overflow != 0u, more = !bad && r.deferred > s->list_to;
    if (more && o->list_steps < kMaxListSteps) {
      s->list_from = s->list_to;
      s->list_to = r.deferred;
      ++o->list_steps;
      s->step = kStepList;
      return;
    }
    r.unsettled = more ? 1u : 0u;
    r.ns = global_ns() - o->t0;
    st->rec[o->n_done++] = r;
    if (bad || more || r.solved || r.full || r.holes || s->k >= a.last_level) {
      if (r.solved && !bad && !more)
        reconstruct_text(cv.prov, r.sol, st->text, unsigned(sizeof(st->text)), &st->text_status);
      s->step = kStepStop;
      return;
    }
    o->level_start[s->k] = o->start;
    o->level_n[s->k] = r.total - o->start;
    o->start = r.total;
    ++s->k;
  }
  if (!small_plan<kGroups>(cv, a, o, s)) {
    s->step = kStepStop;
    return;
  }
  // as k_level_begin
  c->full = 0;
  c->solved = 0;
  c->error = 0;
  c->timed_out = 0;
  c->defer_n[0] = c->defer_n[1] = 0;
  c->defer_overflow = 0;
  c->holes_n = 0;
#pragma unroll
  for (int i = 0; i < kLaunchKinds; ++i) c->built_k[i] = c->inserted_k[i] = 0;
  c->sol = ~0ull;
  o->t0 = global_ns();
  s->list_from = s->list_to = 0;
  o->list_steps = 0;
  s->step = kStepLevel;
}

// The next step, for every block: once all blocks have finished the last one
// (at the beginning there is none to wait for), block 0 closes it and lets the
// others go. False if a wait ran out.
template <bool kGroups>
__device__ bool small_next(const CacheView& cv, const SmallArgs& a, SmallState* st, SmallLocal* o, SmallStep* s,
                           unsigned turn, bool begin) {
  __shared__ unsigned s_ok;
  unsigned* words = reinterpret_cast<unsigned*>(s);
  __syncthreads();  // the block's stores, before its arrival
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) {
      unsigned polls = 0;
      if (!begin) {
        while (ld_acquire_u32(&st->arrived) != gridDim.x - 1u && ++polls < kBarrierPolls) __nanosleep(20);
        st->arrived = 0u;
      }
      s_ok = polls < kBarrierPolls ? 1u : 0u;
      __threadfence();
      if (s_ok) small_close<kGroups>(cv, a, st, o, s, begin);
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < sizeof(SmallStep) / 4; i += blockDim.x) st->words[i] = words[i];
    if (threadIdx.x == 0 && s->step == kStepStop) {
      st->n_done = o->n_done;
      st->call = a.call;
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_ok) {
      __threadfence();
      st_release_u32(&st->turn, turn + 1u);
    }
  } else {
    if (threadIdx.x == 0) {
      if (!begin) {
        __threadfence();
        atomicAdd(&st->arrived, 1u);
      }
      unsigned polls = 0;
      while (ld_acquire_u32(&st->turn) == turn && ++polls < kBarrierPolls) __nanosleep(20);
      s_ok = polls < kBarrierPolls ? 1u : 0u;
      if (!s_ok) atomicExch(&cv.ctr->error, 6u);
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < sizeof(SmallStep) / 4; i += blockDim.x) words[i] = __ldcg(st->words + i);
    __syncthreads();
  }
  return s_ok != 0u;
}

template <typename W, int V>
__global__ void __launch_bounds__(256, 2) k_small_lanes(CacheView cv, const __grid_constant__ SmallArgs a,
                                                        SmallState* st) {
  __shared__ SmallStep s;
  __shared__ SmallLocal own;
  unsigned turn = a.turn;
  for (bool begin = true;; begin = false, ++turn) {
    if (!small_next<false>(cv, a, st, &own, &s, turn, begin)) return;
    if (s.step == kStepStop) return;
    LanesWork w{};
    w.exact = 1;
    if (s.step == kStepLevel && s.k > 1) {
      w.total = s.u_count;
      w.first = s.u_first;
      w.ops = a.u_ops;
      lanes_run<W, V, kLanesUnary, true, 15u>(cv, w, s.plan);
      w.total = s.b_items;
      w.ops = a.b_ops;
      lanes_run<W, V, kLanesBinary, true, 15u>(cv, w, s.plan);
    } else {
      const bool list = s.step == kStepList;
      w.list = list ? cv.defer_out : nullptr;
      w.list_n = cv.defer_out_n;
      w.list_cap = s.list_to;
      w.list_from = s.list_from;
      w.atoms = list ? 0u : a.n_props;
      w.settle = 1;
      lanes_run<W, V, kLanesList, true, 15u>(cv, w, s.plan);
    }
  }
}

template <typename W, bool MP>
__global__ void __launch_bounds__(256, 2) k_small_group(CacheView cv, const __grid_constant__ SmallArgs a,
                                                        SmallState* st) {
  extern __shared__ __align__(128) unsigned char group_mem[];
  __shared__ SmallStep s;
  __shared__ SmallLocal own;
  unsigned turn = a.turn;
  for (bool begin = true;; begin = false, ++turn) {
    if (!small_next<true>(cv, a, st, &own, &s, turn, begin)) return;
    if (s.step == kStepStop) return;
    GroupWork w{};
    if (s.step == kStepLevel && s.k > 1) {
      if (s.u_count) {
        w.warps = int(s.u_warps);
        w.batch = int(s.u_batch);
        w.first = s.u_first;
        w.count = s.u_count;
        w.ops = a.u_ops;
        w.total = (s.u_count + s.u_batch - 1u) / s.u_batch;
        group_run<W, kGroupUnary, MP>(cv, w, s.plan, group_mem);
      }
      __syncthreads();  // the block's groups are cut anew
      if (s.b_items) {
        w.warps = int(s.b_warps);
        w.batch = int(s.b_batch);
        w.ops = a.b_ops;
        w.total = s.b_items;
        group_run<W, kGroupBinary, MP>(cv, w, s.plan, group_mem);
      }
    } else {
      const bool list = s.step == kStepList;
      w.list = list ? cv.defer_out : nullptr;
      w.list_n = cv.defer_out_n;
      w.list_cap = s.list_to;
      w.list_from = s.list_from;
      w.atoms = list ? 0u : a.n_props;
      w.settle = 1;
      w.warps = int(a.list_warps);
      w.batch = 1;
      group_run<W, kGroupList, MP>(cv, w, s.plan, group_mem);
    }
  }
}

// ---------------------------------------------------------------------------
// Launcher
// ---------------------------------------------------------------------------
// The limit of a kernel's dynamic shared memory belongs to the function, not to
// a context or a launch: raised once, to all that a block may have beside the
// kernel's static shared memory. (Set to each context's own need, it went down
// under the contexts with wider matrices, whose launches were then refused.)
template <typename W, bool MP>
cudaError_t small_group_limit() {
  static const cudaError_t set = [] {
    const void* fn = (const void*)k_small_group<W, MP>;
    cudaFuncAttributes fa{};
    int dev = 0, optin = 0;
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - int(fa.sharedSizeBytes));
    return e;
  }();
  return set;
}

template <typename W>
cudaError_t SmallKernels<W>::prepare(const CacheView& cv, int sms, SmallLaunch* out) {
  const void* fn = nullptr;
  size_t smem = 0;
  switch (cv.vecs) {
    case 1: fn = (const void*)k_small_lanes<W, 1>; break;
    case 2: fn = (const void*)k_small_lanes<W, 2>; break;
    case 4: fn = (const void*)k_small_lanes<W, 4>; break;
    case 8: fn = (const void*)k_small_lanes<W, 8>; break;
    default: fn = cv.planes > 1 ? (const void*)k_small_group<W, true> : (const void*)k_small_group<W, false>;
  }
  unsigned blocks_per_sm = 2;
  out->list_warps = 0;
  if (cv.vecs >= 32u) {
    // shared memory for every cut of a block into groups that a level may take
    GroupWork g;
    for (int per_sm = 2; per_sm >= 1; --per_sm) {
      const unsigned resident = unsigned(sms * per_sm * kGroupMaxWarps);
      smem = 0;
      for (int mode : {kGroupUnary, kGroupBinary, kGroupList})
        for (unsigned long long work = 1; work < (1ull << 32); work *= 2) {
          group_shape(cv, mode, work, resident, &g);
          smem = std::max(smem, group_smem(mode, cv.vecs, g.warps, g.batch) * size_t(kGroupMaxWarps / g.warps));
        }
      blocks_per_sm = unsigned(per_sm);
      if (smem <= 100 * 1024) break;  // two blocks fit an SM
    }
    const cudaError_t e = cv.planes > 1 ? small_group_limit<W, true>() : small_group_limit<W, false>();
    if (e != cudaSuccess) return e;
    group_shape(cv, kGroupList, 1, unsigned(sms) * blocks_per_sm * unsigned(kGroupMaxWarps), &g);
    out->list_warps = unsigned(g.warps);
  }
  out->fn = fn;
  out->smem = smem;
  out->blocks = unsigned(sms) * std::min(blocks_per_sm, unsigned(occupancy_blocks(fn, 256, smem)));
  return cudaSuccess;
}

template <typename W>
cudaError_t SmallKernels<W>::run(const CacheView& cv, const SmallLaunch& how, const SmallArgs& args, SmallState* st,
                                 cudaStream_t stream) {
  SmallArgs a = args;
  CacheView v = cv;
  a.list_warps = how.list_warps;
  void* params[] = {&v, &a, &st};
  return cudaLaunchCooperativeKernel(how.fn, dim3(how.blocks), dim3(256), params, how.smem, stream);
}

}  // namespace lsyn

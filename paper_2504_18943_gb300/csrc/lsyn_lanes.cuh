// Level kernels of path A (matrices of at most 128 bytes), included by
// kernels_a32.cu / kernels_a64.cu: V neighbouring lanes hold a CM, one vector each
// (V = 1, 2, 4 or 8), and build the four candidates of a row or pair at once;
// a warp takes 32 / V rows or pairs at a time and settles their candidates
// together, as path C does.
//
// What bounds them: the rate of random accesses (a table sector per candidate,
// a row per duplicate, row, provenance, slot and hash words per insert), and at
// small levels the chain of round trips. So rows are read and written by
// neighbouring lanes (whole sectors in one access), the loads of a warp's
// candidates are in flight together, ids come from one atomic a warp batch and
// the claimed slots are published after one fence a batch. A lane holds 4 x 16
// bytes of candidates whatever V is, where a thread for a whole CM held 4 V
// vectors (142 registers and one block per SM for 128-byte CMs). With four
// blocks per SM (64 registers, no spills; five or a prefetch of the next
// operands spill and lose 8-20 %) they are bound by instructions: about 800 per
// warp batch, 55-60 % of issue slots.
//
// Measured against one thread per CM (complete levels, one GB300): 30 traces
// (120 bytes), four propositions, levels 1-10 in 2.6 ms instead of 5.2, the
// last level's binary launch 13.2 G candidates/s instead of 4.8; 14 traces (56
// bytes), the paper's grammar, levels 1-15 in 8.2 ms instead of 8.9: up to 2.5x
// faster on launches of 10^5 to 10^7 candidates, 22.3 G/s at 28 M. (A loop with
// the same accesses and nothing else - a random bucket a candidate, a random
// 64-byte row of 4 GiB for 27 of 32, a claim and a row written for 5 - does 20 G/s.)
#pragma once

#include "lsyn_device.cuh"

namespace lsyn {

enum : int { kLanesUnary = 0, kLanesBinary = 1, kLanesList = 2 };

// Probes of a pending slot (about a microsecond each) before a candidate is deferred.
constexpr unsigned kLanesWaits = 8;
struct LanesWork {
  unsigned long long total;       // rows or pairs (a list reads its own length)
  uint32_t first, ops;            // unary: first row; enabled operators (4 bits)
  const unsigned long long* list; // list mode: descriptors, or NULL for the atoms
  const unsigned int* list_n;
  unsigned int list_cap, atoms;
  unsigned int list_from;         // list mode: first descriptor
  int exact;                      // 1: reserve exactly the ids that the claims need (as cv.chunk 1)
  int settle;                     // 1: goes on after a solution (deferred candidates)
};

// The work of one launch or, with kFresh, of one step of a launch that builds
// several levels: rows of levels that the same launch built are then read past
// L1 (nothing orders L1 with the other SMs' writes).
//
// kOps: the operators compiled in (4 bits; lw.ops is a subset of them): all, or
// those of the paper's grammar (not, X, F; and, U), whose launches then hash,
// compare and write a quarter less. 64-byte matrices, 92 M candidates of that
// grammar: 886 + 3690 us (unary + binary) with all four compiled in, 859 + 3455
// with three (now 919 + 3932 with ids exactly as claimed, 876 + 3184 with ids
// ahead, see ctx_level_plan). Two operators compiled in were not tried: no grammar
// here has them.
template <typename W, int V, int MODE, bool kFresh, unsigned kOps>
__device__ __forceinline__ void lanes_run(const CacheView& cv, const LanesWork& lw, const BinaryPlan& plan) {
  constexpr unsigned kKind = MODE == kLanesUnary ? kKindUnary : MODE == kLanesBinary ? kKindBinary : kKindOther;
  auto read = [](const uint4* p) { return kFresh ? __ldcg(p) : __ldg(p); };
  constexpr int NG = 32 / V;                          // rows, pairs or descriptors per warp batch
  constexpr int NO = MODE == kLanesList ? 1 : 4;      // candidates of each
  constexpr int R = NO == 4 && V < 4 ? 4 / V : 1;     // candidates that a lane probes for
  const int lane = threadIdx.x & 31, l = lane & (V - 1), g0 = lane & ~(V - 1);
  // candidate r of lane l, and where candidate o is probed
  auto cand_of = [](int ln, int r) { return NO == 1 ? 0 : V == 8 ? ln >> 1 : V == 4 ? ln : ln * R + r; };
  auto owner_of = [](int o) { return NO == 1 ? 0 : V >= 4 ? o * (V / 4) : o / R; };
  const bool owner = NO == 1 ? l == 0 : V == 8 ? (l & 1) == 0 : true;
  // x of the lane that probes for candidate o of this lane's group
  auto from_owner = [&](uint32_t x, int o) { return V == 1 ? x : __shfl_sync(kFull, x, g0 + owner_of(o)); };

  __shared__ uint4 s_const[3][V];  // hash multipliers, labels, length masks
  if (threadIdx.x < V) {
    s_const[0][threadIdx.x] = cv.hmul[threadIdx.x];
    s_const[1][threadIdx.x] = cv.label[threadIdx.x];
    s_const[2][threadIdx.x] = cv.lenmask[threadIdx.x];
  }
  __syncthreads();
  unsigned long long total = lw.total;
  if constexpr (MODE == kLanesList) total = lw.list ? min(__ldcg(lw.list_n), lw.list_cap) - lw.list_from : lw.atoms;
  const uint32_t ops = MODE == kLanesList ? 1u : lw.ops & 0xFu;
  auto enabled = [](int o) { return MODE == kLanesList || ((kOps >> o) & 1u) != 0u; };
  const unsigned long long warp = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) >> 5;
  const unsigned long long nwarps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
  constexpr int kProbing = WarpDedup::kProbing, kDone = WarpDedup::kDone, kClaimed = WarpDedup::kClaimed;
  constexpr int kCompare = 4, kWait = 5;
  uint32_t pend_pos[R], pend_tag[R], pend_id[R];  // claimed slots whose rows are written: id + 1, 0 = none
#pragma unroll
  for (int r = 0; r < R; ++r) pend_pos[r] = pend_tag[r] = pend_id[r] = 0;
  unsigned long long built = 0;
  static_assert(sizeof(built) == sizeof(cv.ctr->built_k[0]), "a warp's share of a level may need all of its bits");
  unsigned inserted = 0, iter = 0;  // (ids fit 32 bits)
  IdStock ids;
  // All warps' reservations meet at one counter. In a large level a warp
  // reserves up to kLanesAhead ids more than its claims need, in the same
  // atomic; fewer towards its last batch, so that almost none are left over
  // (holes, to be closed).
  const bool ahead = cv.chunk > 1u && !lw.exact;
  // batches after this one (with `ahead`, the level's candidates fit 32 bits)
  unsigned batches = total > warp * NG ? unsigned((total - warp * NG - 1) / (nwarps * NG)) : 0u;
  bool full = false;  // the arena is full: the specification check only

  // As WarpDedup::flush: the warp barrier orders the other lanes' row stores
  // before the fence, the fence before the slot stores.
  auto flush = [&]() {
    bool any = false;
#pragma unroll
    for (int r = 0; r < R; ++r) any = any || pend_id[r] != 0u;
    if (!__any_sync(kFull, any)) return;
    __syncwarp();
    fence_acq_rel_gpu();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (pend_id[r]) st_relaxed(cv.table + pend_pos[r], ((unsigned long long)pend_tag[r] << 32) | pend_id[r]);
      pend_id[r] = 0;
    }
  };

  auto row = [&](uint32_t id) { return cv.arena + size_t(id) * V; };
  // operands of this lane's row, pair or descriptor `i`
  struct Item {
    uint32_t a_id, b_id, op;
    bool valid;
  };
  auto load_item = [&](unsigned long long i, Item& it, uint4& a, uint4& b) {
    it.a_id = it.b_id = it.op = 0;
    it.valid = i < total;
    a = b = make_uint4(0u, 0u, 0u, 0u);
    if (!it.valid) return;
    if constexpr (MODE == kLanesUnary) {
      it.a_id = lw.first + uint32_t(i);
      a = read(row(it.a_id) + l);
    } else if constexpr (MODE == kLanesBinary) {
      int sp = 0;
      while (sp + 1 < plan.n_splits && plan.s[sp + 1].pairs_begin <= i) ++sp;
      const Split& S = plan.s[sp];
      const uint2 ab = split_pair(S, i - S.pairs_begin, false);
      it.a_id = S.left_start + ab.x;
      it.b_id = S.right_start + ab.y;
      a = read(row(it.a_id) + l);
      b = read(row(it.b_id) + l);
    } else {
      const uint64_t d = lw.list ? __ldcg(lw.list + lw.list_from + i) : pack_desc(kAtom, uint32_t(i), 0);
      it.op = desc_op(d);
      it.a_id = desc_left(d);
      it.b_id = desc_right(d);
      a = read((it.op == kAtom ? cv.atoms + size_t(it.a_id) * V : row(it.a_id)) + l);
      if (it.op == kAnd || it.op == kOr || it.op == kUntil) b = read(row(it.b_id) + l);
    }
  };

  for (unsigned long long base = warp * NG; base < total; base += nwarps * NG, ++iter, --batches) {
    // The flags are polled every few batches only (every warp's polls go to one
    // L2 slice, which the id counter's atomics load already); a warp whose own
    // claims found the arena full stops claiming at once.
    if ((iter & 3u) == 0) {
      if (__any_sync(kFull, lane == 0 && !lw.settle && stop_requested(cv))) break;
      full = full || __any_sync(kFull, lane == 0 && ld_relaxed_u32(&cv.ctr->full) != 0u);
    }
    Item it;
    uint4 a, b;
    load_item(base + unsigned(g0 / V), it, a, b);
    const bool valid = it.valid;
    const uint32_t a_id = it.a_id, b_id = it.b_id, op = it.op;
    uint4 c[NO];
    if constexpr (MODE == kLanesUnary) {
      const uint4 lm = s_const[2][l];
      c[0] = v_op<W>(kNot, a, a, lm, 0);
      c[1] = v_op<W>(kNext, a, a, lm, 0);
      c[2] = v_op<W>(kFuture, a, a, lm, 0);
      c[3] = v_op<W>(kGlobally, a, a, lm, 0);
    } else if constexpr (MODE == kLanesBinary) {
      c[0] = v_op<W>(kAnd, a, b, a, 0);
      c[1] = v_op<W>(kOr, a, b, a, 0);
      c[2] = v_op<W>(kUntil, a, b, a, 0);
      c[3] = v_op<W>(kUntil, b, a, a, 0);
    } else {
      c[0] = op == kAtom ? a : v_op<W>(op, a, b, s_const[2][l], 0);
    }
    auto desc_of = [&](int o) -> uint64_t {
      if constexpr (MODE == kLanesUnary) return pack_desc(unary_code(o), a_id, 0);
      else if constexpr (MODE == kLanesBinary)
        return o == 3 ? pack_desc(kUntil, b_id, a_id) : pack_desc(o == 0 ? kAnd : o == 1 ? kOr : kUntil, a_id, b_id);
      else return pack_desc(op, a_id, b_id);
    };

    // Hash and specification check: each lane its vector; the partial sums are
    // added up so that every candidate's total ends in the lane that probes it.
    uint32_t lo[NO], hi[NO], bad = 0;
    {
      const uint4 mul = s_const[0][l], lab = s_const[1][l];
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        lo[o] = hi[o] = 0;
        if (!enabled(o)) continue;
        h_acc(c[o], mul, lo[o], hi[o]);
        bad |= (label_miss<W>(c[o], lab) >> 31) << o;
      }
    }
    int m = V / 2;
    if constexpr (NO == 4) {
      if constexpr (V >= 2) {  // two of the four to each half of the group
        const bool up = (l & m) != 0;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const uint32_t sl = up ? lo[q] : lo[2 + q], sh = up ? hi[q] : hi[2 + q];
          lo[q] = (up ? lo[2 + q] : lo[q]) + __shfl_xor_sync(kFull, sl, m);
          hi[q] = (up ? hi[2 + q] : hi[q]) + __shfl_xor_sync(kFull, sh, m);
        }
        m /= 2;
      }
      if constexpr (V >= 4) {  // one of the two
        const bool up = (l & m) != 0;
        const uint32_t sl = up ? lo[0] : lo[1], sh = up ? hi[0] : hi[1];
        lo[0] = (up ? lo[1] : lo[0]) + __shfl_xor_sync(kFull, sl, m);
        hi[0] = (up ? hi[1] : hi[0]) + __shfl_xor_sync(kFull, sh, m);
        m /= 2;
      }
    }
#pragma unroll
    for (; m > 0; m /= 2) {
      lo[0] += __shfl_xor_sync(kFull, lo[0], m);
      hi[0] += __shfl_xor_sync(kFull, hi[0], m);
    }
#pragma unroll
    for (int x = V / 2; x > 0; x /= 2) bad |= __shfl_xor_sync(kFull, bad, x);

    int state[R];
    uint32_t tag[R], home[R], pos[R];  // the hash's two words; the slot being probed (tables hold at most 2^32)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int o = cand_of(l, r);
      const bool mine = valid && owner && ((ops >> o) & 1u);
      if (mine && !((bad >> o) & 1u)) record_solution(cv, desc_of(o));
      state[r] = mine && !full ? kProbing : kDone;
      const uint64_t h = h_fin(hi[r], lo[r]);
      tag[r] = uint32_t(h >> 32);
      home[r] = uint32_t(h);
      pos[r] = uint32_t(home_slot(h, cv.table_mask));
      built += unsigned(__popc(__ballot_sync(kFull, mine)));
    }
    flush();  // the previous batch's rows: a warp never meets its own earlier claims as pending

    unsigned waits = 0;
    unsigned long long guard = 0;
    while (true) {
      // A round. Read the buckets; then, in flight together: claims of empty
      // slots, ids for them, and the rows behind matching tags. A lost claim
      // reads its bucket again in the next round.
      uint32_t cmp[R], claim[R];
      int won[R];  // the claim's outcome
      unsigned n_claim = 0;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        cmp[r] = 0u;  // id + 1 of the row to compare with
        won[r] = 2;
        bool empty = false;
        if (state[r] == kProbing) {
          uint32_t id1;
          unsigned long long at = pos[r];
          const int saw = see_bucket(cv.table, cv.table_mask, at, tag[r], id1);
          pos[r] = uint32_t(at);
          if (saw == kSeeEmpty) empty = true;
          else if (saw == kSeeFull) state[r] = kDone;  // the arena is full
          else if (saw == kSeePending) state[r] = kWait;
          else if (saw == kSeeMatch) {
            state[r] = kCompare;
            cmp[r] = id1;
          }
        }
        if (empty) won[r] = claim_slot(cv.table + pos[r], tag[r]);
      }
      __syncwarp();  // the probing lanes' acquires, before every lane's row reads
      uint4 st[NO];
      uint32_t ne = 0;
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        if (!enabled(o)) continue;
        const uint32_t id = from_owner(cmp[NO == 4 && V < 4 ? o % R : 0], o);
        st[o] = id ? __ldcg(row(id - 1u) + l) : c[o];
      }
#pragma unroll
      for (int o = 0; o < NO; ++o)
        if (enabled(o)) ne |= v_ne(st[o], c[o]) ? 1u << o : 0u;
#pragma unroll
      for (int x = V / 2; x > 0; x /= 2) ne |= __shfl_xor_sync(kFull, ne, x);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (state[r] == kCompare) {
          if ((ne >> cand_of(l, r)) & 1u) {
            state[r] = kProbing;
            pos[r] = (pos[r] + 1u) & uint32_t(cv.table_mask);
          } else {
            state[r] = kDone;  // an equal CM is already cached
          }
        }
        if (won[r] < 2) state[r] = won[r] == 0 ? kClaimed : kWait;
        claim[r] = __ballot_sync(kFull, state[r] == kClaimed);
        n_claim += unsigned(__popc(claim[r]));
      }
      // claims: ids (the warp's stock, then the fresh ones), rows written by the groups
      if (n_claim) {
        const unsigned asked = ids.ask(n_claim, ahead ? min(kLanesAhead, 2u * batches) : 0u);
        unsigned fresh = 0;
        if (asked) {
          if (lane == 0) fresh = atomicAdd(&cv.ctr->n_entries, asked);
          fresh = __shfl_sync(kFull, fresh, 0);
        }
        uint32_t id1[R];  // id + 1 of a row to write
        unsigned rank0 = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const unsigned rank = rank0 + unsigned(__popc(claim[r] & ((1u << lane) - 1u)));
          const unsigned id = ids.id(rank, fresh);
          rank0 += unsigned(__popc(claim[r]));
          const bool ok = state[r] == kClaimed && id < cv.max_entries;
          id1[r] = ok ? id + 1u : 0u;
          if (state[r] == kClaimed) {
            if (ok) {
              cv.prov[id] = desc_of(cand_of(l, r));
              cv.slotpos[id] = pos[r];
              cv.homes[id] = home[r];
              pend_pos[r] = pos[r];
              pend_tag[r] = tag[r];
              pend_id[r] = id + 1u;
            } else {
              st_relaxed(cv.table + pos[r], ((unsigned long long)tag[r] << 32) | kSlotTomb);  // nothing to order: no row behind it
              atomicExch(&cv.ctr->full, 1u);
            }
            state[r] = kDone;
          }
          const unsigned written = unsigned(__popc(__ballot_sync(kFull, ok)));
          inserted += written;
          full = full || written < unsigned(__popc(claim[r]));
        }
#pragma unroll
        for (int o = 0; o < NO; ++o) {
          if (!enabled(o)) continue;
          const uint32_t id = from_owner(id1[NO == 4 && V < 4 ? o % R : 0], o);
          if (id) cv.arena[size_t(id - 1u) * V + l] = c[o];
        }
        ids.use(n_claim, asked, fresh);
      }
      bool more = false;
#pragma unroll
      for (int r = 0; r < R; ++r) more = more || state[r] == kProbing;
      const bool again = __any_sync(kFull, more);
      if (again && ++guard > cv.table_mask) {  // every slot seen: cannot happen at load <= 0.9
        if (lane == 0) atomicExch(&cv.ctr->error, 1u);
        break;
      }
      // A candidate that met a pending slot is mostly a twin of one that this
      // warp has just claimed: settled by comparing the two in registers.
#pragma unroll
      for (int r = 0; r < R; ++r)
        for (uint32_t t = __ballot_sync(kFull, state[r] == kWait); t; t &= t - 1u) {
          const int q = __ffs(t) - 1;
          const uint32_t tq = __shfl_sync(kFull, tag[r], q), hq = __shfl_sync(kFull, home[r], q);
#pragma unroll
          for (int r2 = 0; r2 < R; ++r2) {
            const uint32_t twins = __ballot_sync(kFull, tag[r2] == tq && home[r2] == hq) & claim[r2];
            if (twins == 0u) continue;
            const int tw = __ffs(twins) - 1, oq = cand_of(q & (V - 1), r), ot = cand_of(tw & (V - 1), r2);
            uint4 x = c[0], y = c[0];
#pragma unroll
            for (int o = 1; o < NO; ++o) {
              if (o == oq) x = c[o];
              if (o == ot) y = c[o];
            }
            const int src = (tw & ~(V - 1)) + l;
            y = make_uint4(__shfl_sync(kFull, y.x, src), __shfl_sync(kFull, y.y, src), __shfl_sync(kFull, y.z, src),
                           __shfl_sync(kFull, y.w, src));
            const bool ne = g0 == (q & ~(V - 1)) && v_ne(x, y) != 0u;
            if (!__any_sync(kFull, ne) && lane == q) state[r] = kDone;
          }
        }
      bool wait = false;
#pragma unroll
      for (int r = 0; r < R; ++r) wait = wait || state[r] == kWait;
      if (!__any_sync(kFull, wait)) {
        if (!again) break;
        flush();  // (rare) a lane probes on while this round's claims are pending
        continue;
      }
      if (waits++ >= kLanesWaits) {
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (state[r] == kWait) {
            defer(cv, desc_of(cand_of(l, r)));
            state[r] = kDone;
          }
        if (!again) break;
      }
      flush();  // another warp may wait for these, as this one waits for another's
      if (!again) __nanosleep(64);
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (state[r] == kWait) state[r] = kProbing;
    }
  }
  flush();
  if (lane == 0) {
    WarpDedup::log_hole(cv, ids.next, ids.end);
    if (inserted) atomicAdd(&cv.ctr->inserted_k[kKind], (unsigned long long)inserted);
    if (MODE != kLanesList && built) atomicAdd(&cv.ctr->built_k[kKind], built);
    if (MODE == kLanesList && lw.atoms && blockIdx.x == 0 && threadIdx.x == 0)
      atomicAdd(&cv.ctr->built_k[kKind], total);  // deferred candidates were counted when first built
  }
}

template <typename W, int V, int MODE, unsigned kOps>
__global__ void __launch_bounds__(256, V >= 4 ? 4 : 2) k_lanes(CacheView cv, LanesWork lw,
                                                               const __grid_constant__ BinaryPlan plan) {
  lanes_run<W, V, MODE, false, kOps>(cv, lw, plan);
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
template <typename W, int V>
struct LaunchA {
  template <int MODE, unsigned kOps>
  static cudaError_t run(const CacheView& cv, const LanesWork& lw, const BinaryPlan& plan, unsigned long long n,
                         const LaunchCfg& lc) {
    static int occ = occupancy_blocks((const void*)k_lanes<W, V, MODE, kOps>, 256, 0);
    constexpr unsigned long long per_block = 8ull * (32 / V);
    const unsigned long long want = (n + per_block - 1) / per_block;
    const unsigned blocks = unsigned(std::max(1ull, std::min(want, (unsigned long long)lc.sms * occ)));
    k_lanes<W, V, MODE, kOps><<<blocks, 256, 0, lc.stream>>>(cv, lw, plan);
    return cudaGetLastError();
  }
  static cudaError_t desc_list(const CacheView& cv, const unsigned long long* list, const unsigned int* list_n,
                               unsigned int cap, unsigned int atoms, const LaunchCfg& lc) {
    LanesWork lw{};
    lw.list = list;
    lw.list_n = list_n;
    lw.list_cap = cap;
    lw.atoms = atoms;
    lw.exact = 1;
    BinaryPlan none;
    none.n_splits = 0;
    return run<kLanesList, 15u>(cv, lw, none, list ? cap : atoms, lc);
  }
  static cudaError_t unary(const CacheView& cv, uint32_t first, uint32_t count, uint32_t ops, const LaunchCfg& lc) {
    LanesWork lw{};
    lw.total = count;
    lw.first = first;
    lw.ops = ops;
    BinaryPlan none;
    none.n_splits = 0;
    // bit 3: G
    return (ops & 8u) == 0u ? run<kLanesUnary, 7u>(cv, lw, none, count, lc)
                            : run<kLanesUnary, 15u>(cv, lw, none, count, lc);
  }
  static cudaError_t binary(const CacheView& cv, const BinaryPlan& plan, const LaunchCfg& lc) {
    LanesWork lw{};
    lw.total = plan.total_pairs;
    lw.ops = plan.ops;
    // bit 1: or
    return (plan.ops & 2u) == 0u ? run<kLanesBinary, 13u>(cv, lw, plan, plan.total_pairs, lc)
                                 : run<kLanesBinary, 15u>(cv, lw, plan, plan.total_pairs, lc);
  }
};

#define LSYN_LANES(CALL)                     \
  switch (cv.vecs) {                         \
    case 1: return LaunchA<W, 1>::CALL;      \
    case 2: return LaunchA<W, 2>::CALL;      \
    case 4: return LaunchA<W, 4>::CALL;      \
    case 8: return LaunchA<W, 8>::CALL;      \
    default: return cudaErrorInvalidValue;   \
  }

template <typename W>
cudaError_t LaneKernels<W>::desc_list(const CacheView& cv, const unsigned long long* list, const unsigned int* list_n,
                                      unsigned int cap, unsigned int atoms, const LaunchCfg& lc) {
  LSYN_LANES(desc_list(cv, list, list_n, cap, atoms, lc))
}

template <typename W>
cudaError_t LaneKernels<W>::unary(const CacheView& cv, uint32_t first, uint32_t count, uint32_t ops,
                                  const LaunchCfg& lc) {
  LSYN_LANES(unary(cv, first, count, ops, lc))
}

template <typename W>
cudaError_t LaneKernels<W>::binary(const CacheView& cv, const BinaryPlan& plan, const LaunchCfg& lc) {
  LSYN_LANES(binary(cv, plan, lc))
}

}  // namespace lsyn

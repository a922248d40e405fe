// Level kernels for characteristic matrices above 512 bytes (and for traces of
// several words): a group of warps takes one or a few operand rows or pairs at a
// time (an item), builds their candidates, four each, and settles them
// together. Included by kernels_g32.cu / kernels_g64.cu.
//
// What bounds them: streaming rows (operands, compare reads of stored rows,
// new rows) at HBM rate; below a few hundred thousand candidates, the chain of
// round trips of one candidate. Each thread holds at most kGroupVecs vectors of
// each operand, staged in shared memory (cp.async, each thread its own
// vectors, so that no barrier is needed), and every pass (hash and
// specification check, compares, writes) computes the candidates from there: an
// operand is fetched once. Wide matrices take several warps to a candidate,
// narrow ones several pairs to a warp, so that every SM has about 200 KB of
// candidates in flight whatever the width.
//
// Per item: (1) every thread hashes its columns of the candidates and checks
// the specification; (2) warp 0 adds the partial hashes up, publishes what the
// group claimed before, probes and claims table slots (one lane per candidate);
// (3) every thread
// compares its columns with the stored rows that the probes found, while warp 0
// reserves ids, then writes the claimed rows and fetches its part of the next
// item's operands. A candidate that meets a pending slot with its own tag is
// probed again a bounded number of times after the group has published its own
// claims (the other group's row is then usually there), and deferred only when
// that runs out.
//
// Measured against the kernels that walked a matrix with one warp (complete
// levels, one GB300): 10 propositions, 2048 traces (16 KiB), levels 1-7 in 8.6
// ms instead of 12.1; 3 propositions, 250 traces of up to 64 positions (2000
// bytes), levels 1-10 in 4.2 ms instead of 6.8; 200 traces of up to 200
// positions (four words each), levels 1-9 in 4.3 ms instead of 13.8. The level
// kernels of the last levels then run at 3.8-5.0 TB/s of algorithmic bytes (3.0-3.8
// with four words), bound by instructions and the latency that 24 warps an SM
// hide; levels below 10^4 candidates take 12-20 us a launch instead of 40-440.
#pragma once

#include "lsyn_device.cuh"

namespace lsyn {

enum : int { kGroupUnary = 0, kGroupBinary = 1, kGroupList = 2 };

constexpr int kGroupMaxWarps = 8;  // warps that share a candidate (a block)
// Operand vectors staged per thread, all rows of an item. 16 (8 KiB a warp) let
// three blocks of one-plane kernels share an SM; measured at 2000-byte and
// 16 KiB matrices: 12 (less in flight) took 15-30 % longer, 20 (two blocks)
// 5-7 %.
constexpr int kGroupVecs = 16;
constexpr int kGroupMaxBatch = 4;  // left rows per item
// A group hands its count of candidates in when it gets here: a level may have
// more of them than 32 bits hold for each group, above all one that goes on with
// the specification check alone in a full arena. The check costs 0.4 % of the
// kernels of 2 and 16 KiB matrices; a 64-bit count 1 %, as a register or in
// shared memory, a count in every lane 1.7 %, the check at the item's end 4 %.
constexpr unsigned kCountMost = 1u << 31;
constexpr unsigned kGroupWaits = 12;   // probes of a pending slot (a round trip and two barriers each) before deferring

// Blocks per SM that the compiler is to leave registers for: three (80
// registers) fit the one-plane kernels without spills, and four cost 15-25 % in
// spills; the carries between planes need 105-117 registers.
constexpr int group_blocks(bool several_planes) { return several_planes ? 2 : 3; }

struct GroupWork {
  unsigned long long total;            // items (a list, one descriptor an item, reads its own length)
  uint32_t count;                      // unary: rows
  uint32_t first, ops;                 // unary: first row; enabled operators (4 bits)
  const unsigned long long* list;      // list mode: descriptors, or NULL for the atoms
  const unsigned int* list_n;
  unsigned int list_cap, atoms;
  unsigned int list_from;              // list mode: first descriptor
  int settle;                          // 1: goes on after a solution (deferred candidates)
  int warps, batch;                    // warps per group, left rows per item
};

// One column, its planes visited from the last to the first (a later plane
// carries into an earlier one, see mp_op).
template <typename W, int MODE, bool MP>
struct ColumnOps {
  using V = Words<W>;
  V s0, s1, s2;  // what the planes after this one carry into it
  __device__ __forceinline__ ColumnOps() {
#pragma unroll
    for (int i = 0; i < V::N; ++i) s0.w[i] = s1.w[i] = s2.w[i] = 0;
  }
  // f(o, c): the next plane of candidate o, for every o in `sub` (of four; list
  // mode: one, of operator `op`). `sub` is the same in the whole warp, and for
  // all planes of a column.
  template <class F>
  __device__ __forceinline__ void step(uint32_t sub, uint32_t op, uint4 av, uint4 bv, uint4 lv, F&& f) {
    const V a = V::load(av);
    V r;
    if constexpr (MODE == kGroupUnary) {
      const V m = V::load(lv);
      if (sub & 1u) {
#pragma unroll
        for (int i = 0; i < V::N; ++i) r.w[i] = ~a.w[i] & m.w[i];
        f(0, r.store());
      }
      if (sub & 2u) {
#pragma unroll
        for (int i = 0; i < V::N; ++i) {
          r.w[i] = a.w[i] << 1;
          if (MP) {
            r.w[i] |= s0.w[i];
            s0.w[i] = w_top<W>(a.w[i]);
          }
        }
        f(1, r.store());
      }
      if (sub & 4u) {
#pragma unroll
        for (int i = 0; i < V::N; ++i) {
          r.w[i] = w_future<W>(a.w[i]);
          if (MP) {
            r.w[i] |= s1.w[i] ? m.w[i] : W(0);
            s1.w[i] |= a.w[i];
          }
        }
        f(2, r.store());
      }
      if (sub & 8u) {
#pragma unroll
        for (int i = 0; i < V::N; ++i) {
          const W n = ~a.w[i] & m.w[i];
          r.w[i] = w_future<W>(n);
          if (MP) {
            r.w[i] |= s2.w[i] ? m.w[i] : W(0);
            s2.w[i] |= n;
          }
          r.w[i] = ~r.w[i] & m.w[i];
        }
        f(3, r.store());
      }
    } else if constexpr (MODE == kGroupBinary) {
      const V b = V::load(bv);
      if (sub & 1u) f(0, make_uint4(av.x & bv.x, av.y & bv.y, av.z & bv.z, av.w & bv.w));
      if (sub & 2u) f(1, make_uint4(av.x | bv.x, av.y | bv.y, av.z | bv.z, av.w | bv.w));
      if (sub & 4u) {
#pragma unroll
        for (int i = 0; i < V::N; ++i) {
          r.w[i] = MP ? w_until_cin<W>(a.w[i], b.w[i], s0.w[i]) : w_until<W>(a.w[i], b.w[i]);
          if (MP) s0.w[i] = w_top<W>(r.w[i]);
        }
        f(2, r.store());
      }
      if (sub & 8u) {
#pragma unroll
        for (int i = 0; i < V::N; ++i) {
          r.w[i] = MP ? w_until_cin<W>(b.w[i], a.w[i], s1.w[i]) : w_until<W>(b.w[i], a.w[i]);
          if (MP) s1.w[i] = w_top<W>(r.w[i]);
        }
        f(3, r.store());
      }
    } else {
      const V b = V::load(bv), m = V::load(lv);
#pragma unroll
      for (int i = 0; i < V::N; ++i) {
        const W ai = a.w[i], bi = b.w[i], mi = m.w[i], x = op == kGlobally ? (~ai & mi) : ai;
        const W carry = MP ? s0.w[i] : W(0);
        W y;
        switch (op) {
          case kNot: y = ~ai & mi; break;
          case kAnd: y = ai & bi; break;
          case kOr: y = ai | bi; break;
          case kNext: y = (ai << 1) | carry; break;
          case kFuture:
          case kGlobally:
            y = w_future<W>(x) | (carry ? mi : W(0));
            if (op == kGlobally) y = ~y & mi;
            break;
          case kUntil: y = w_until_cin<W>(ai, bi, carry); break;
          default: y = ai;  // an atom
        }
        if (MP) s0.w[i] = op == kNext ? w_top<W>(ai) : op == kUntil ? w_top<W>(y) : (carry | x);
        r.w[i] = y;
      }
      f(0, r.store());
    }
  }
};

// What warp 0 tells the group's other warps, and what they tell it.
struct GroupCtl {
  uint32_t diff[kGroupMaxWarps];  // per warp: bit q set when candidate q misses a label
  uint32_t ne[kGroupMaxWarps];    // per warp: bit q set when candidate q differs from what it was compared with
  uint32_t cmp_id[4 * kGroupMaxBatch], new_id[4 * kGroupMaxBatch];  // rows to compare with, and to write to
  uint32_t twin_of[4 * kGroupMaxBatch];
  uint32_t a[2], b[2], op[2], n[2];  // this and the next item: first left row, right row, operator (list), left rows
  uint32_t cmp, claim, twin, wait, stop;
};
constexpr size_t kGroupCtlBytes = (sizeof(GroupCtl) + 15) / 16 * 16;

// A value that every lane of the warp holds, in a form that the compiler knows
// to be uniform (branches on it then need no reconvergence code).
__device__ __forceinline__ uint32_t uniform(uint32_t x) { return __reduce_or_sync(kFull, x); }

// Operand rows of an item: `batch` rows; with one right-hand row for all (binary); a descriptor's two (list).
__host__ __device__ inline int group_rows(int mode, int batch) {
  return mode == kGroupUnary ? batch : mode == kGroupBinary ? batch + 1 : 2;
}

// Shared memory of one group: partial hashes (several warps only), control
// words, the staged rows.
__host__ __device__ inline size_t group_smem(int mode, unsigned vecs, int warps, int batch) {
  return (warps > 1 ? size_t(warps) * 4 * batch * 256 : 0) + kGroupCtlBytes + size_t(group_rows(mode, batch)) * vecs * 16;
}

// The work of one launch, or of one step of a launch that builds several levels
// (operand rows are copied and compared past L1, so that rows built by the same
// launch are read as written); `mem` is the block's dynamic shared memory.
template <typename W, int MODE, bool MP>
__device__ __forceinline__ void group_run(const CacheView& cv, const GroupWork& gw, const BinaryPlan& plan,
                                          unsigned char* mem) {
  constexpr unsigned kKind = MODE == kGroupUnary ? kKindUnary : MODE == kGroupBinary ? kKindBinary : kKindOther;
  constexpr int NO = MODE == kGroupList ? 1 : 4;   // candidates per row, pair or descriptor
  constexpr int NR = MODE == kGroupUnary ? 1 : 2;  // operand rows of a candidate
  using Ops = ColumnOps<W, MODE, MP>;
  const int warps = gw.warps, T = 32 * warps, B = gw.batch;
  const int planes = MP ? int(cv.planes) : 1;
  const unsigned pv = MP ? cv.plane_vecs : cv.vecs;
  const int gi = int(threadIdx.x) / T, t = int(threadIdx.x) - gi * T, w = t >> 5, lane = t & 31;
  const int per_block = int(blockDim.x) / T;
  if (gi >= per_block) return;  // threads left over (a block of eight warps, groups of three)
  unsigned char* base = mem + size_t(gi) * group_smem(MODE, cv.vecs, warps, B);
  unsigned long long* red = reinterpret_cast<unsigned long long*>(base);  // [warps][4 B][32]
  if (warps > 1) base += size_t(warps) * 4 * B * 256;
  GroupCtl* ctl = reinterpret_cast<GroupCtl*>(base);
  uint4* buf = reinterpret_cast<uint4*>(base + kGroupCtlBytes);  // [rows][vecs]; a thread touches only its own vectors
  auto sync = [&]() {
    if (warps == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(gi + 1), "r"(T) : "memory");
  };
  auto staged = [&](int r) { return buf + unsigned(r) * cv.vecs; };
  const int other_row = MODE == kGroupList ? 1 : B;  // where the right-hand operand is staged
  auto two_rows = [](uint32_t o) {
    return MODE == kGroupBinary || (MODE == kGroupList && (o == kAnd || o == kOr || o == kUntil));
  };
  const int my_cols = int((pv - unsigned(t) + unsigned(T) - 1u) / unsigned(T));  // columns t, t + T, ... of a plane (pv >= T)

  unsigned long long total = gw.total;
  if constexpr (MODE == kGroupList) total = gw.list ? min(__ldcg(gw.list_n), gw.list_cap) - gw.list_from : gw.atoms;
  const unsigned long long stride = (unsigned long long)gridDim.x * per_block;
  unsigned long long item = (unsigned long long)blockIdx.x * per_block + gi;
  if (MODE == kGroupList && gw.atoms && blockIdx.x == 0 && threadIdx.x == 0)
    atomicAdd(&cv.ctr->built_k[kKind], total);  // deferred candidates were counted when first built

  // operands of item i, by warp 0: n consecutive rows a (left), one row b (right)
  auto map_item = [&](unsigned long long i, int x) {
    if (i >= total) return;
    uint32_t a = 0, b = 0, op = 0;
    int n = 1;
    if constexpr (MODE == kGroupUnary) {
      const uint32_t r = uint32_t(i) * uint32_t(B);
      a = gw.first + r;
      n = int(min(uint32_t(B), gw.count - r));
    } else if constexpr (MODE == kGroupBinary) {
      int sp = 0;
      while (sp + 1 < plan.n_splits && plan.s[sp + 1].tiles_begin <= i) ++sp;
      const Split& S = plan.s[sp];
      const unsigned long long l = i - S.tiles_begin;
      // lt_tiles items a right-hand row
      uint32_t r, k;
      if ((l >> 32) == 0ull) {
        r = uint32_t(l) / S.lt_tiles;
        k = uint32_t(l) - r * S.lt_tiles;
      } else {
        r = uint32_t(l / S.lt_tiles);
        k = uint32_t(l - (unsigned long long)r * S.lt_tiles);
      }
      uint32_t limit = S.left_n;  // left rows that pair with this right-hand row
      if (S.tri) {
        // pairs a < b: right-hand row n - 1 - r, then row r, share the fold's items
        const uint32_t last = S.left_n - 1u, c1 = (last - r + uint32_t(B) - 1u) / uint32_t(B);
        if (k < c1) {
          r = last - r;
        } else {
          k = r < last - r ? k - c1 : 0x40000000u / uint32_t(B);  // the middle row has no partner
        }
        limit = r;
      }
      const uint32_t a0 = k * uint32_t(B);
      n = a0 < limit ? int(min(uint32_t(B), limit - a0)) : 0;
      a = S.left_start + a0;
      b = S.right_start + r;
    } else {
      const uint64_t d = gw.list ? __ldcg(gw.list + gw.list_from + i) : pack_desc(kAtom, uint32_t(i), 0);
      a = desc_left(d);
      b = desc_right(d);
      op = desc_op(d);
    }
    if (lane == 0) {
      ctl->n[x] = uint32_t(n);
      ctl->a[x] = a;
      ctl->b[x] = b;
      ctl->op[x] = op;
    }
  };
  // this thread's vectors of the item's operands
  auto fetch = [&](int x) {
    const int n = int(ctl->n[x]);
    const uint32_t op = ctl->op[x];
    const uint4* ra = (MODE == kGroupList && op == kAtom) ? cv.atoms + size_t(ctl->a[x]) * cv.vecs : row_ptr(cv, ctl->a[x]);
    const uint4* rb = row_ptr(cv, ctl->b[x]);
    auto copy = [&](uint4* dst, const uint4* src) {
#pragma unroll 2
      for (int c = 0; c < my_cols; ++c)
        for (int j = 0; j < planes; ++j) {
          const unsigned v = unsigned(j) * pv + unsigned(t + T * c);
          cp_async16(dst + v, src + v);
        }
    };
    for (int p = 0; p < n; ++p, ra += cv.vecs) copy(staged(p), ra);
    if (n && two_rows(op)) copy(staged(other_row), rb);
  };
  // pre(v, j), then f(o, c) for every candidate o in `sub` of row, pair or
  // descriptor p: every vector v (plane j) of this thread
  auto each = [&](int p, uint32_t op, uint32_t sub, auto&& pre, auto&& f) {
    const bool two = two_rows(op);
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    const uint4 *ra = staged(p), *rb = staged(other_row);
#pragma unroll 1  // (two columns at a time spill: 5-10 % slower)
    for (int c = 0; c < my_cols; ++c) {
      Ops col;
      for (int j = planes - 1; j >= 0; --j) {
        const unsigned v = unsigned(j) * pv + unsigned(t + T * c);
        const uint4 lm = MODE != kGroupBinary ? __ldg(cv.lenmask + v) : zero;
        pre(v, j);
        col.step(sub, op, ra[v], NR == 2 && two ? rb[v] : zero, lm, f);
      }
    }
  };

  if (w == 0) {
    map_item(item, 0);
    if (lane == 0) ctl->stop = !gw.settle && stop_requested(cv) ? 1u : 0u;
  }
  sync();
  if (item >= total || ctl->stop) return;  // the same for the whole group
  fetch(0);
  int cur = 0;
  const uint32_t ops = MODE == kGroupList ? 1u : gw.ops & 0xFu;

  // warp 0's state, a lane per candidate
  constexpr int kProbing = WarpDedup::kProbing, kDone = WarpDedup::kDone, kClaimed = WarpDedup::kClaimed;
  constexpr int kCompare = 4, kWait = 5, kTwin = 6;
  WarpDedup::Pending pend;
  unsigned built = 0, inserted = 0;  // (ids fit 32 bits; candidates: see kCountMost)

  while (true) {
    const int n = int(uniform(ctl->n[cur]));
    const uint32_t op = uniform(ctl->op[cur]);
    cp_async_wait_all();
    const bool full = w == 0 && lane == 0 && ld_relaxed_u32(&cv.ctr->full) != 0u;
    // (1) hash and specification check
    uint32_t my_lo = 0, my_hi = 0, diff = 0;
    for (int p = 0; p < n; ++p) {
      unsigned long long acc[NO];
      uint32_t miss[NO];  // top bit: a position-0 bit differs from its trace's label
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        acc[o] = 0;
        miss[o] = 0;
      }
      uint4 mul, lab;
      bool first_plane = true;
      each(
          p, op, 0xFu,
          [&](unsigned v, int j) {
            mul = __ldg(cv.hmul + v);
            first_plane = !MP || j == 0;
            if (first_plane) lab = __ldg(cv.label + v);
          },
          [&](int o, uint4 c) {
            acc[o] = h_mac(c, mul, acc[o]);
            if (first_plane) miss[o] |= label_miss<W>(c, lab);
          });
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        const int q = NO * p + o;
        diff |= (miss[o] >> 31) << q;
        if (warps == 1) {
          const uint32_t lo = __reduce_add_sync(kFull, uint32_t(acc[o]));
          const uint32_t hi = __reduce_add_sync(kFull, uint32_t(acc[o] >> 32));
          if (lane == q) {
            my_lo = lo;
            my_hi = hi;
          }
        } else {
          red[(w * 4 * B + q) * 32 + lane] = acc[o];
        }
      }
    }
    diff = __reduce_or_sync(kFull, diff);
    if (lane == 0) ctl->diff[w] = diff;
    sync();

    // (2) first round: warp 0 finishes the hashes
    const int nq = NO * n;
    int state = kDone, twin = 0;
    uint64_t h = 0, my_desc = 0;
    unsigned long long pos = 0;
    unsigned waits = 0;
    unsigned long long guard = 0;
    if (w == 0) {
      if (warps > 1) {
        for (int q = 0; q < nq; ++q) {
          unsigned long long s = 0;
          for (int x = 0; x < warps; ++x) s += red[(x * 4 * B + q) * 32 + lane];
          const uint32_t lo = __reduce_add_sync(kFull, uint32_t(s)), hi = __reduce_add_sync(kFull, uint32_t(s >> 32));
          if (lane == q) {
            my_lo = lo;
            my_hi = hi;
          }
        }
        for (int x = 0; x < warps; ++x) diff |= ctl->diff[x];
      }
      const int my_p = lane < nq ? lane / NO : 0, my_o = lane & (NO - 1);
      const bool mine = lane < nq && ((ops >> my_o) & 1u);
      const uint32_t a_id = ctl->a[cur] + uint32_t(my_p), b_id = ctl->b[cur];
      if constexpr (MODE == kGroupUnary) my_desc = pack_desc(unary_code(my_o), a_id, 0);
      else if constexpr (MODE == kGroupBinary)
        my_desc = my_o == 3 ? pack_desc(kUntil, b_id, a_id)
                            : pack_desc(my_o == 0 ? kAnd : my_o == 1 ? kOr : kUntil, a_id, b_id);
      else my_desc = pack_desc(op, a_id, b_id);
      if (mine && !((diff >> lane) & 1u)) record_solution(cv, my_desc);
      const bool is_full = __any_sync(kFull, full);  // a full arena: the specification check only
      state = mine && !is_full ? kProbing : kDone;
      h = h_fin(my_hi, my_lo);
      pos = home_slot(h, cv.table_mask);
      // twins inside the item (equal hashes): compared with the lowest one from
      // their operands, without a probe of their own
      const uint32_t mine_m = __ballot_sync(kFull, mine);
      const uint32_t peers = __match_any_sync(kFull, (unsigned long long)h) & mine_m;
      if (state == kProbing && (peers & ((1u << lane) - 1u))) {
        state = kTwin;
        twin = __ffs(peers) - 1;
      }
      WarpDedup::flush(pend);  // the previous item's rows: the group never meets its own claims as pending
      built += __popc(mine_m);
      if (built >= kCountMost) {
        if (MODE != kGroupList && lane == 0) atomicAdd(&cv.ctr->built_k[kKind], (unsigned long long)built);
        built = 0;
      }
    }

    bool first = true;
    while (true) {
      unsigned fresh = 0;
      uint32_t claimed = 0;
      if (w == 0) {
        uint32_t cmp_id = 0;
        while (__any_sync(kFull, state == kProbing)) {
          if (state == kProbing) {
            uint32_t id1;
            const int saw = see_bucket(cv.table, cv.table_mask, pos, uint32_t(h >> 32), id1);
            if (saw == kSeeEmpty) {
              const int claim = claim_slot(cv.table + pos, uint32_t(h >> 32));
              if (claim < 2) state = claim == 0 ? kClaimed : kWait;
            }
            else if (saw == kSeeFull) state = kDone;  // the arena is full
            else if (saw == kSeePending) state = kWait;
            else if (saw == kSeeMatch) {
              state = kCompare;
              cmp_id = id1 - 1u;
            }
          }
          if (++guard > cv.table_mask) {  // every slot seen: cannot happen at load <= 0.9
            if (lane == 0) atomicExch(&cv.ctr->error, 1u);
            if (state == kProbing) state = kDone;
          }
        }
        claimed = __ballot_sync(kFull, state == kClaimed);
        // ids for the claims, exactly as many: a level has no holes to close
        // (8 at a time on matrices up to 2 KiB measured the same)
        if (claimed && lane == 0) fresh = atomicAdd(&cv.ctr->n_entries, unsigned(__popc(claimed)));
        const uint32_t cm = __ballot_sync(kFull, state == kCompare), tm = __ballot_sync(kFull, state == kTwin);
        const uint32_t wait = __ballot_sync(kFull, state == kWait);
        if (lane < nq) {
          ctl->cmp_id[lane] = cmp_id;
          ctl->twin_of[lane] = uint32_t(twin);
        }
        if (first) map_item(item + stride, 1 - cur);
        if (lane == 0) {
          if (first) ctl->stop = !gw.settle && stop_requested(cv) ? 1u : 0u;
          ctl->cmp = cm;
          ctl->twin = tm;
          ctl->wait = wait;
        }
      }
      sync();  // the probing lanes' acquires, before every thread's row reads
      // (3) compares, while the ids are on their way
      const uint32_t cmp = uniform(ctl->cmp), tw = uniform(ctl->twin), wait = uniform(ctl->wait);
      uint32_t ne = 0;
      for (int p = 0; p < n; ++p) {
        const uint32_t sub = (cmp >> (NO * p)) & ((1u << NO) - 1u);
        if (!sub) continue;
        const uint4* row[NO];
#pragma unroll
        for (int o = 0; o < NO; ++o) row[o] = row_ptr(cv, ctl->cmp_id[NO * p + o]);
        uint32_t d[NO];
#pragma unroll
        for (int o = 0; o < NO; ++o) d[o] = 0;
        uint4 st[NO];
        each(
            p, op, sub,
            [&](unsigned v, int) {
#pragma unroll
              for (int o = 0; o < NO; ++o)
                if ((sub >> o) & 1u) st[o] = __ldcg(row[o] + v);
            },
            [&](int o, uint4 c) { d[o] |= v_ne(st[o], c); });
#pragma unroll
        for (int o = 0; o < NO; ++o) ne |= d[o] ? 1u << (NO * p + o) : 0u;
      }
      for (uint32_t m = tw; m; m &= m - 1u) {  // (rare) candidate q against its twin, a vector at a time
        const int q = __ffs(m) - 1, z = int(ctl->twin_of[q]);
        const int qp = q / NO, zp = z / NO, qo = q & (NO - 1), zo = z & (NO - 1);
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        uint32_t d = 0;
        for (int c = 0; c < my_cols; ++c) {
          Ops cq, cz;
          for (int j = planes - 1; j >= 0; --j) {
            const unsigned v = unsigned(j) * pv + unsigned(t + T * c);
            const uint4 lm = MODE != kGroupBinary ? __ldg(cv.lenmask + v) : zero;
            const uint4 rv = NR == 2 && two_rows(op) ? staged(other_row)[v] : zero;
            uint4 x = zero, y = zero;
            cq.step(1u << qo, op, staged(qp)[v], rv, lm, [&](int, uint4 r) { x = r; });
            cz.step(1u << zo, op, staged(zp)[v], rv, lm, [&](int, uint4 r) { y = r; });
            d |= v_ne(x, y);
          }
        }
        if (d) ne |= 1u << q;
      }
      ne = __reduce_or_sync(kFull, ne);
      if (lane == 0) ctl->ne[w] = ne;
      if (w == 0) {  // ids for the claims
        uint32_t wrote = 0;
        if (claimed) {
          const unsigned id = __shfl_sync(kFull, fresh, 0) + unsigned(__popc(claimed & ((1u << lane) - 1u)));
          const bool ok = state == kClaimed && id < cv.max_entries;
          if (state == kClaimed) {
            unsigned long long* slot = cv.table + pos;
            if (ok) {
              cv.prov[id] = my_desc;
              cv.slotpos[id] = unsigned(pos);
              cv.homes[id] = uint32_t(h);
              pend.slot = slot;
              pend.val = ((h >> 32) << 32) | (unsigned long long)(id + 1u);
              ctl->new_id[lane] = id;
            } else {
              st_relaxed(slot, ((h >> 32) << 32) | kSlotTomb);  // nothing to order: no row behind it
              atomicExch(&cv.ctr->full, 1u);
            }
            state = kDone;
          }
          wrote = __ballot_sync(kFull, ok);
          inserted += __popc(wrote);
        }
        if (lane == 0) ctl->claim = wrote;
      }
      sync();
      const uint32_t claim = uniform(ctl->claim);
      for (int x = 0; x < warps; ++x) ne |= ctl->ne[x];
      for (int p = 0; p < n; ++p) {
        const uint32_t sub = (claim >> (NO * p)) & ((1u << NO) - 1u);
        if (!sub) continue;
        uint4* row[NO];
#pragma unroll
        for (int o = 0; o < NO; ++o)
          row[o] = (sub >> o) & 1u ? cv.arena + size_t(ctl->new_id[NO * p + o]) * cv.vecs : nullptr;
        unsigned at = 0;
        each(p, op, sub, [&](unsigned v, int) { at = v; }, [&](int o, uint4 c) { row[o][at] = c; });
      }
      first = false;
      if (!((ne & (cmp | tw)) | wait)) break;
      sync();  // every warp's rows, before warp 0 publishes them
      // a compare that failed probes on; a pending slot is probed again
      if (w == 0) {
        if (state == kCompare) {
          state = (ne >> lane) & 1u ? kProbing : kDone;
          pos = (pos + 1) & cv.table_mask;
        } else if (state == kTwin) {
          state = (ne >> lane) & 1u ? kProbing : kDone;
        }
        WarpDedup::flush(pend);  // another group may wait for these, as this one waits for another's
        if (wait) {
          if (waits++ < kGroupWaits) {
            __nanosleep(64);
            if (state == kWait) state = kProbing;
          } else if (state == kWait) {
            defer(cv, my_desc);
            state = kDone;
          }
        }
      }
    }
    if (ctl->stop || item + stride >= total) break;
    cur = 1 - cur;
    item += stride;
    fetch(cur);
  }
  if (warps > 1) sync();  // every warp's rows of the last item, before warp 0 publishes them
  if (w == 0) {
    WarpDedup::flush(pend);
    if (lane == 0) {
      if (inserted) atomicAdd(&cv.ctr->inserted_k[kKind], (unsigned long long)inserted);
      if (MODE != kGroupList && built) atomicAdd(&cv.ctr->built_k[kKind], (unsigned long long)built);
    }
  }
}

template <typename W, int MODE, bool MP>
__global__ void __launch_bounds__(256, group_blocks(MP)) k_group(CacheView cv, GroupWork gw,
                                                                 const __grid_constant__ BinaryPlan plan) {
  extern __shared__ __align__(128) unsigned char group_mem[];
  group_run<W, MODE, MP>(cv, gw, plan, group_mem);
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
// resident: warps of the launch that are resident together
__host__ __device__ inline void group_shape(const CacheView& cv, int mode, unsigned long long work, unsigned resident,
                                            GroupWork* gw) {
  const int planes = cv.planes <= 1 ? 1 : int(cv.planes);
  const int n = int((planes == 1 ? cv.vecs : cv.plane_vecs) / 32u);  // columns, in warps
  // groups of w warps resident together (a block holds eight warps)
  auto groups = [&](int w) {
    return (unsigned long long)(resident / unsigned(kGroupMaxWarps)) * (unsigned(kGroupMaxWarps) / unsigned(w));
  };
  // The largest item that one warp holds with kGroupVecs vectors a thread and
  // that leaves every group a few; wider matrices take one row or pair an item
  // and as few warps as hold it (past eight warps, more vectors a thread).
  // Several warps cost barriers: at 16 KiB, items of four pairs over eight
  // warps took 5.7 ms where one pair over four warps takes 4.6 (level 7 of ten
  // propositions).
  int batch = mode == kGroupList ? 1 : kGroupMaxBatch;
  while (batch > 1 && (n * planes * group_rows(mode, batch) > kGroupVecs || work < groups(1) * batch * 4)) --batch;
  const int full = (n * planes * group_rows(mode, batch) + kGroupVecs - 1) / kGroupVecs;
  int warps = n < full ? n : full;
  warps = warps < 1 ? 1 : warps > kGroupMaxWarps ? kGroupMaxWarps : warps;
  // A launch with too little work to fill half of the GPU's groups: more warps
  // to a candidate, since the chain of one candidate is then what counts.
  while (batch == 1 && warps * 2 <= kGroupMaxWarps && warps * 2 <= n && work * 2 < groups(warps)) warps *= 2;
  gw->warps = warps;
  gw->batch = batch;
}

// Cuts the splits into items: `batch` rows of the smaller level with one row of
// the larger; a level with itself in folds of two right-hand rows (n - 1 - r and
// r) whose items together number the same for every r, or one less.
__host__ __device__ inline unsigned long long group_items(BinaryPlan* plan, unsigned batch) {
  unsigned long long total = 0;
  for (int i = 0; i < plan->n_splits; ++i) {
    Split& S = plan->s[i];
    const unsigned rows = S.tri ? S.left_n - 1u : S.left_n;
    S.lt_tiles = (rows + batch - 1u) / batch + (S.tri ? 1u : 0u);
    S.rt_tiles = S.tri ? S.left_n / 2u + (S.left_n & 1u) : S.right_n;
    S.tiles_begin = total;
    total += (unsigned long long)S.lt_tiles * S.rt_tiles;
  }
  plan->total_tiles = total;
  return total;
}

inline unsigned group_resident(const CacheView& cv, const LaunchCfg& lc) {
  return unsigned(lc.sms) * unsigned(group_blocks(cv.planes > 1)) * unsigned(kGroupMaxWarps);
}

template <typename W, int MODE, bool MP>
cudaError_t group_launch(const CacheView& cv, const GroupWork& gw, const BinaryPlan& plan, unsigned long long items,
                         const LaunchCfg& lc) {
  const int per_block = kGroupMaxWarps / gw.warps, threads = per_block * gw.warps * 32;
  const size_t smem = group_smem(MODE, cv.vecs, gw.warps, gw.batch) * size_t(per_block);
  const void* fn = (const void*)k_group<W, MODE, MP>;
  static const int optin = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
      v = 0;
    return v;
  }();
  static const cudaError_t attr = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (attr != cudaSuccess) return attr;
  const int occ = occupancy_blocks(fn, threads, smem);
  const unsigned long long want = (items + per_block - 1) / per_block;
  const unsigned blocks = unsigned(std::max(1ull, std::min(want, (unsigned long long)lc.sms * occ)));
  k_group<W, MODE, MP><<<blocks, threads, smem, lc.stream>>>(cv, gw, plan);
  return cudaGetLastError();
}

template <typename W, int MODE>
cudaError_t group_dispatch(const CacheView& cv, const GroupWork& gw, const BinaryPlan& plan, unsigned long long items,
                           const LaunchCfg& lc) {
  return cv.planes > 1 ? group_launch<W, MODE, true>(cv, gw, plan, items, lc)
                       : group_launch<W, MODE, false>(cv, gw, plan, items, lc);
}

template <typename W>
cudaError_t GroupKernels<W>::unary(const CacheView& cv, uint32_t first, uint32_t count, uint32_t ops,
                                   const LaunchCfg& lc) {
  GroupWork gw{};
  group_shape(cv, kGroupUnary, count, group_resident(cv, lc), &gw);
  gw.first = first;
  gw.count = count;
  gw.ops = ops;
  gw.total = (count + unsigned(gw.batch) - 1u) / unsigned(gw.batch);
  BinaryPlan none;
  none.n_splits = 0;
  return group_dispatch<W, kGroupUnary>(cv, gw, none, gw.total, lc);
}

template <typename W>
cudaError_t GroupKernels<W>::binary(const CacheView& cv, const BinaryPlan& plan, const LaunchCfg& lc) {
  GroupWork gw{};
  group_shape(cv, kGroupBinary, plan.total_pairs, group_resident(cv, lc), &gw);
  gw.ops = plan.ops;
  BinaryPlan items = plan;
  gw.total = group_items(&items, unsigned(gw.batch));
  return group_dispatch<W, kGroupBinary>(cv, gw, items, gw.total, lc);
}

template <typename W>
cudaError_t GroupKernels<W>::desc_list(const CacheView& cv, const unsigned long long* list, const unsigned int* list_n,
                                       unsigned int cap, unsigned int atoms, const LaunchCfg& lc) {
  GroupWork gw{};
  const unsigned n = list ? cap : atoms;
  group_shape(cv, kGroupList, n, group_resident(cv, lc), &gw);
  gw.list = list;
  gw.list_n = list_n;
  gw.list_cap = cap;
  gw.atoms = atoms;
  BinaryPlan none;
  none.n_splits = 0;
  return group_dispatch<W, kGroupList>(cv, gw, none, n, lc);
}

}  // namespace lsyn

// Ids that a warp of a path-A level has reserved from the cache's counter and
// not used yet. Plain C++ as well, so that the bookkeeping can be run on a CPU.
#pragma once

#ifdef __CUDACC__
#define LSYN_HD __host__ __device__ __forceinline__
#else
#define LSYN_HD inline
#endif

namespace lsyn {

// Ids that a warp of a large path-A level reserves beyond its need.
constexpr unsigned kLanesAhead = 64;

// One range, [next, end). A warp asks for ids once it knows how many claims it
// has won, so the range it had is used up before it gets another: what it leaves
// over is one range of at most kLanesAhead ids, whatever number of claims are
// lost. (Asking by the empty slots that it met, before the claims, saves the
// round trip, but when other claims take enough of them the old range is not
// used up, and one of the two becomes a hole: such holes grew with the level, 4-5
// of every 1000 ids of 32-byte matrices.)
struct IdStock {
  unsigned next = 0, end = 0;
  LSYN_HD unsigned have() const { return end - next; }
  // How many ids to reserve for n claims: those that are missing, and, if any
  // is, `ahead` more.
  LSYN_HD unsigned ask(unsigned n, unsigned ahead) const { return n > have() ? n - have() + ahead : 0u; }
  // The id of claim `rank` (below n), if ids from `fresh` on were reserved.
  LSYN_HD unsigned id(unsigned rank, unsigned fresh) const {
    return rank < have() ? next + rank : fresh + (rank - have());
  }
  // After n claims took their ids, `asked` of them reserved at `fresh`.
  LSYN_HD void use(unsigned n, unsigned asked, unsigned fresh) {
    const unsigned had = have();
    next = asked ? fresh + (n - had) : next + n;
    end = asked ? fresh + asked : end;
  }
};

// What the warps of a path-A level can leave over at most, for a device of
// `sms`: two launches (unary and binary) of up to 64 warps an SM, a range each.
LSYN_HD unsigned lanes_ranges(int sms) { return unsigned(sms) * 64u * 2u; }
LSYN_HD unsigned long long lanes_left_over(int sms) { return (unsigned long long)lanes_ranges(sms) * kLanesAhead; }

}  // namespace lsyn

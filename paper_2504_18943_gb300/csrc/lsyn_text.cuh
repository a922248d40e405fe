// The formula text of a cache entry, walked from its provenance on the device.
#pragma once

#include "lsyn_internal.h"

namespace lsyn {

// Formula text of descriptor `root` from the provenance records (read past L1:
// the same launch may have written them).
static __device__ void reconstruct_text(const unsigned long long* prov, unsigned long long root, char* buf, unsigned cap,
                                        int* status) {
  const char kOp[8] = {'p', '!', '&', '|', 'X', 'F', 'G', 'U'};
  struct Frame {
    unsigned long long d;
    int stage;
  };
  Frame st[80];
  int sp = 0;
  unsigned n = 0;
  int bad = 0;
  st[sp++] = {root, 0};
  auto put = [&](char ch) {
    if (n + 1 < cap) buf[n++] = ch;
    else bad = 1;
  };
  while (sp > 0 && !bad) {
    Frame& f = st[sp - 1];
    const unsigned op = desc_op(f.d);
    if (op == kAtom) {
      put('p');
      char tmp[12];
      int m = 0;
      unsigned v = desc_left(f.d);
      do { tmp[m++] = char('0' + v % 10); v /= 10; } while (v);
      while (m) put(tmp[--m]);
      --sp;
      continue;
    }
    const bool bin = op == kAnd || op == kOr || op == kUntil;
    if (f.stage == 0) {
      put('(');
      put(kOp[op & 7]);
      put(' ');
      f.stage = 1;
      if (sp >= 80) { bad = 2; break; }
      st[sp++] = {__ldcg(prov + desc_left(f.d)), 0};
    } else if (f.stage == 1 && bin) {
      put(' ');
      f.stage = 2;
      if (sp >= 80) { bad = 2; break; }
      st[sp++] = {__ldcg(prov + desc_right(f.d)), 0};
    } else {
      put(')');
      --sp;
    }
  }
  buf[n < cap ? n : cap - 1] = '\0';
  *status = bad;
}

}  // namespace lsyn

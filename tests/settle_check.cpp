// Host check of settle_moves (run by test_settle_moves.py): the settled list
// leaves every slot as the ordered list does, none of its writes reads what
// another one writes, and no slot is written twice.
#include <cstdio>
#include <cstdlib>
#include <set>
#include <vector>

#include "../paper_2001_08250_gb300/csrc/tpir_internal.h"

using namespace tpir;

static uint64_t rng_state = 1;
static uint64_t rnd() {
  rng_state += 0x9E3779B97F4A7C15ull;
  uint64_t x = rng_state;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

static int check(const std::vector<MoveOp>& ops, uint64_t slots) {
  std::vector<uint64_t> a(slots), b(slots);
  for (uint64_t i = 0; i < slots; ++i) a[i] = b[i] = 1000000 + i;
  uint64_t tmp = 0;
  for (const MoveOp& op : ops) {
    const uint64_t v = op.kind == 2 ? 0 : op.kind == 1 ? 1 + op.src : op.src == kTmpSlot ? tmp : a[op.src];
    (op.dst == kTmpSlot ? tmp : a[op.dst]) = v;
  }
  uint32_t nsave = 0;
  const std::vector<MoveOp> s = settle_moves(ops, &nsave);
  std::vector<uint64_t> saved(nsave);
  for (uint32_t i = 0; i < nsave; ++i) {
    if (s[i].kind != 4 || s[i].dst >= nsave) return 1;
    saved[s[i].dst] = b[s[i].src];
  }
  std::set<uint64_t> written;
  for (size_t i = nsave; i < s.size(); ++i)
    if (s[i].kind == 4 || s[i].dst >= slots || !written.insert(s[i].dst).second) return 2;
  for (size_t i = nsave; i < s.size(); ++i) {
    const MoveOp& op = s[i];
    if (op.kind == 0 && (op.src >= slots || written.count(op.src))) return 3;
    b[op.dst] = op.kind == 2 ? 0 : op.kind == 1 ? 1 + op.src : op.kind == 3 ? saved.at(op.src) : b[op.src];
  }
  return a == b ? 0 : 4;
}

int main() {
  // arbitrary lists
  for (int t = 0; t < 20000; ++t) {
    const uint64_t slots = 1 + rnd() % 12;
    std::vector<MoveOp> ops;
    bool tmp = false;
    for (uint64_t i = rnd() % 30; i > 0; --i) {
      MoveOp op{rnd() % slots, rnd() % slots, static_cast<uint32_t>(rnd() % 3), 0u};
      if (rnd() % 8 == 0 && op.kind == 0) {
        op.dst = kTmpSlot;
        tmp = true;
      } else if (tmp && rnd() % 4 == 0 && op.kind == 0) {
        op.src = kTmpSlot;
      }
      ops.push_back(op);
    }
    if (int rc = check(ops, slots)) return std::printf("arbitrary list %d: %d\n", t, rc), 1;
  }
  // the lists of cuckoo inserts: evictions, collection, walks that fail
  for (int t = 0; t < 200; ++t) {
    const uint64_t n = 4 + rnd() % 20;
    const uint32_t d = 1 + rnd() % 4;
    CuckooMeta m(n, d);
    m.set_policy(t % 3 ? 0 : n * d * 3 / 4, 30, t);
    for (int batch = 0; batch < 4; ++batch) {
      std::vector<MoveOp> ops;
      uint32_t ev = 0;
      for (uint64_t i = 0; i < n * d / 2; ++i) m.insert(rnd() % n, rnd() % n, i, ops, &ev);
      if (int rc = check(ops, n * d)) return std::printf("inserts %d: %d\n", t, rc), 1;
    }
  }
  std::puts("ok");
  return 0;
}

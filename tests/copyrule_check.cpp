// Host check of the rule by which smaller batches earn the transposed copy (run by
// test_copyrule.py): sequences of batches, loads and small writes against the same on
// the register-tiled kernel alone.
#include <cmath>
#include <cstdint>
#include <cstdio>

#include "../paper_2001_08250_gb300/csrc/copyrule.h"

using tpir::CopyRule;

namespace {
uint64_t state = 1;
uint64_t rnd() {
  state += 0x9E3779B97F4A7C15ull;
  uint64_t x = state;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

// A table: time beyond (or, negative, below) the register-tiled kernel's.
struct Table {
  CopyRule rule;
  double build, alloc;
  bool valid = false, allocated = false;
  double more = 0, missed = 0;  // savings of batches that ran without the copy
  int with = 0;                 // batches that ran with it

  Table(double b, double a) : build(b), alloc(a) {}
  void read(double save) {
    if (!valid && rule.make(save, build, allocated ? 0 : alloc)) {
      more += build + (allocated ? 0 : alloc);
      valid = allocated = true;
      rule.built(build);
    }
    rule.read(save);
    if (valid) {
      more -= save;
      ++with;
    } else {
      missed += save;
    }
  }
  void load() {
    rule.changed(build);
    valid = false;
  }
  void write(double update) {
    if (rule.wrote(update, build))
      load();
    else if (valid)
      more += update;
  }
};
int fail(const char* what, double a, double b) {
  std::printf("%s: %g against %g\n", what, a, b);
  return 1;
}
}  // namespace

int main() {
  // cycles of a load and k batches: at most one cost is lost, and where k batches save
  // two builds, all but the first cycles read with the copy throughout (two until the
  // allocation has been missed; then a build may come with a cycle's last batch, and an
  // eighth of the other is back with each cycle)
  const double saves[] = {1, 6, 12, 36, 70, 200};
  for (double save : saves)
    for (int k = 1; k <= 16; ++k) {
      Table t(63, 113);
      for (int c = 0; c < 200; ++c) {
        t.load();
        for (int i = 0; i < k; ++i) t.read(save);
        if (t.more > 63 + 113) return fail("cycles", t.more, 63 + 113);
      }
      if (k * save >= 2 * 63 && t.with < 184 * k) return fail("gain of cycles", t.with, 184 * k);
      if (k * save < 63 && t.with) return fail("no copy that does not pay", t.with, 0);
    }
  // one long life
  {
    Table t(63, 113);
    for (int i = 0; i < 1000; ++i) t.read(36);
    if (t.with < 990) return fail("a life", t.with, 990);
  }
  // many small writes to each batch, few, and writes only
  for (int w : {1, 3, 30}) {
    Table t(63, 113);
    for (int i = 0; i < 2000; ++i) {
      if (i < 1000) t.read(12);
      for (int j = 0; j < w; ++j) t.write(6);
      if (t.more > 63 + 113 + t.missed / 8) return fail("small writes", t.more, t.missed);
    }
    if (w == 1 && t.with < 900) return fail("gain beside writes", t.with, 900);
  }
  // anything: never more than one cost and an eighth of what was missed
  for (int s = 0; s < 20000; ++s) {
    const double build = 1 + rnd() % 200, alloc = rnd() % 2 ? 100 + rnd() % 100 : 0;
    const double scale = 1 + rnd() % 300, update = 1 + rnd() % 10;
    const uint64_t loads = 1 + rnd() % 30, writes = rnd() % 60;
    Table t(build, alloc);
    for (int i = 0; i < 300; ++i) {
      const uint64_t r = rnd() % 100;
      if (r < loads)
        t.load();
      else if (r < loads + writes)
        t.write(update);
      else
        t.read(static_cast<double>(rnd() % 1000) / 1000 * scale);
      if (t.more > build + alloc + t.missed / 8 + 1e-6) return fail("any sequence", t.more, build + alloc + t.missed / 8);
    }
  }
  std::printf("ok\n");
  return 0;
}

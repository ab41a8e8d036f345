// When a table that only smaller batches read is worth its transposed copy.
//
// The tensor-core kernel reads the batches of tensor_mid size faster than the
// register-tiled one, but only from the copy, which costs a build (two passes over
// the table; the first time its allocation too), loses its worth with the next load
// or large batch of writes, and makes every small write update it.  So the time
// that the batches since the last such change would have saved is added up, and the
// copy is made
//   - at once where this batch alone saves its cost;
//   - else when the batches since the change would have saved it, or those between
//     the two changes before did (tables are loaded and read in cycles).
// Its allocation has to have been missed as well, over all such changes.
// What builds cost and saved is kept in an account; while that is negative no copy
// is made on a guess.  Small writes drop the copy rather than update it once their
// updates since the last batch have cost another build, or where the account would
// fall below minus a build.  A sequence of reads, loads and writes thus takes at most
// an allocation and a build more than on the register-tiled kernel alone, whatever the
// sequence (and an eighth of what copies would have saved meanwhile, by which a
// negative account recovers).  All times in microseconds.
#pragma once

#include <algorithm>

namespace tpir {

struct CopyRule {
  double owed = 0;     // saved, or to be saved, by the batches since the last change
  double last = 0;     // the same between the two changes before
  double net = 0;      // what the copy made since then has saved, less its cost
  double idle = 0;     // updates of the copy since the last batch that read it
  double account = 0;  // what copies have saved less their builds, at most a build
  double missed = 0;   // what copies would have saved, beyond their builds, where there were none
  bool made = false;

  // A batch that would save `save` comes: is the copy made first, for a build and (0:
  // it has its memory) an allocation?
  bool make(double save, double build, double alloc) const {
    if (save >= build + alloc) return true;
    return account >= 0 && std::max(owed + save, last) >= build + std::max(0.0, alloc - missed);
  }
  void built(double build) {
    made = true;
    net = -build;
    idle = 0;
  }
  void read(double save) {
    save = std::max(save, 0.0);
    owed += save;
    if (made) net += save;
    idle = 0;
  }
  // A small write, which takes `update` more with the copy; true: drop the copy instead.
  bool wrote(double update, double build) {
    owed = std::max(0.0, owed - update);
    if (!made) return false;
    idle += update;
    if (idle > build || account + net - update < -build) return true;
    net -= update;
    return false;
  }
  // The table's content has changed (or the copy was dropped).
  void changed(double build) {
    if (made) {
      account = std::min(build, account + net);
    } else {
      const double gone = std::max(0.0, owed - build);
      missed += gone;
      if (account < 0) account = std::min(0.0, account + gone / 8);
    }
    last = owed;
    owed = net = idle = 0;
    made = false;
  }
};

// Costs, measured: building the copy (15 us for 32 MiB, 61 for 128, 485 for 1 GiB),
// its allocation (95 us for 4 MiB, 150 for 128, 165 for 1 GiB), its update after a
// small write (a launch).
inline double copy_build_us(double bytes) { return 2.0 + 0.48 * bytes / (1 << 20); }
inline double copy_alloc_us(double bytes) { return 100.0 + 0.1 * bytes / (1 << 20); }
constexpr double kCopyUpdateUs = 6.0;

}  // namespace tpir

// State of wide elimination (rips_wide.cuh), and its sizes for the launch code.
#pragma once
#include "rips_internal.cuh"

namespace rips {

enum { L_FRONT = 0, L_MID = 1, L_FAR = 2 };  // L_FAR: beyond the mid list, in the table only

struct WideList {
  unsigned long long off, cap;  // arena entries [off, off + cap)
};

constexpr int WIDE_SPARES = 4;

// what a team's threads count during one section (between two team barriers)
struct WideCount {
  unsigned add[2];  // rows appended to each list
  unsigned fresh;   // rows entered into the table, and
  unsigned ents;    // entries added (one 64-bit count)
  unsigned count;   // rows with an owner among those that join the front (or rows of a stored run), and
  unsigned settled; // owned rows that the round before last settled (one 64-bit count)
  unsigned todo;    // rows put on the work list
  unsigned nlong;   // stored runs left to the whole team
  unsigned stop;    // 1: out of time, 2: give way to a larger team
  unsigned long long un, ow;   // oldest live row without and with an owner
  unsigned long long longsum;  // entries of the runs offered to the team
  unsigned long long longroom; // and of those it takes
  unsigned long long tmp;      // arena offset handed out by the leader
};

// Sections rotate through three sets of counters: the one in use, the one read
// at the last barrier and the one the leader clears for the next section.
struct WideShared {
  WideCount c[3];
  unsigned bar_count, bar_gen;
};

// state of a column's reduction, the same in every block of its team
struct WideState {
  uint32_t j, cl, step, dil;
  float pace, each;      // owned rows settled a round, entries an added column
  uint64_t lo, hi;       // oldest live owned row of the last check but one, and of the last
  int ph, tcur;
  uint32_t n[2];
  int cur[2];
  WideList list[2][2];
  WideList tab[2];
  WideList todo, lng;
  WideList spare[WIDE_SPARES];  // buffers outgrown by their list or table
  uint64_t tmask, used;
  uint64_t bound, mbound;
  unsigned long long t0;
  WideCount d;  // the last section's counts
};

struct WideCtx {
  WideState st;
  WideShared sh;
};

constexpr int WIDE_MAX_BLOCKS = 1280;  // blocks of a reduction (three lists of them fit the control block)

}  // namespace rips

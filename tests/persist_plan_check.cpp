// Checks of the persistent solvers' plan (persist_plan.hpp), compiled and run by
// test_persist_plan_cpu.py: every entry that a kernel reads lies in the part of
// its shared memory that the plan gave it, also for a system without rows.
#include <cstdio>
#include <cstring>

#include "persist_plan.hpp"

static int failures = 0;
#define CHECK(c)                                              \
  do {                                                        \
    if (!(c)) {                                               \
      std::printf("FAILED line %d: %s\n", __LINE__, #c);      \
      ++failures;                                             \
    }                                                         \
  } while (0)

// The parts in order, none overlapping the next, all inside `room`.
static void check_layout(const helm::PLayout& L, size_t bytes, size_t elem, size_t room) {
  const size_t entries = static_cast<size_t>(L.rounds) * L.warps;
  CHECK(bytes <= room);
  if (L.tab) {
    CHECK(static_cast<size_t>(L.tlen_at) >= entries * helm::kRoundTabBytes);
    CHECK(static_cast<size_t>(L.xchg_at) >= L.tlen_at + entries * 32 * sizeof(int32_t));
  }
  CHECK(static_cast<size_t>(L.own_at) >= L.xchg_at + static_cast<size_t>(L.split - 1) * L.warps * 32 * 16);
  CHECK(static_cast<size_t>(L.own_len) == entries * 32);
  CHECK(bytes >= L.own_at + static_cast<size_t>(L.nown) * L.own_len * elem);
  CHECK(L.tlen_at % 16 == 0 && L.xchg_at % 16 == 0 && L.own_at % 16 == 0);
}

// No rows: one round all the same, whose entry (no slice) a split kernel reads
// before anything else.
static void empty_system() {
  for (int split : {1, 3})
    for (int owners : {32, 128}) {
      helm::PLayout L;
      size_t bytes = 0;
      std::memset(&L, 0, sizeof(L));
      CHECK(helm::persist_plan(0, 1, owners, split, 7, 16, 200000, &L, &bytes));
      CHECK(L.rounds >= 1 && L.tab);
      check_layout(L, bytes, 16, 200000);
    }
}

// Two blocks of 16 warps on each of 152 SMs, some 113 kB each: a plan for every
// number of rounds, with the table while it fits; a split kernel never goes without.
static void many_rounds() {
  const int grid = 304, owners = 512;
  const size_t room = 113000;
  int last_tab = 0;
  for (int rounds = 1; rounds <= 400; ++rounds)
    for (int extra : {-31, 0}) {
      const int32_t n = rounds * grid * owners + extra;
      helm::PLayout L;
      size_t bytes = 0;
      std::memset(&L, 0, sizeof(L));
      CHECK(helm::persist_plan(n, grid, owners, 1, 7, 16, room, &L, &bytes));
      CHECK(L.rounds == rounds);
      check_layout(L, bytes, 16, room);
      if (L.tab) {
        CHECK(last_tab >= rounds - 1);
        last_tab = rounds;
      }
    }
  CHECK(last_tab == 44);
  helm::PLayout L;
  size_t bytes = 0;
  CHECK(!helm::persist_plan(100 * grid * 128, grid, 128, 3, 7, 16, 20000, &L, &bytes));
}

// Unless neighbouring rows have neighbouring columns, the blocks of an SM leave more
// than half of its 256 kB to L1, whatever the system (GB300: 228 kB of shared memory
// per SM, 227 kB a block, 1 kB reserved).
static void leaves_l1() {
  for (bool near : {false, true})
    for (int bps : {1, 2})
      for (int owners : {32, 384, 512, 672, 768}) {
        const size_t room = helm::persist_room(233472, 232448, 1024, 3000, bps, near);
        for (int32_t n = 1000; n < 100000000; n += n / 7) {
          helm::PLayout L;
          size_t bytes = 0;
          std::memset(&L, 0, sizeof(L));
          CHECK(helm::persist_plan(n, 152 * bps, owners, 1, 9, 16, room, &L, &bytes));
          check_layout(L, bytes, 16, room);
          CHECK((bytes + 3000 + 1024) * bps <= (near && bps == 1 ? 228 : 128) * 1024);
          CHECK(bytes + 3000 <= 232448);
        }
      }
  CHECK(helm::persist_room(233472, 232448, 1024, 200000, 2, false) == 0);
}

// By default a step of a persistent kernel stays well inside a wait's 2 s: the longest
// row that it takes, in each of a warp's rounds, with 4 us an entry to spare; and the
// deeper pipeline of the graph gets the long rows where the kernel's own is shallower.
static void long_rows() {
  for (int rounds = 1; rounds <= 7; ++rounds) CHECK(helm::persist_max_row(false, false, rounds) * rounds * 4e-6 <= 1.1);
  CHECK(helm::persist_max_row(false, false, 7) > helm::persist_max_row(true, false, 7));
  CHECK(helm::persist_max_row(true, false, 7) > helm::persist_max_row(false, true, 7));
  CHECK(helm::persist_max_row(false, true, 7) >= 64);  // meshes of second order stay on it
}

int main(int argc, char** argv) {
  const char* what = argc > 1 ? argv[1] : "";
  if (!std::strcmp(what, "empty")) empty_system();
  else if (!std::strcmp(what, "rounds")) many_rounds();
  else if (!std::strcmp(what, "l1")) leaves_l1();
  else if (!std::strcmp(what, "long")) long_rows();
  else if (!std::strcmp(what, "wait")) CHECK(helm::kBarrierPolls * 0.2277e-6 >= 2.0);
  else ++failures;
  if (failures == 0) std::printf("ok\n");
  return failures == 0 ? 0 : 1;
}

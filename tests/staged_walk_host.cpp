// The way of staged warps through a size bin (csrc/staged_walk.h) on the host: warps are threads, copies and
// their analysis are book-keeping, and waits for copies give up where a seed says so.  Prints what went
// wrong; exit code 1.
//   staged_walk_host COUNT CHUNK WARPS SHARE_DECIDED SHARE_STAGEABLE GIVE_UP STAGES SEED
#include "../paper_2406_05221_b200/csrc/staged_walk.h"

#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <thread>
#include <vector>

static std::atomic<int> wrong{0};
#define EXPECT(what)                                   \
  do {                                                 \
    if (!(what)) {                                     \
      std::printf("line %d: %s\n", __LINE__, #what);   \
      wrong = 1;                                       \
    }                                                  \
  } while (0)

struct Bin {
  unsigned count;
  std::atomic<unsigned> next{0}, marked{0}, tries{0}, undecided{0};
  std::vector<int> results, marks;  // by entry: results written in the first launch, marks for the second
  std::vector<char> decidable, stageable;
};

struct Warp {
  Bin &b;
  unsigned chunk;
  double give_up;
  std::mt19937 rng;
  unsigned asked = 0, half[2] = {0, 0}, current = 0, under_way = 0, kept[kLeftMost];
  bool busy = false, arrived = false, gave_up = false, waited_again = false, reported = false;

  unsigned pull(unsigned n) { return b.next.fetch_add(n); }
  void ask(unsigned n) { asked = pull(n); }
  unsigned answer() { return asked; }
  void look_up(unsigned first, int h) { half[h] = first; }
  void take(int h, int c) { current = half[h] + c; }
  bool start_copies(int h, int c) {
    EXPECT(!busy && !gave_up);  // (the stage is free, and never used again after a wait that gave up)
    const unsigned entry = half[h] + c;
    EXPECT(entry < b.count);
    arrived = false;
    if (!b.stageable[entry]) return false;
    busy = true, under_way = entry;
    return true;
  }
  bool wait() {
    EXPECT(busy);
    if (gave_up) waited_again = true;
    if (gave_up || std::uniform_real_distribution<>(0, 1)(rng) < give_up) {
      gave_up = true;
      return false;
    }
    busy = false, arrived = true;
    return true;
  }
  template <class Next>
  bool head(Next next) {
    EXPECT(arrived && !busy && under_way == current);
    arrived = false;
    next();
    if (b.decidable[current]) b.results[current] += 1;
    return b.decidable[current];
  }
  void first_try(bool decided) { b.tries += 1, b.undecided += !decided; }
  bool most_undecided() { return b.tries >= 32 && 4 * b.undecided >= 3 * b.tries; }
  void keep(int k, unsigned entry) { kept[k] = entry; }
  void mark(unsigned first, unsigned n) {
    EXPECT(n <= 32 && first + n <= b.count);
    for (unsigned k = 0; k < n; ++k) b.marks[first + k] += 1;
  }
  void mark_kept(int k) { mark(kept[k], 1); }
  void full_pass(int k) {
    EXPECT(!busy);  // (it works in the stage)
    b.results[kept[k]] += 1;
  }
  void marked(unsigned n) {
    EXPECT(!reported);
    reported = true, b.marked += n;
  }
};

int main(int argc, char **argv) {
  if (argc != 9) return 2;
  Bin b;
  b.count = (unsigned)std::atoi(argv[1]);
  const unsigned chunk = (unsigned)std::atoi(argv[2]), warps = (unsigned)std::atoi(argv[3]);
  const double decided = std::atof(argv[4]), stageable = std::atof(argv[5]), give_up = std::atof(argv[6]);
  const bool stages = std::atoi(argv[7]) != 0;
  std::mt19937 rng((unsigned)std::atoi(argv[8]));
  std::uniform_real_distribution<> unit(0, 1);
  b.results.assign(b.count, 0), b.marks.assign(b.count, 0);
  for (unsigned k = 0; k < b.count; ++k) b.decidable.push_back(unit(rng) < decided), b.stageable.push_back(unit(rng) < stageable);
  std::vector<Warp> ws;
  ws.reserve(warps);
  for (unsigned k = 0; k < warps; ++k) ws.push_back(Warp{b, chunk, give_up, std::mt19937(rng())});
  std::vector<std::thread> threads;
  for (auto &w : ws) threads.emplace_back([&w, stages] { walk_staged_bin(w, w.b.count, w.chunk, stages); });
  for (auto &t : threads) t.join();
  unsigned marks = 0;
  for (unsigned k = 0; k < b.count; ++k) {
    EXPECT(b.results[k] + b.marks[k] == 1);  // every taskset has one result or one mark
    marks += (unsigned)b.marks[k];
  }
  EXPECT(marks == b.marked);  // what the second launch is told is what it finds
  for (auto &w : ws) EXPECT(!w.busy || w.waited_again);  // nobody leaves with copies under way unwaited
  return wrong;
}

/* staged_walk.h -- the way of one warp through a size bin whose tasksets it stages: what it pulls, tries,
 * keeps for its own end and leaves to the second launch.  Plain C++ without CUDA: the kernel
 * (rta_staged.cuh) supplies the steps, and a host program can too. */
#ifndef GCAPS_STAGED_WALK_H_
#define GCAPS_STAGED_WALK_H_

#ifdef __CUDACC__
#define STAGED_FN __device__ __forceinline__
#else
#define STAGED_FN inline
#endif

constexpr int kLeftMost = 8; /* undecided tasksets a warp keeps for its own end */
constexpr int kRunMost = 8;  /* undecided ones in a row after which it stages no more */

/* Far from schedulable, a taskset ends with a miss among its first ranks, and this is the way to find
 * it; where more ranks converge, looking at the first ones alone is wasted.  Tasksets of a batch tend
 * to be alike: a warp that meets kRunMost undecided ones in a row, or one when most warps' first taskset
 * was undecided too, marks what it pulls for the second launch and only tries one in 256.  A few
 * undecided ones it keeps and takes through the full pass itself when there is nothing left to pull.
 *
 * A wait for copies that gives up ends the use of the stage, never the work: all that the warp holds and
 * all that it pulls from then on goes to the second launch, which needs no stage.
 *
 * Entries of the bin are numbered from 0 to count - 1; a warp pulls `chunk` of them at a time.  Steps of w:
 *   pull(n)             the first of the next n entries (the counter moves on)
 *   ask(n), answer()    the same in two halves, so that the answer can take its time
 *   look_up(first, h)   looks entries first .. first + chunk - 1 up into half h of its table
 *   take(h, c)          the taskset in place c of half h is the current one
 *   start_copies(h, c)  starts the copies of the taskset in place c of half h; false: it cannot be staged
 *   wait()              the copies under way have arrived; false: gave up waiting
 *   head(next)          tries the first ranks of the current taskset, which is staged; calls next() once,
 *                       when nothing reads the stage any more; true: decided, results written
 *   first_try(decided)  how the warp's first try went
 *   most_undecided()    whether most warps' first tries were undecided
 *   keep(k, entry)      notes the k-th entry kept for the end
 *   mark(first, n)      leaves entries to the second launch (n <= 32)
 *   mark_kept(k)        the same for a kept one
 *   full_pass(k)        the whole analysis of a kept one; the stage is free
 *   marked(n)           how many were left to the second launch
 * `stages`: false if no taskset of this call can be staged. */
template <class Warp>
STAGED_FN void walk_staged_bin(Warp &w, unsigned int count, unsigned int chunk, bool stages) {
  bool defer_all = !stages, first_one = true, gave_up = false;
  int undecided_run = 0, n_left = 0, which = 0;
  bool staged = false; /* the copies of the coming taskset have been started */
  unsigned int deferred = 0;
  unsigned int first = w.pull(chunk);
  if (first >= count) return;
  w.look_up(first, which);
  if (!defer_all) staged = w.start_copies(which, 0);
  while (first < count) {
    unsigned int nfirst = 0;
    w.ask(chunk);
    const int in_chunk = count - first < chunk ? (int)(count - first) : (int)chunk;
#ifdef __CUDACC__
#pragma unroll 1
#endif
    for (int c = 0; c < in_chunk; ++c) {
      if (c == 1 || in_chunk == 1) { /* the next chunk's index has arrived by now */
        nfirst = w.answer();
        w.look_up(nfirst, which ^ 1);
      }
      w.take(which, c);
      const bool more = c + 1 < in_chunk || nfirst < count;
      const int next_half = c + 1 < in_chunk ? which : which ^ 1, next_place = c + 1 < in_chunk ? c + 1 : 0;
      bool decided = false;
      if (staged) {
        staged = false;
        if (!w.wait()) {
          gave_up = true, stages = false, defer_all = true;
        } else if (!defer_all) {
          decided = w.head([&] {
            if (more) staged = w.start_copies(next_half, next_place);
          });
          undecided_run = decided ? 0 : undecided_run + 1;
          if (first_one) w.first_try(decided);
          first_one = false;
          if (undecided_run > 0) defer_all = undecided_run >= kRunMost || w.most_undecided();
        }
      } else if (more && !defer_all) {
        staged = w.start_copies(next_half, next_place);
      }
      if (!decided) {
        if (defer_all || n_left == kLeftMost) {
          w.mark(first + (unsigned int)c, 1);
          deferred += 1;
        } else {
          w.keep(n_left, first + (unsigned int)c);
          n_left += 1;
        }
      }
    }
    first = nfirst;
    which ^= 1;
    if (defer_all && first < count) {
      if (staged) { /* (what has been copied for the coming taskset is not looked at) */
        staged = false;
        if (!w.wait()) gave_up = true, stages = false;
      }
      const unsigned int held = count - first < chunk ? count - first : chunk;
      w.mark(first, held);
      deferred += held;
      int k = 0;
      do {
        first = w.pull(32);
        if (first < count) {
          const unsigned int n = count - first < 32u ? count - first : 32u;
          w.mark(first, n);
          deferred += n;
        }
      } while (first < count && (++k < 8 || !stages));
      if (first < count) first = w.pull(chunk);
      if (first < count) { /* one try: if it is undecided too, the rest of its chunk is deferred again */
        w.look_up(first, which);
        defer_all = false;
        undecided_run = kRunMost - 1;
        staged = w.start_copies(which, 0);
      }
    }
  }
  if (gave_up) {
    for (int k = 0; k < n_left; ++k) w.mark_kept(k);
    deferred += (unsigned int)n_left;
    w.wait(); /* the warp's shared memory goes to another block: its own copies get one more wait */
  }
  if (deferred > 0) w.marked(deferred);
  if (!gave_up) {
#ifdef __CUDACC__
#pragma unroll 1
#endif
    for (int k = 0; k < n_left; ++k) w.full_pass(k);
  }
}

#endif /* GCAPS_STAGED_WALK_H_ */

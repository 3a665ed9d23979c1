// spin_limit.h -- when a wait on another block's progress gives up: after a
// second (or 2^26 polls) in which the word that shows the others at work did
// not change.  Plain C as well as CUDA, so that a host test can check it.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define SPIN_FN __host__ __device__ __forceinline__
#else
#define SPIN_FN static inline
#endif

#define SPIN_LIMIT_NS 1000000000ull
#define SPIN_LIMIT_POLLS (1u << 26)

typedef struct {
  uint64_t t0, seen;  // start of the current second, the word's value then
  uint32_t polls;     // since then
} spin_limit;

SPIN_FN void spin_start(spin_limit* s, uint64_t word) {
  s->t0 = 0;
  s->seen = word;
  s->polls = 0;
}
// after a poll in vain at time now: is it time to look at the word?
SPIN_FN int spin_due(spin_limit* s, uint64_t now) {
  if (s->polls++ == 0) s->t0 = now;
  return s->polls > SPIN_LIMIT_POLLS || now - s->t0 > SPIN_LIMIT_NS;
}
// the word's value at that time: give up?  If not, a new second starts.
SPIN_FN int spin_over(spin_limit* s, uint64_t now, uint64_t word) {
  if (word == s->seen) return 1;
  s->t0 = now;
  s->seen = word;
  s->polls = 1;
  return 0;
}

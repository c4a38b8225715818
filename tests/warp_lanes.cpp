// The lanes of warp_lanes.h.  Compiled without ThreadSanitizer, so that the
// scheduler's own data do not count; it only reports the fibers and the memory
// order of __syncwarp.
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <functional>

#include <ucontext.h>

extern "C" {
void* __tsan_get_current_fiber(void);
void* __tsan_create_fiber(unsigned flags);
void __tsan_switch_to_fiber(void* fiber, unsigned flags);
void __tsan_acquire(void* at);
void __tsan_release(void* at);
}

namespace warp {
struct Index {
  int x;
};
namespace {
struct Token;
constexpr unsigned kNoSync = 1;  // a switch of fibers orders nothing
constexpr size_t kStack = 1 << 18;
constexpr int kMost = 1024;
struct Lane {
  ucontext_t ctx;
  void* fiber;
  char* stack;
  bool done, waiting;
  unsigned mask;
  Token* token;  // a barrier's
  int line;
  uint64_t val;
  volatile uint64_t out[32];
};
Lane lanes[kMost];
ucontext_t home;
void* home_fiber;
int current;
const std::function<void(int)>* body;
// What orders memory at a barrier, one per mask of a lane group (first lane,
// number of lanes) and one for the block.  A lane resumes from a barrier when
// others may be at the next one already, which must not count: two in turn.
struct Token {
  char at[2];
  unsigned passed;
};
Token token[kMost / 32][32][33], block_token;

void enter(int l) {
  (*body)(l);
  lanes[l].done = true;
  __tsan_switch_to_fiber(home_fiber, 0);
  swapcontext(&lanes[l].ctx, &home);
}
}  // namespace

Index thread_idx() { return Index{current}; }

void meet(unsigned mask, uint64_t val, uint64_t out[32], int line, bool orders_memory) {
  Lane& me = lanes[current];
  const int l = current & 31;
  if (!(mask >> l & 1)) {
    std::printf("lane %d is not in its mask %x, line %d\n", l, mask, line);
    std::exit(2);
  }
  Token& k = token[current >> 5][__builtin_ctz(mask)][__builtin_popcount(mask)];
  char* const t = &k.at[k.passed & 1];
  if (orders_memory) __tsan_release(t);
  me.mask = mask;
  me.token = orders_memory ? &k : nullptr;
  me.val = val;
  me.line = line;
  me.waiting = true;
  __tsan_switch_to_fiber(home_fiber, kNoSync);
  swapcontext(&me.ctx, &home);
  if (orders_memory) __tsan_acquire(t);
  for (int i = 0; i < 32; ++i) out[i] = me.out[i];
}

// mask 0: the whole block
void block_barrier(int line) {
  Lane& me = lanes[current];
  char* const t = &block_token.at[block_token.passed & 1];
  __tsan_release(t);
  me.mask = 0;
  me.line = line;
  me.waiting = true;
  __tsan_switch_to_fiber(home_fiber, kNoSync);
  swapcontext(&me.ctx, &home);
  __tsan_acquire(t);
}

bool run(const std::function<void(int)>& f, int n, bool downwards) {
  body = &f;
  home_fiber = __tsan_get_current_fiber();
  for (int l = 0; l < n; ++l) {
    Lane& me = lanes[l];
    me.done = me.waiting = false;
    if (!me.stack) me.stack = (char*)std::malloc(kStack);
    me.fiber = __tsan_create_fiber(0);
    getcontext(&me.ctx);
    me.ctx.uc_stack.ss_sp = me.stack;
    me.ctx.uc_stack.ss_size = kStack;
    me.ctx.uc_link = &home;
    makecontext(&me.ctx, (void (*)())enter, 1, l);
  }
  for (;;) {
    bool ran = false, all = true, block = true;
    for (int i = 0; i < n; ++i) {
      const int l = downwards ? n - 1 - i : i;
      if (lanes[l].done) continue;
      all = false;
      if (!lanes[l].waiting) {
        ran = true;
        current = l;
        __tsan_switch_to_fiber(lanes[l].fiber, kNoSync);
        swapcontext(&home, &lanes[l].ctx);
      }
    }
    if (all) return true;
    for (int l = 0; l < n; ++l) {
      if (lanes[l].done || !lanes[l].waiting) continue;
      const unsigned m = lanes[l].mask;
      if (m == 0) continue;
      Lane* const w = &lanes[l & ~31];
      bool ready = true;
      for (int i = 0; i < 32; ++i)
        if (m >> i & 1)
          ready = ready && !w[i].done && w[i].waiting && w[i].mask == m && w[i].line == lanes[l].line;
      if (!ready) continue;
      ran = true;
      if (lanes[l].token) ++lanes[l].token->passed;
      for (int i = 0; i < 32; ++i)
        if (m >> i & 1) {
          for (int q = 0; q < 32; ++q) w[i].out[q] = m >> q & 1 ? w[q].val : 0;
          w[i].waiting = false;
        }
    }
    for (int l = 0; l < n; ++l)
      block = block && !lanes[l].done && lanes[l].waiting && lanes[l].mask == 0;
    if (block) {
      ran = true;
      ++block_token.passed;
      for (int l = 0; l < n; ++l) lanes[l].waiting = false;
    }
    if (!ran) {
      for (int l = 0; l < n; ++l)
        std::printf("thread %d done %d waits at line %d, mask %x\n", l, lanes[l].done,
                    lanes[l].line, lanes[l].mask);
      return false;
    }
  }
}
}  // namespace warp

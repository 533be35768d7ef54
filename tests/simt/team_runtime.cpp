// TEST INFRASTRUCTURE: simt_runtime.cpp with teams (thread-block clusters).
//
// A CTA is a host thread whose CUDA threads are fibers, as in simt_runtime.cpp;
// the CTAs of a team take turns, one at a time, so a run is deterministic.
// SIMT_TEAM_FIRST=K sets the turns: from one team barrier to the next, every
// CTA but rank 0 runs K fiber slices (a slice: one fiber up to its next
// wait), then rank 0 runs until it waits at the team barrier, then the others
// do.  K = 0 is rank 0 first; a small K leaves the others' CTAs cut in two by
// whatever rank 0 does in the whole phase.  A kernel without races
// between its CTAs gives the same bits for every K.  Barriers that do not match
// (some fibers at a CTA's barrier, the rest at the team's, or a CTA's fibers at
// different barriers with none to open) end the process with a message.
#include <ucontext.h>

#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

#include "simt_prelude.h"
#include "team_prelude.h"

namespace simt {
namespace {

enum State { RUNNABLE, AT_BLOCK, AT_WARP, AT_NAMED, AT_TEAM, DONE };
enum Cta { RUNNING, WAITING, FINISHED };         // WAITING: every live fiber is at the team barrier

struct Fiber {
  ucontext_t ctx;
  std::unique_ptr<char[]> stack;
  State state = RUNNABLE;
  Idx tid{0, 0, 0};
  int bar_id = 0, bar_count = 0;
};

constexpr size_t kStack = 256 * 1024;

struct Block {
  std::vector<Fiber> fibers;
  std::vector<unsigned char> smem;
  std::vector<uint64_t> xbuf;
  ucontext_t main;
  Fiber* cur = nullptr;
  Idx bid{0, 0, 0}, bdim{1, 1, 1}, gdim{1, 1, 1};
  const std::function<void()>* body = nullptr;
  size_t next = 0;                               // fiber of the next slice
  Cta state = RUNNING;
  // turn: slices granted by the main thread (-1: none)
  std::mutex mu;
  std::condition_variable cv;
  long turn = -1;
  bool quit = false;
  std::thread host;
};

thread_local Block* g_b = nullptr;

void wait(State s) {
  g_b->cur->state = s;
  swapcontext(&g_b->cur->ctx, &g_b->main);
}

void entry() {
  (*g_b->body)();
  g_b->cur->state = DONE;
  swapcontext(&g_b->cur->ctx, &g_b->main);
}

void open_all(Block& b, State s) {
  for (Fiber& f : b.fibers)
    if (f.state == s) f.state = RUNNABLE;
}

// Opens the barriers of a CTA whose live fibers all wait at them.
bool release(Block& b) {
  bool any = false, all_block = true, some_block = false;
  for (const Fiber& f : b.fibers) {
    if (f.state == DONE) continue;
    if (f.state == AT_BLOCK) some_block = true;
    else all_block = false;
  }
  if (some_block && all_block) {
    open_all(b, AT_BLOCK);
    return true;
  }
  for (int id = 1; id < 16; ++id) {
    int waiting = 0, count = -1;
    for (const Fiber& f : b.fibers)
      if (f.state == AT_NAMED && f.bar_id == id) ++waiting, count = f.bar_count;
    if (waiting == 0 || waiting != count) continue;
    for (Fiber& f : b.fibers)
      if (f.state == AT_NAMED && f.bar_id == id) f.state = RUNNABLE;
    any = true;
  }
  const size_t n = b.fibers.size();
  for (size_t w0 = 0; w0 < n; w0 += 32) {
    bool all = true, some = false;
    for (size_t i = w0; i < std::min(n, w0 + 32); ++i) {
      if (b.fibers[i].state == DONE) continue;
      if (b.fibers[i].state == AT_WARP) some = true;
      else all = false;
    }
    if (!some || !all) continue;
    for (size_t i = w0; i < std::min(n, w0 + 32); ++i)
      if (b.fibers[i].state == AT_WARP) b.fibers[i].state = RUNNABLE;
    any = true;
  }
  return any;
}

// Runs up to `slices` fiber slices of b (on its own host thread).
void run(Block& b, long slices) {
  while (slices > 0) {
    bool runnable = false, live = false, team = true;
    for (const Fiber& f : b.fibers) {
      if (f.state == DONE) continue;
      live = true;
      if (f.state == RUNNABLE) runnable = true;
      if (f.state != AT_TEAM) team = false;
    }
    if (!live) {
      b.state = FINISHED;
      return;
    }
    if (team) {
      b.state = WAITING;
      return;
    }
    if (!runnable && !release(b)) {
      std::fprintf(stderr, "simt: block %u: barriers do not match (no fiber can run)\n", b.bid.x);
      std::abort();
    }
    for (size_t k = 0; k < b.fibers.size() && slices > 0; ++k) {
      Fiber& f = b.fibers[b.next];
      b.next = (b.next + 1) % b.fibers.size();
      if (f.state != RUNNABLE) continue;
      b.cur = &f;
      swapcontext(&b.main, &f.ctx);
      --slices;
    }
  }
}

void host_main(Block* b) {
  g_b = b;
  for (Fiber& f : b->fibers) {
    getcontext(&f.ctx);
    f.ctx.uc_stack.ss_sp = f.stack.get();
    f.ctx.uc_stack.ss_size = kStack;
    f.ctx.uc_link = nullptr;
    makecontext(&f.ctx, entry, 0);
  }
  std::unique_lock<std::mutex> lock(b->mu);
  for (;;) {
    b->cv.wait(lock, [b] { return b->turn >= 0 || b->quit; });
    if (b->quit) return;
    run(*b, b->turn);
    b->turn = -1;
    b->cv.notify_all();
  }
}

void give(Block& b, long slices) {
  if (b.state != RUNNING || slices <= 0) return;
  std::unique_lock<std::mutex> lock(b.mu);
  b.turn = slices;
  b.cv.notify_all();
  b.cv.wait(lock, [&b] { return b.turn < 0; });
}

}  // namespace

Idx tid() { return g_b->cur->tid; }
Idx bid() { return g_b->bid; }
Idx bdim() { return g_b->bdim; }
Idx gdim() { return g_b->gdim; }
void sync() { wait(AT_BLOCK); }
void syncwarp() { wait(AT_WARP); }
void team_sync() { wait(AT_TEAM); }
void named_sync(int id, int count) {
  g_b->cur->bar_id = id;
  g_b->cur->bar_count = count;
  wait(AT_NAMED);
}
uint64_t exchange(uint64_t bits, int lane_xor) {
  const unsigned t = g_b->cur->tid.x, w0 = t & ~31u;
  g_b->xbuf[t] = bits;
  wait(AT_WARP);
  const uint64_t out = g_b->xbuf[w0 + (((t - w0) ^ (unsigned)lane_xor) & 31u)];
  wait(AT_WARP);
  return out;
}
void* dynamic_smem() { return g_b->smem.data(); }

void launch_team(int team, unsigned grid, unsigned block, size_t smem, const std::function<void()>& body) {
  const char* e = std::getenv("SIMT_TEAM_FIRST");
  const long first = e ? std::atol(e) : 0, all = 1L << 60;
  for (unsigned b0 = 0; b0 < grid; b0 += team) {
    std::vector<std::unique_ptr<Block>> ctas;
    for (int r = 0; r < team; ++r) {
      ctas.emplace_back(new Block);
      Block& b = *ctas.back();
      b.bid = {b0 + r, 0, 0};
      b.bdim = {block, 1, 1};
      b.gdim = {grid, 1, 1};
      b.smem.assign(smem + 16, 0);
      b.xbuf.assign(block, 0);
      b.body = &body;
      b.fibers.resize(block);
      for (unsigned t = 0; t < block; ++t) {
        b.fibers[t].tid = {t, 0, 0};
        b.fibers[t].stack.reset(new char[kStack]);
      }
      b.host = std::thread(host_main, &b);
    }
    for (;;) {
      for (int r = 1; r < team; ++r) give(*ctas[r], first);
      for (int r = 0; r < team; ++r) give(*ctas[r], all);
      bool live = false;
      for (auto& b : ctas)
        if (b->state == WAITING) {
          live = true;
          b->state = RUNNING;
          open_all(*b, AT_TEAM);
        }
      if (!live) break;
    }
    for (auto& b : ctas) {
      {
        std::lock_guard<std::mutex> lock(b->mu);
        b->quit = true;
        b->cv.notify_all();
      }
      b->host.join();
    }
  }
}

void launch(unsigned grid, unsigned block, size_t smem, const std::function<void()>& body) {
  launch_team(1, grid, block, smem, body);
}

}  // namespace simt

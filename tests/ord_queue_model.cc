// The ordered queue (csrc/lr_ordq.h) under arbitrary interleavings, on the
// host: every group of threads is a coroutine that gives way before each
// memory operation, and a scheduler decides who goes on.  Usage:
//   ord_queue_model SCHEDULES   random schedules, some of which hold groups
//                               back before they look for the next chunk
//   ord_queue_model held        groups held back while a window is opened,
//                               so that they share out the chunk after it
// Prints "ok" when every position was handed out exactly once.
#include <ucontext.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <memory>
#include <random>
#include <vector>

#include "lr_ordq.h"

namespace {

enum Op { kAddWindow, kExchangeWindow, kWindow, kTakeNext, kGiveNext, kDraw, kOut, kSetOut, kNewRequest };

struct Cta {
  unsigned long long win = 0, next = 0;
  uint32_t out = 0;
};

struct Group {
  ucontext_t ctx;
  std::vector<char> stack;
  std::function<void()> body;
  Op pending = kNewRequest;          // what it does when it goes on
  bool done = false;
};

ucontext_t g_scheduler;
Group *g_running = nullptr;

void give_way(Op op) {
  Group *g = g_running;
  g->pending = op;
  swapcontext(&g->ctx, &g_scheduler);
}

struct Queue {
  Cta *c;
  uint32_t *counter;
  unsigned long long add_window(uint32_t n) const { give_way(kAddWindow); auto w = c->win; c->win += n; return w; }
  void exchange_window(unsigned long long w) const { give_way(kExchangeWindow); c->win = w; }
  unsigned long long window() const { give_way(kWindow); return c->win; }
  unsigned long long exchange_next(unsigned long long w) const {
    give_way(w ? kGiveNext : kTakeNext);
    auto old = c->next;
    c->next = w;
    return old;
  }
  uint32_t draw(uint32_t n) const { give_way(kDraw); uint32_t j = *counter; *counter += n; return j; }
  bool out() const { give_way(kOut); return c->out != 0; }
  void set_out() const { give_way(kSetOut); c->out = 1; }
};

struct World {
  uint64_t total;
  uint32_t counter = 0;
  std::vector<Cta> ctas;
  std::vector<std::unique_ptr<Group>> groups;
  std::vector<uint32_t> seen;

  World(uint64_t n, int nctas, uint32_t first) : total(n), ctas(nctas), seen(n, 0) {
    for (Cta &c : ctas) {            // the CTA's first window, as k_chase draws it
      const uint32_t j = counter;
      counter += first;
      c.win = j < total ? lr::ord_window(j, (uint32_t)std::min<uint64_t>(j + first, total)) : 0;
      c.out = j >= total;
    }
  }
  static void enter() {
    g_running->body();
    g_running->done = true;
    swapcontext(&g_running->ctx, &g_scheduler);
  }
  Group *add(std::function<void()> body) {
    groups.emplace_back(new Group);
    Group *g = groups.back().get();
    g->stack.resize(64 << 10);
    g->body = std::move(body);
    getcontext(&g->ctx);
    g->ctx.uc_stack.ss_sp = g->stack.data();
    g->ctx.uc_stack.ss_size = g->stack.size();
    g->ctx.uc_link = nullptr;
    makecontext(&g->ctx, (void (*)())enter, 0);
    return g;
  }
  void step(Group *g) {
    g_running = g;
    swapcontext(&g_scheduler, &g->ctx);
  }
  void run(Group *g) { while (!g->done) step(g); }
  void run_until(Group *g, Op op) { do step(g); while (!g->done && g->pending != op); }
  // One request of cnt threads: how many got a position.
  uint32_t ask(int cta, uint32_t cnt) {
    uint32_t fresh = 0xFFFFFFFFu, got = 0, again = 0;
    const Queue q{&ctas[cta], &counter};
    const unsigned long long win = q.add_window(cnt);
    const unsigned long long s = lr::ord_ask(q, win, cnt, (uint32_t)total, &fresh);
    for (uint32_t i = 0; i < cnt; ++i) {
      const uint32_t p = lr::ord_position(win, lr::ord_window_has(win, cnt), s, (uint32_t)total, i);
      if (p == lr::kOrdAgain) { again++; continue; }
      if (p >= total) continue;
      ++seen[p];
      ++got;
    }
    return got + (again ? ask(cta, again) : 0);
  }
  bool good() const {
    for (uint64_t p = 0; p < total; ++p)
      if (seen[p] != 1) {
        printf("position %llu handed out %u times\n", (unsigned long long)p, seen[p]);
        return false;
      }
    return true;
  }
};

bool random_schedule(uint32_t seed) {
  std::mt19937 rng(seed);
  auto below = [&](uint32_t n) { return (uint32_t)(rng() % n); };
  const int nctas = 1 + (int)below(3), warps = 2 + (int)below(14);
  const uint64_t total = 1 + below(6000);
  World w(total, nctas, 2u * 32u * (1u + below(4)));
  for (int c = 0; c < nctas; ++c)
    for (int k = 0; k < warps; ++k)
      w.add([&w, &below, c] {
        uint32_t alive = 32;
        while (alive) {
          const uint32_t cnt = below(2) ? alive : 1u + below(alive);
          alive -= cnt - w.ask(c, cnt);
        }
      });
  const uint32_t hold = below(2) ? 0u : 50u + below(400);      // steps a held group is passed over
  std::vector<uint32_t> held(w.groups.size(), 0);
  for (size_t left = w.groups.size(); left;) {
    const size_t i = below((uint32_t)w.groups.size());
    Group *g = w.groups[i].get();
    if (g->done) continue;
    if (hold && g->pending == kTakeNext && held[i]++ < hold / w.groups.size()) continue;
    held[i] = 0;
    w.step(g);
    if (g->done) --left;
  }
  return w.good();
}

// The groups of one CTA ask for `lanes` each at a window that has run out and
// are held back; another opens the next window, brings it down to the mark,
// and draws the chunk after it, which the held ones then share out.
bool held_schedule(uint32_t lanes, int ngroups, uint64_t total) {
  World w(total, 2, 128);
  for (int i = 0; i < 4; ++i) w.run(w.add([&] { w.ask(0, 32); }));      // the first window, and a chunk drawn at its mark
  std::vector<Group *> held;
  for (int i = 0; i < ngroups; ++i) {
    held.push_back(w.add([&] { w.ask(0, lanes); }));
    w.run_until(held.back(), kTakeNext);
  }
  w.run(w.add([&] { w.ask(0, 32); }));          // opens the next window
  w.run(w.add([&] { w.ask(0, 32); }));          // brings it down to the mark
  for (Group *g : held) w.run(g);
  for (int c = 0; c < 2; ++c)                   // the rest, in turns
    w.run(w.add([&w, c] { while (w.ask(c, 32)) {} }));
  return w.good();
}

}  // namespace

int main(int argc, char **argv) {
  if (argc > 1 && !strcmp(argv[1], "held")) {
    for (uint32_t lanes = 1; lanes <= 32; ++lanes)
      for (int groups = 1; groups <= 16; ++groups)
        for (uint64_t total : {300u, 384u, 430u, 512u, 560u, 2000u})
          if (!held_schedule(lanes, groups, total)) {
            printf("%u lanes, %d groups, %llu positions\n", lanes, groups, (unsigned long long)total);
            return 1;
          }
  } else {
    const int n = argc > 1 ? atoi(argv[1]) : 1000;
    for (int seed = 0; seed < n; ++seed)
      if (!random_schedule((uint32_t)seed)) {
        printf("schedule %d\n", seed);
        return 1;
      }
  }
  printf("ok\n");
  return 0;
}

// Every order in which the blocks of a sequence can take the steps of seq_status.cuh, on the CPU: a block is a coroutine that
// stops ahead of each access to memory, and the program goes through all choices of who is next.
// Prints the number of orders; exits 1 with the first that loses a failure, reports one that did not happen, leaves the word
// other than zero or makes a block wait for good.
#include <ucontext.h>

#include <cstdio>
#include <cstdlib>
#include <functional>
#include <vector>

#include "seq_status.cuh"

enum Fate { kFine, kAborted, kLate };

static unsigned long long g_word;
static int g_status, g_blocks;
static ucontext_t g_main;
struct Task {
  ucontext_t ctx;
  std::vector<char> stack = std::vector<char>(32768);
  Fate fate;
  bool done, polls;   // polls: its next step looks whether the count is zero
};
static std::vector<Task> g_tasks(3);
static int g_now;

static void step() { swapcontext(&g_tasks[g_now].ctx, &g_main); }

struct Words {
  unsigned long long add(unsigned long long v) { step(); const unsigned long long was = g_word; g_word += v; return was; }
  unsigned count() {   // asked again only when it is zero: what it sees before changes nothing
    g_tasks[g_now].polls = true;
    step();
    g_tasks[g_now].polls = false;
    return (unsigned)g_word;
  }
  void clear() { step(); g_word = 0; }
  void put(int s) { step(); g_status = s; }
  void fence() {}
  void correct() { step(); if (g_status == CLV_OK) g_status = CLV_ERR_TIMEOUT; }
  bool expired() { return false; }
};

static void block() {
  Task& t = g_tasks[g_now];
  Words w;
  const unsigned long long found = clv::add_block(w, t.fate == kAborted);
  clv::publish_if_last(w, found, (unsigned)g_blocks);
  if (t.fate == kLate) clv::report_late(w, (unsigned)g_blocks);
  t.done = true;
  swapcontext(&t.ctx, &g_main);
}

static long run_all(int blocks, const std::vector<Fate>& fate, bool malformed, int before) {
  std::vector<int> choice, of;   // at each step: which of the blocks that can go on, and how many there were
  long orders = 0;
  const auto fail = [&](const char* what) {
    std::printf("%s: %d blocks, fates", what, blocks);
    for (Fate f : fate) std::printf(" %d", f);
    std::printf(", malformed %d, before %d, status %d, word %llx, choices", malformed, before, g_status, g_word);
    for (int c : choice) std::printf(" %d", c);
    std::printf("\n");
    std::exit(1);
  };
  for (;;) {
    g_word = malformed ? 1ull << 32 : 0ull;   // put there ahead of its block's count
    g_status = before;
    g_blocks = blocks;
    for (int i = 0; i < blocks; ++i) {
      Task& t = g_tasks[i];
      t.fate = fate[i];
      t.done = t.polls = false;
      getcontext(&t.ctx);
      t.ctx.uc_stack.ss_sp = t.stack.data();
      t.ctx.uc_stack.ss_size = t.stack.size();
      t.ctx.uc_link = &g_main;
      makecontext(&t.ctx, block, 0);
      g_now = i;
      swapcontext(&g_main, &t.ctx);   // to its first access
    }
    for (size_t n = 0;; ++n) {
      std::vector<int> able;
      bool all_done = true;
      for (int i = 0; i < blocks; ++i) {
        all_done &= g_tasks[i].done;
        if (!g_tasks[i].done && !(g_tasks[i].polls && (unsigned)g_word != 0u)) able.push_back(i);
      }
      if (all_done) break;
      if (able.empty()) fail("a block waits for good");
      if (n == choice.size()) { choice.push_back(0); of.push_back((int)able.size()); }
      g_now = able[choice[n]];
      swapcontext(&g_main, &g_tasks[g_now].ctx);
    }
    ++orders;
    bool failed = false;
    for (Fate f : fate) failed |= f != kFine;
    if (g_status != (malformed ? CLV_ERR_TREE : failed ? CLV_ERR_TIMEOUT : CLV_OK)) fail("wrong status");
    if (g_word != 0) fail("the word is left other than zero");
    while (!choice.empty() && choice.back() + 1 == of.back()) { choice.pop_back(); of.pop_back(); }
    if (choice.empty()) return orders;
    ++choice.back();
  }
}

int main() {
  long orders = 0;
  for (int blocks = 1; blocks <= 3; ++blocks) {
    int all = 1;
    for (int i = 0; i < blocks; ++i) all *= 3;
    for (int code = 0; code < all; ++code) {
      std::vector<Fate> fate;
      int late = 0;
      for (int i = 0, c = code; i < blocks; ++i, c /= 3) { fate.push_back((Fate)(c % 3)); late += c % 3 == kLate; }
      if (late > 2) continue;   // (three late ones of three: over a million orders)
      for (int before : {(int)CLV_OK, (int)CLV_ERR_TIMEOUT, -7}) {
        orders += run_all(blocks, fate, false, before);
        if (late < 2) orders += run_all(blocks, fate, true, before);
      }
    }
  }
  std::printf("%ld\n", orders);
}

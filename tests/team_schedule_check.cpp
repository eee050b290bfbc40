// Host check of the team evolver's exchange buffers (team_schedule.h): every write of a
// buffer is ordered against every other access of it.
//
// Cluster form: two CTAs of two threads each, thread t of either sending to CTA t (the
// sparsest pattern the kernel has: a CTA's words for one partner come from some of its
// threads only).  The accesses of several steps are laid out as the kernel makes them;
// a happens-before relation is closed over program order, the CTA's barriers and the
// arrival of sent words (a wait orders the waiting CTA behind the threads that sent to
// it, no others).
//
// Word form: the same two CTAs, the fences run by a third thread of each or by the first
// one.  Between
// CTAs only a fence before the sent words and a fence behind their arrival order
// anything: the arrival itself is a relaxed load.
// Prints "ok" and exits 0, else prints the first violation and exits 1.
#include <cstdio>
#include <utility>
#include <vector>

#include "team_schedule.h"

namespace {

constexpr int kSteps = 11;

struct Event {
  int cta, thread, step;
  const char* what;
  int mem_cta, buffer;  // memory accessed; buffer -1: none
  bool write;
};

struct Graph {
  std::vector<Event> ev;
  std::vector<std::vector<int>> next;
  std::vector<std::pair<int, int>> own;  // a store and the take that waits for its word
  int last[2][3];
  Graph() {
    for (auto& c : last)
      for (int& t : c) t = -1;
  }
  int add(const Event& e) {
    ev.push_back(e);
    next.emplace_back();
    const int i = static_cast<int>(ev.size()) - 1;
    int& l = last[e.cta][e.thread];
    if (l >= 0) next[l].push_back(i);
    return l = i;
  }
  // a barrier among the threads [0, nt) of every CTA
  void barrier(int j, int nt) {
    for (int c = 0; c < 2; ++c) {
      std::vector<int> in, out;
      for (int t = 0; t < nt; ++t) in.push_back(add({c, t, j, "arrive", c, -1, false}));
      for (int t = 0; t < nt; ++t) out.push_back(add({c, t, j, "leave", c, -1, false}));
      for (int a : in)
        for (int b : out) next[a].push_back(b);
    }
  }
  std::vector<char> after(int i) const {
    std::vector<char> seen(ev.size(), 0);
    std::vector<int> todo{i};
    while (!todo.empty()) {
      const int k = todo.back();
      todo.pop_back();
      for (int m : next[k])
        if (!seen[m]) seen[m] = 1, todo.push_back(m);
    }
    return seen;
  }
  int check(const char* form) const {
    std::vector<std::vector<char>> reach;
    for (size_t i = 0; i < ev.size(); ++i) reach.push_back(after(static_cast<int>(i)));
    for (size_t a = 0; a < ev.size(); ++a)
      for (size_t b = a + 1; b < ev.size(); ++b) {
        const Event &x = ev[a], &y = ev[b];
        if (x.buffer < 0 || x.buffer != y.buffer || x.mem_cta != y.mem_cta || !(x.write || y.write)) continue;
        // threads write parts of their own of one transpose or exchange
        if (x.write && y.write && x.step == y.step && x.what == y.what) continue;
        bool word = false;
        for (const auto& p : own) word = word || (p.first == static_cast<int>(a) && p.second == static_cast<int>(b));
        if (!word && !reach[a][b] && !reach[b][a]) {
          std::printf("%s: buffer %d of CTA %d: %s of CTA %d thread %d step %d and %s of CTA %d thread %d step %d unordered\n", form,
                      x.buffer, x.mem_cta, x.what, x.cta, x.thread, x.step, y.what, y.cta, y.thread, y.step);
          return 1;
        }
      }
    return 0;
  }
};

int cluster() {
  Graph g;
  auto all = [&](int j, const char* what, int buffer, bool write) {
    for (int c = 0; c < 2; ++c)
      for (int t = 0; t < 2; ++t) g.add({c, t, j, what, c, buffer, write});
  };
  for (int j = 0; j < kSteps; ++j) {
    for (int k = 0; k < 2; ++k) {
      all(j, k ? "put 1" : "put 0", qaa::cluster_transpose(j, k), true);
      g.barrier(j, 2);
      all(j, k ? "get 1" : "get 0", qaa::cluster_transpose(j, k), false);
    }
    int sent[2][2];  // [receiver][sender]
    for (int c = 0; c < 2; ++c)
      for (int t = 0; t < 2; ++t) sent[t][c] = g.add({c, t, j, "send", t, qaa::cluster_receive(j), true});
    for (int c = 0; c < 2; ++c)
      for (int t = 0; t < 2; ++t) {
        const int w = g.add({c, t, j, "wait", c, -1, false});
        for (int s = 0; s < 2; ++s) g.next[sent[c][s]].push_back(w);
      }
    g.barrier(j, 2);
    all(j, "get received", qaa::cluster_receive(j), false);
  }
  return g.check("cluster");
}

// A fence warp of its own (the stores of step j + kWordFenceLag wait for the fence behind
// step j), or thread 0 between the transposes of step j + 1.
int words(bool warp) {
  Graph g;
  const int lag = warp ? qaa::kWordFenceLag : 1;
  int fence[2][kSteps], leave[2][kSteps];  // the fence warp's fence and its release of step j
  int sent[2][2];                          // [receiver][sender], this step's
  for (int j = 0; j < kSteps; ++j) {
    g.barrier(j, 2);  // of the transposes
    if (!warp && j > 0) {
      for (int c = 0; c < 2; ++c) fence[c][j - 1] = g.add({c, 0, j, "fence", c, -1, false});
      g.barrier(j, 2);
    }
    if (warp && j >= lag)
      for (int c = 0; c < 2; ++c)
        for (int t = 0; t < 2; ++t) g.next[leave[c][j - lag]].push_back(g.add({c, t, j, "await fence", c, -1, false}));
    // slot of a buffer: by sender; thread s of the receiver takes the words of CTA s
    auto slot = [&](int sender) { return 2 * qaa::word_buffer(j) + sender; };
    for (int c = 0; c < 2; ++c)
      for (int t = 0; t < 2; ++t) sent[t][c] = g.add({c, t, j, "store", t, slot(c), true});
    for (int c = 0; c < 2; ++c)
      for (int t = 0; t < 2; ++t) g.own.push_back({sent[c][t], g.add({c, t, j, "take and empty", c, slot(t), true})});
    // the threads arrive, the fence warp waits for them
    for (int c = 0; warp && c < 2; ++c) {
      const int a0 = g.add({c, 0, j, "arrive", c, -1, false}), a1 = g.add({c, 1, j, "arrive", c, -1, false});
      fence[c][j] = g.add({c, 2, j, "fence", c, -1, false});
      g.next[a0].push_back(fence[c][j]);
      g.next[a1].push_back(fence[c][j]);
    }
    for (int c = 0; warp && c < 2; ++c) leave[c][j] = g.add({c, 2, j, "release", c, -1, false});
  }
  // a fence of the sender before a word it sends, and a fence of the receiver behind it
  for (int r = 0; r < 2; ++r)
    for (int j = lag; j < kSteps - 1; ++j) g.next[fence[1 - r][j - lag]].push_back(fence[r][j]);
  return g.check(warp ? "words, fence warp" : "words, thread 0's fence");
}

}  // namespace

int main() {
  if (cluster() || words(true) || words(false)) return 1;
  std::puts("ok");
  return 0;
}

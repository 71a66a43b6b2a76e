// A model of one CTA of the attention kernels: its warps as coroutines over
// named barriers, mbarriers, TMA loads and the MMA pipe, under random
// schedules.  The order of the hand-offs and what a role does after a failed
// wait are the kernels' own (handoff.h); the waits between them are restated
// here.  A wait that polls an mbarrier may fail at any time (a random
// failure) and fails for certain once nothing else can run (its time limit);
// a sync on a named barrier never does.  When only such syncs are left, the
// kernel would not end: the run is reported as stuck, as is one in which a warp
// arrived twice in a generation.
//
//   handoff_model KERNEL PROTOCOL SEEDS     KERNEL: fwd64 fwd128 dkdv dq
//   PROTOCOL: shipped, or a planted mistake: "burst" (the arrivals owed after a
//   failed wait are made all at once), "blocking" (each as a sync, without the
//   wait for the commit that shows the one before consumed), "one-ds" (dq: one
//   dS barrier)
// prints the number of runs, of those with a failed wait, and of stuck ones.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <ucontext.h>

#include <deque>
#include <functional>
#include <map>
#include <memory>
#include <random>
#include <string>
#include <utility>
#include <vector>

#include "handoff.h"

using namespace fastvr::handoff;

namespace {

struct Model;
Model* M = nullptr;

struct Task {
  ucontext_t ctx;
  std::vector<char> stack;
  std::function<void()> body;
  std::function<bool()> ready;  // what it waits for
  bool bounded = false;         // a wait with a time limit
  bool expired = false;
  bool done = false;
};

// A named barrier: counts warps.  Who they are, the hardware does not look at;
// here a warp that comes twice in a generation is noted.
struct Named {
  int count = 0, generation = 0;
  std::vector<const Task*> who;
  bool twice = false;
  bool arrive(const Task* t, int warps) {  // true: the generation is complete
    for (const Task* w : who) twice |= w == t;
    who.push_back(t);
    if (++count < warps) return false;
    count = 0, ++generation;
    who.clear();
    return true;
  }
};

// Mbarrier: phases completed so far (a phase takes `need` arrivals).
struct Phase {
  int done = 0, count = 0, need = 1;
  void arrive() {
    if (++count == need) count = 0, ++done;
  }
  bool complete(int parity) const { return (done & 1) != parity; }
};

struct Model {
  std::mt19937 rng;
  double fail = 0;                // chance that a wait's time limit passes
  double lose = 0;                // chance that a load never lands
  std::vector<std::unique_ptr<Task>> tasks;
  Task* current = nullptr;
  ucontext_t main_ctx;
  Named named[16];
  std::map<std::string, Phase> bars;
  std::deque<std::vector<std::string>> mma;  // commits, in issue order
  std::vector<std::string> tma;              // loads in flight
  bool abort = false, burst = false, blocking = false, one_ds = false;

  explicit Model(unsigned seed) : rng(seed) {}
  double uniform() { return std::uniform_real_distribution<>(0, 1)(rng); }
  int below(int n) { return (int)(rng() % (unsigned)n); }

  static void entry() {
    M->current->body();
    M->current->done = true;
    swapcontext(&M->current->ctx, &M->main_ctx);
  }
  void spawn(std::function<void()> body) {
    std::unique_ptr<Task> t(new Task());
    t->stack.resize(64 * 1024);
    t->body = std::move(body);
    getcontext(&t->ctx);
    t->ctx.uc_stack.ss_sp = t->stack.data();
    t->ctx.uc_stack.ss_size = t->stack.size();
    t->ctx.uc_link = nullptr;
    makecontext(&t->ctx, entry, 0);
    tasks.push_back(std::move(t));
  }
  void yield(std::function<bool()> ready, bool bounded) {
    Task* t = current;
    t->ready = std::move(ready);
    t->bounded = bounded;
    swapcontext(&t->ctx, &main_ctx);
  }
  void pause() { yield([] { return true; }, false); }

  // ---- what the roles call
  void arrive(int id, int warps) {
    pause();
    named[id].arrive(current, warps);
  }
  void sync(int id, int warps) {
    const int g = named[id].generation;
    if (named[id].arrive(current, warps)) return pause();
    yield([this, id, g] { return named[id].generation != g; }, false);
  }
  // A bounded wait: try, then look at the abort flag, then at the time.
  bool wait(const std::string& name, int parity) {
    Phase* b = &bars[name];
    if (b->complete(parity)) {
      pause();
      return true;
    }
    current->expired = false;
    yield([this, b, parity] { return b->complete(parity) || abort; }, true);
    if (b->complete(parity)) return true;
    abort = true;
    return false;
  }
  // The wait of a role that has failed: deaf to the abort flag.  In the model it
  // has no time limit: the tensor pipe goes on.
  void prove(const std::string& name, int parity) {
    Phase* b = &bars[name];
    if (!burst && !blocking)
      yield([b, parity] { return b->complete(parity); }, false);
  }
  void commit(std::vector<std::string> names) { mma.push_back(std::move(names)); }
  void load(const std::string& name) {
    if (uniform() >= lose) tma.push_back(name);
  }

  // Returns false when stuck, or when a warp arrived twice in a generation.
  bool run() {
    M = this;
    for (;;) {
      std::vector<Task*> can, limited;
      bool all_done = true;
      for (auto& t : tasks) {
        if (t->done) continue;
        all_done = false;
        if (!t->ready || t->ready()) can.push_back(t.get());
        else if (t->bounded) limited.push_back(t.get());
      }
      if (all_done) break;
      if (!mma.empty() && uniform() < 0.4) {
        for (auto& n : mma.front()) bars[n].arrive();
        mma.pop_front();
        continue;
      }
      if (!tma.empty() && uniform() < 0.4) {
        const int i = below((int)tma.size());
        bars[tma[i]].arrive();
        tma.erase(tma.begin() + i);
        continue;
      }
      Task* t = nullptr;
      if (!limited.empty() && fail > 0 && uniform() < fail) {
        t = limited[below((int)limited.size())];  // its time limit has passed
        t->expired = true;
      } else if (!can.empty()) {
        t = can[below((int)can.size())];
      } else if (!mma.empty() || !tma.empty()) {
        continue;
      } else if (!limited.empty()) {
        t = limited[below((int)limited.size())];
        t->expired = true;
      } else {
        return false;
      }
      current = t;
      swapcontext(&main_ctx, &t->ctx);
    }
    for (const Named& n : named)
      if (n.twice || n.count != 0) return false;
    return true;
  }
};

std::string nm(const char* base, int i) { return base + std::to_string(i); }

// An arrival owed after a failed wait.
void owe(Model& m, int id, int warps) {
  if (m.blocking) m.sync(id, warps); else m.arrive(id, warps);
}

// ------------------------------------------------------------------ forward
struct FwdRelay {
  Model& m;
  bool ok = true;
  bool wait_k(int j) {
    return ok = m.wait(nm("kf", j % kFwdKStages), (j / kFwdKStages) & 1);
  }
  bool wait_v(int j) {
    return ok = m.wait(nm("vf", j % kFwdVStages), (j / kFwdVStages) & 1);
  }
  void wait_k_slot(int j) {
    m.prove(nm("ke", j % kFwdKStages), ((j / kFwdKStages) & 1) ^ 1);
  }
  void wait_v_slot(int j) {
    m.prove(nm("ve", j % kFwdVStages), ((j / kFwdVStages) & 1) ^ 1);
  }
  void arrive(int id) {
    if (ok) m.arrive(id, kRelayWarps); else owe(m, id, kRelayWarps);
  }
};

struct FwdMma {
  Model& m;
  void relay_sync(int id) { m.sync(id, kRelayWarps); }
  void softmax_sync(int id) { m.sync(id, kFwdSoftmaxWarps); }
  void qk(int t, int st, bool last) {
    m.commit({nm("sf", t)});
    if (last) m.commit({nm("ke", st)});
  }
  void pv(int t, int st, bool, bool last) {
    m.commit({nm("pf", t)});
    if (last) m.commit({nm("ve", st)});
  }
};

void forward(Model& m, int n, int tiles, bool own_s, bool stall) {
  m.spawn([&m, n] {
    m.load("qf");
    for (int j = 0; j < n; ++j) {
      if (!m.wait(nm("ke", j % kFwdKStages), ((j / kFwdKStages) & 1) ^ 1)) break;
      m.load(nm("kf", j % kFwdKStages));
    }
  });
  m.spawn([&m, n] {
    for (int j = 0; j < n; ++j) {
      if (!m.wait(nm("ve", j % kFwdVStages), ((j / kFwdVStages) & 1) ^ 1)) break;
      m.load(nm("vf", j % kFwdVStages));
    }
  });
  m.spawn([&m, n] {
    FwdRelay ops{m};
    fwd_relay_steps(n, ops);
  });
  m.spawn([&m, n, tiles, own_s, stall] {
    const bool ok = (!stall || m.wait("of", 0)) && m.wait("qf", 0);
    FwdMma ops{m};
    fwd_mma_steps(n, tiles == 2, own_s, ops);
    if (ok) m.commit({"of"});
  });
  for (int t = 0; t < tiles; ++t)
    for (int w = 0; w < 4; ++w)
      m.spawn([&m, n, t, tiles, own_s] {
        const int total = fwd_s_arrivals(n, t, tiles, own_s);
        int s_done = n, j = 0;
        for (; j < n; ++j) {
          if (!m.wait(nm("sf", t), j & 1)) {
            s_done = j;
            break;
          }
          if (j < total) m.arrive(fwd_s_free(t, own_s), kFwdSoftmaxWarps);
          if (j > 0 && !m.wait(nm("pf", t), (j - 1) & 1)) {
            s_done = j + 1;
            break;
          }
          m.arrive(fwd_p_full(t), kFwdSoftmaxWarps);
        }
        const bool ok = j == n;
        struct Rest {
          Model& m;
          int t;
          void wait_s(int j) { m.prove(nm("sf", t), j & 1); }
          void wait_p(int j) { m.prove(nm("pf", t), j & 1); }
          void arrive(int id) { owe(m, id, kFwdSoftmaxWarps); }
        };
        fwd_softmax_rest(n, t, own_s, total, s_done, j, Rest{m, t});
        if (ok) m.wait("of", 0);
      });
}

// ----------------------------------------------------------------- backward
struct BwdRelay {
  Model& m;
  bool ok = true;
  bool wait(int ring, int j) {
    const int depth = ring ? kBwdStages1 : kBwdStages0;
    return ok = m.wait(nm(ring ? "f1." : "f0.", j % depth), (j / depth) & 1);
  }
  void wait_slot(int ring, int j) {
    const int depth = ring ? kBwdStages1 : kBwdStages0;
    m.prove(nm(ring ? "e1." : "e0.", j % depth), ((j / depth) & 1) ^ 1);
  }
  void arrive(int id) {
    if (ok) m.arrive(id, kRelayWarps); else owe(m, id, kRelayWarps);
  }
};

struct BwdMma {
  Model& m;
  bool dq;
  void relay_sync(int id) { m.sync(id, kRelayWarps); }
  void compute_sync(int id) {
    if (m.one_ds && id == bwd_ds(1, true)) id = bwd_ds(0, true);
    m.sync(id, kBwdComputeWarps);
  }
  void s(int) { m.commit({"s"}); }
  void dp(int j) {
    m.commit({nm("dp", dq ? j & 1 : 0)});
    if (dq) m.commit({nm("e1.", j % kBwdStages1)});
  }
  void dv(int j) { m.commit({nm("e1.", j % kBwdStages1)}); }
  void out(int j) { m.commit({nm("e0.", j % kBwdStages0)}); }
};

void backward(Model& m, int n, bool dq, bool stall) {
  for (int sl = 0; sl < 2; ++sl) m.bars[nm("ve", sl)].need = 8;
  m.spawn([&m, n] {
    m.load("fixed");
    for (int j = 0; j < n; ++j)
      for (int ring = 1; ring >= 0; --ring) {
        const int depth = ring ? kBwdStages1 : kBwdStages0;
        if (!m.wait(nm(ring ? "e1." : "e0.", j % depth), ((j / depth) & 1) ^ 1))
          return;
        m.load(nm(ring ? "f1." : "f0.", j % depth));
      }
  });
  m.spawn([&m, n] {
    BwdRelay ops{m};
    bwd_relay_steps(n, ops);
  });
  if (!dq)
    m.spawn([&m, n] {
      for (int j = 0; j < n; ++j) {
        if (!m.wait(nm("ve", j & 1), ((j >> 1) & 1) ^ 1)) break;
        m.load(nm("vf", j & 1));
      }
    });
  m.spawn([&m, n, dq, stall] {
    const bool ok = (!stall || m.wait("of", 0)) && m.wait("fixed", 0);
    BwdMma ops{m, dq};
    if (dq) dq_mma_steps(n, ops); else dkdv_mma_steps(n, ops);
    if (ok) m.commit({"of"});
  });
  for (int w = 0; w < 8; ++w)
    m.spawn([&m, n, dq] {
      auto id_of = [&m](int id) {
        return m.one_ds && id == bwd_ds(1, true) ? bwd_ds(0, true) : id;
      };
      bool ok = true;
      int p = 0, ds = 0;
      for (int j = 0; j < n; ++j) {
        if (!dq && !(ok = m.wait(nm("vf", j & 1), (j >> 1) & 1))) break;
        if (!(ok = m.wait("s", j & 1))) break;
        m.arrive(kBwdP, kBwdComputeWarps);
        ++p;
        if (!(ok = dq ? m.wait(nm("dp", j & 1), (j >> 1) & 1)
                      : m.wait("dp0", j & 1)))
          break;
        m.arrive(id_of(bwd_ds(j, dq)), kBwdComputeWarps);
        ++ds;
        if (!dq) m.bars[nm("ve", j & 1)].arrive();
      }
      struct Rest {
        Model& m;
        bool dq;
        std::function<int(int)> id_of;
        void wait_s(int j) { m.prove("s", j & 1); }
        void wait_dp(int j) {
          m.prove(dq ? nm("dp", j & 1) : "dp0", (dq ? j >> 1 : j) & 1);
        }
        void arrive(int id) { owe(m, id_of(id), kBwdComputeWarps); }
      };
      bwd_compute_rest(n, dq, p, ds, Rest{m, dq, id_of});
      if (ok) m.wait("of", 0);
    });
}

}  // namespace

int main(int argc, char** argv) {
  if (argc != 4) return 2;
  const std::string kernel = argv[1], protocol = argv[2];
  const int seeds = atoi(argv[3]);
  int failed = 0, stuck = 0;
  for (int seed = 0; seed < seeds; ++seed) {
    Model m(1000003u * (unsigned)seed + 17u);
    const double rates[] = {0, 0.001, 0.01, 0.1};
    m.fail = rates[m.below(4)];
    m.lose = m.below(8) ? 0 : 0.1;
    m.burst = protocol == "burst";
    m.blocking = protocol == "blocking";
    m.one_ds = protocol == "one-ds";
    const int lengths[] = {1, 2, 3, 4, 5, 7, 11, 16};
    const int n = lengths[m.below(8)];
    const bool stall = m.below(8) == 0;
    if (kernel == "fwd64" || kernel == "fwd128")
      forward(m, n, 1 + m.below(2), kernel == "fwd64", stall);
    else
      backward(m, n, kernel == "dq", stall);
    const bool ended = m.run();
    failed += m.abort;
    stuck += !ended;
    if (m.fail == 0 && m.lose == 0 && !stall && m.abort) {  // nothing may fail by itself
      printf("seed %d: a wait failed in a run without failures\n", seed);
      return 1;
    }
  }
  printf("%d %d %d\n", seeds, failed, stuck);
  return 0;
}

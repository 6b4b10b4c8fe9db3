// Every actor of the KVarN streaming decode's ring, one thread each and one of them
// running at a time, in an order drawn at random: the producer that refills stages, a
// landing copy per stage in flight, and the consumer warps with the blocks, head
// segments and barriers of the kernel.  Barriers are waited for by parity, as an
// mbarrier is.  Reports the first read of a stage whose copies have not landed, a
// refill under a reader, or that nothing can go on any more.
// argv: consumer warps, blocks per stage, ring stages, blocks, first head end, seeds,
// rule (0: as the kernel, 1: a warp goes straight to the stage of its next block).
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <mutex>
#include <random>
#include <thread>
#include <vector>

#include "ring_pass.h"

namespace {

int NW, SB, NS, NB, HEAD, RULE;

struct Sim {
  std::mutex mu;
  std::condition_variable cv;
  int turn = -1;                        // the actor that runs
  std::vector<std::function<bool()>> ready;
  std::vector<char> done;
  std::mt19937 rng;
  const char* fault = nullptr;

  std::vector<int> full, empty_count, empty_phase, holds, landed, readers;
  int issued = 0, arrived = 0, generation = 0;

  // picks the next actor; called with mu held
  void pick() {
    std::vector<int> can;
    bool left = false;
    for (size_t i = 0; i < ready.size(); ++i)
      if (!done[i]) {
        left = true;
        if (ready[i]()) can.push_back((int)i);
      }
    if (can.empty() && left && !fault) fault = "nothing can go on";
    turn = can.empty() || fault ? -2 : can[rng() % can.size()];
    cv.notify_all();
  }
  // gives the turn away until `cond` holds and the actor is picked; false: stop
  bool yield(int me, std::function<bool()> cond) {
    std::unique_lock<std::mutex> lk(mu, std::adopt_lock);
    ready[me] = cond;
    pick();
    cv.wait(lk, [&] { return turn == me || turn == -2; });
    lk.release();
    return turn == me;
  }
};

struct Stop {};

bool run(unsigned seed) {
  Sim s;
  s.rng.seed(seed);
  const int nst = (NB + SB - 1) / SB;
  s.full.assign(NS, 0);
  s.empty_count.assign(NS, 0);
  s.empty_phase.assign(NS, 0);
  s.holds.assign(NS, -1);
  s.readers.assign(NS, 0);
  s.landed.assign(nst, 0);
  const int actors = NW + 1 + nst;      // warps, producer, the copies of each stage
  s.ready.assign(actors, [] { return true; });
  s.done.assign(actors, 0);
  const bool skip = RULE == 1;

  auto arrive_empty = [&](int st, int count) {
    if (++s.empty_count[st] == count) {
      s.empty_count[st] = 0;
      ++s.empty_phase[st];
    }
  };
  auto consumer = [&](int me) {
    auto go = [&](std::function<bool()> c) { if (!s.yield(me, c)) throw Stop(); };
    // parity wait: true while the phase in progress has the other parity
    auto wait = [&](int st) {
      go([&, st] { return (s.full[st % NS] & 1) != ((st / NS) & 1); });
      if (!s.landed[st] || s.holds[st % NS] != st) s.fault = "a stage was taken for another phase";
      if (s.fault) throw Stop();
      return true;
    };
    auto leave = [&](int st) { arrive_empty(st % NS, skip ? SB : NW); };
    int next = 0;
    for (int a = 0; a < NB;) {
      const int e = a < HEAD && HEAD < NB ? HEAD : NB;
      for (int j = a + ((me - a) % NW + NW) % NW; j < e; j += NW) {
        const int sj = j / SB;
        if (!skip) kvq::stream::ring_pass(next, sj, wait, leave);
        wait(sj);
        ++s.readers[sj % NS];
        go([] { return true; });
        --s.readers[sj % NS];
        if (s.holds[sj % NS] != sj) s.fault = "a stage was refilled under a reader";
        if (s.fault) throw Stop();
        if (skip) leave(sj);
        else leave(next++);
      }
      if (!skip) kvq::stream::ring_pass(next, (e - 1) / SB, wait, leave);
      // the consumers' barrier
      const int gen = s.generation;
      if (++s.arrived == NW) {
        s.arrived = 0;
        ++s.generation;
      }
      go([&, gen] { return s.generation != gen; });
      a = e;
    }
  };
  auto producer = [&](int me) {
    for (int st = 0; st < nst; ++st) {
      if (!s.yield(me, [&, st] { return st < NS || (s.empty_phase[st % NS] & 1) != ((st / NS - 1) & 1); }))
        throw Stop();
      if (s.readers[st % NS]) s.fault = "a stage was refilled under a reader";
      s.holds[st % NS] = st;
      s.issued = st + 1;
    }
  };
  auto copies = [&](int me) {
    const int st = me - NW - 1;
    if (!s.yield(me, [&, st] { return s.issued > st; })) throw Stop();
    s.landed[st] = 1;
    ++s.full[st % NS];
  };

  std::vector<std::thread> th;
  for (int i = 0; i < actors; ++i)
    th.emplace_back([&, i] {
      std::unique_lock<std::mutex> lk(s.mu);
      s.cv.wait(lk, [&] { return s.turn == i || s.turn == -2; });
      lk.release();
      if (s.turn == i) {
        try {
          if (i < NW) consumer(i);
          else if (i == NW) producer(i);
          else copies(i);
        } catch (Stop&) {
        }
      }
      s.done[i] = 1;
      s.pick();
      s.mu.unlock();
    });
  {
    std::lock_guard<std::mutex> lk(s.mu);
    s.pick();
  }
  for (auto& t : th) t.join();
  if (s.fault) std::printf("seed %u: %s\n", seed, s.fault);
  return s.fault == nullptr;
}

}  // namespace

int main(int argc, char** argv) {
  if (argc < 8) return 2;
  NW = std::atoi(argv[1]); SB = std::atoi(argv[2]); NS = std::atoi(argv[3]); NB = std::atoi(argv[4]);
  HEAD = std::atoi(argv[5]); RULE = std::atoi(argv[7]);
  for (unsigned seed = 0; seed < (unsigned)std::atoi(argv[6]); ++seed)
    if (!run(seed)) return 1;
  return 0;
}

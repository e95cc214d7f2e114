// Host model of a pair of CTAs around the MMA role of attention_pair_sm100.cu.  The role itself is the kernel's source, put in
// ROLE_FILE by tests/test_pair_mma_model.py; everything that it calls is here: barriers with the rules of mbarrier (phases, pending
// arrivals, bytes; a parity test is true while the phase with the other parity is open), and the roles at their other ends, in simulated time.
// Every QK^T and P V that the role issues is checked against what has arrived by then.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <map>
#include <queue>
#include <random>
#include <string>
#include <vector>

// ---------------------------------------------------------------- what the role's source names
#define __device__
#define __forceinline__ inline
#define __align__(x) alignas(x)
#define CP_LIKELY(x) (x)
#define CP_UNLIKELY(x) (x)
struct uint2 { uint32_t x, y; };
struct DeviceStatus {};
struct Unit { int T, nA, nB, cnt; };
constexpr int kTile = 128, kHalfBytes = 128 * 64 * 2;
constexpr int kBadList = -1, kEmptyUnit = -3, kZeroUnit = -4;
template <int NS> struct Args { int n_units; DeviceStatus* st; };
template <bool> struct Idesc2 { static constexpr uint32_t qk = 1, pv = 2; };
struct Bars;
static void fail(const char* what, long n);
static bool mbar_test(unsigned long long* bar, uint32_t parity);
static bool mbar_ready(unsigned long long* bar, uint32_t parity) { return mbar_test(bar, parity); }
static bool wait_slow(unsigned long long* bar, uint32_t parity, Bars*, DeviceStatus*, int site);
static bool wait(unsigned long long* bar, uint32_t parity, Bars* b, DeviceStatus* st, int site) { return wait_slow(bar, parity, b, st, site); }
static void mbar_arrive(unsigned long long* bar);
static void umma2_qk8(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc);
static void umma2_pv8(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc);
static void umma2_ts_second(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc);
static void umma2_commit(unsigned long long* bar);
static void tc_fence_after() {}
static void __syncwarp() {}
template <typename T> static T __shfl_sync(unsigned, T v, int) { return v; }
static bool __any_sync(unsigned, bool v) { return v; }
static uint64_t desc_base(uint32_t) { return 0; }
static uint64_t desc_at(uint64_t, uint32_t addr) { return addr; }

#include ROLE_FILE

// ---------------------------------------------------------------- simulated time and barriers
struct Event { long t; long order; std::function<void()> f; bool operator<(const Event& o) const { return t != o.t ? t > o.t : order > o.order; } };
struct Barrier { int count, pending; long tx, phase; };
static std::priority_queue<Event> events;
static std::map<unsigned long long*, Barrier> barriers;
static long now, n_events;
static std::string scenario;
static std::vector<std::function<bool()>> actors;     // each does what it can without waiting; true if that was anything

static void fail(const char* what, long n) {
  std::printf("%s (tile or unit %ld) at time %ld of: %s\n", what, n, now, scenario.c_str());
  std::exit(1);
}
static void after(long dt, std::function<void()> f) { events.push({now + dt, n_events++, std::move(f)}); }
static void init(unsigned long long* b, int count) { barriers[b] = {count, count, 0, 0}; }
static void settle(Barrier& b) {
  if (b.pending < 0) fail("more arrivals than a phase takes", b.phase);
  if (b.pending == 0 && b.tx == 0) { ++b.phase; b.pending = b.count; }
}
static void arrive(unsigned long long* b, long tx = 0) { Barrier& x = barriers.at(b); x.tx += tx; --x.pending; settle(x); }
static void complete(unsigned long long* b, long tx) { Barrier& x = barriers.at(b); x.tx -= tx; settle(x); }
static bool test(unsigned long long* b, uint32_t parity) { return (uint32_t(barriers.at(b).phase) & 1u) != parity; }
static void run_actors() { for (bool any = true; any;) { any = false; for (auto& f : actors) any = f() || any; } }
static bool next_event() {
  if (events.empty()) return false;
  const Event e = events.top();
  events.pop();
  now = std::max(now, e.t);
  e.f();
  run_actors();
  return true;
}
static void pass(long dt) {                            // the role runs for dt cycles
  const long until = now + dt;
  while (!events.empty() && events.top().t <= until) next_event();
  now = until;
}
static bool mbar_test(unsigned long long* bar, uint32_t parity) { pass(20); return test(bar, parity); }
static bool wait_slow(unsigned long long* bar, uint32_t parity, Bars*, DeviceStatus*, int site) {
  pass(20);
  while (!test(bar, parity)) if (!next_event()) fail("nothing left that could end a wait", site);
  return true;
}
static void mbar_arrive(unsigned long long* bar) { arrive(bar); run_actors(); }

// ---------------------------------------------------------------- the pair around the role
struct Tile { int unit, index; bool last; };
static Bars bars;
static std::vector<Unit> units;                       // as published
static std::vector<int> with_tiles;                   // those that stream tiles
static std::vector<Tile> tiles;                       // of all units
static std::vector<bool> k_there, v_there, p_there, q_there, o_read;
static long qk, pv, pv_second;                        // issued
static long pipe_free;                                // when the tensor cores have done what was issued
constexpr uint32_t kTmem = 0, kBase = 1u << 20;

static void umma2_qk8(uint32_t d, uint64_t a, uint64_t b, uint32_t) {
  pass(120);
  const long g = qk++;
  if (g >= long(tiles.size())) fail("QK^T beyond the last tile", g);
  const int u = tiles[g].unit;
  if (d != kTmem + g % kSlots * 128 || b != uint64_t(kBase + kSmemK + g % kSlots * kSlotBytes) || a != uint64_t(kBase + kSmemQ + u % 2 * kQBytes))
    fail("QK^T with another tile's operands", g);
  if (!q_there[u]) fail("QK^T before its Q has arrived", g);
  if (!k_there[g]) fail("QK^T before its K tile has arrived", g);
  if (pv < g - (kSlots - 1)) fail("QK^T over an S that P V has not consumed", g);
  pipe_free = std::max(pipe_free, now) + 520;
}
static void check_pv(uint32_t d, uint32_t a, uint64_t b) {
  const long g = pv;
  if (g >= qk) fail("P V before its QK^T", g);
  if (d != kTmem + 384 || a != kTmem + g % kSlots * 128 || b != uint64_t(kBase + kSmemV + g % kSlots * kSlotBytes)) fail("P V with another tile's operands", g);
  if (!p_there[g]) fail("P V before its P is there", g);
  if (!v_there[g]) fail("P V before its V tile has arrived", g);
  if (tiles[g].index == 0 && tiles[g].unit > 0 && !o_read[tiles[g].unit - 1]) fail("P V over an O that has not been read", g);
}
static void umma2_pv8(uint32_t d, uint32_t a, uint64_t b, uint32_t, uint32_t acc) {
  pass(120);
  check_pv(d, a, b);
  const Unit& u = units[with_tiles[tiles[pv].unit]];
  if (tiles[pv].last && u.nB > u.nA) fail("P V of both CTAs for the second one's tile", pv);
  if (acc != (tiles[pv].index > 0 ? 1u : 0u)) fail("P V accumulates wrongly", pv);
  ++pv;
  pipe_free = std::max(pipe_free, now) + 520;
}
static void umma2_ts_second(uint32_t d, uint32_t a, uint64_t b, uint32_t) {
  pass(30);
  const uint32_t kk = uint32_t(pv_second++ % 8);
  check_pv(d, a - kk * 8, b - kk * 128);
  const Unit& u = units[with_tiles[tiles[pv].unit]];
  if (!tiles[pv].last || u.nB <= u.nA) fail("P V of the second CTA alone for a tile of both", pv);
  pipe_free = std::max(pipe_free, now) + 65;
  if (kk == 7) ++pv;
}
static void umma2_commit(unsigned long long* bar) {
  pass(20);
  after(std::max(pipe_free - now, 0L) + 100, [bar] { arrive(bar); });
}

static void simulate(const std::vector<Unit>& list, const std::vector<long>& publish, std::mt19937& rng, long load_min, long load_max, long softmax_max) {
  events = {};
  barriers.clear();
  actors.clear();
  bars = Bars{};
  units = list;
  with_tiles.clear();
  tiles.clear();
  now = 0; pipe_free = 0; qk = pv = pv_second = 0;
  for (size_t i = 0; i < units.size(); ++i)
    if (units[i].cnt > 0) {
      for (int j = 0; j < units[i].T; ++j) tiles.push_back({int(with_tiles.size()), j, j == units[i].T - 1});
      with_tiles.push_back(int(i));
    }
  const size_t n_tiles = tiles.size();
  k_there.assign(n_tiles, false); v_there = p_there = k_there;
  q_there.assign(with_tiles.size(), false); o_read = q_there;
  for (int i = 0; i < 2; ++i) { init(&bars.q_full[i], 1); init(&bars.q_empty[i], 1); }
  for (int i = 0; i < kSlots; ++i) {
    init(&bars.k_full[i], 1); init(&bars.v_full[i], 1); init(&bars.s_full[i], 1); init(&bars.p_full[i], 1); init(&bars.v_empty[i], 1);
  }
  init(&bars.o_full, 1);
  init(&bars.o_empty, 1);
  for (int i = 0; i < kSched; ++i) { init(&bars.sched_full[i], 1); init(&bars.sched_empty[i], 2); }   // the MMA warp and the K producer

  // scheduler: unit q is published publish[q] cycles after the K producer has taken the one before
  static long drawn, taken, published;                  // static: the events and actors outlive this scope
  drawn = taken = published = 0;
  actors.push_back([&publish] {
    const long q = drawn;
    if (q > long(units.size()) || q > taken || (q >= kSched && !test(&bars.sched_empty[q % kSched], uint32_t(q / kSched - 1) & 1))) return false;
    ++drawn;
    after(q < long(publish.size()) ? publish[q] : 100, [q] {
      bars.sched_unit[q % kSched] = int(q);                       // the one after the last says that there are none left
      if (q < long(units.size())) bars.sched_u[q % kSched] = units[q];
      ++published;
      arrive(&bars.sched_full[q % kSched]);
    });
    return true;
  });
  // K producer: units in turn; Q when the buffer is free, K tiles when QK^T three tiles back is complete
  auto load = [=, &rng] { return load_min + long(rng() % uint32_t(load_max - load_min + 1)); };
  static long unit_at, tile_at, tile_end;
  unit_at = -1; tile_at = tile_end = 0;
  actors.push_back([load] {
    if (tile_at < tile_end) {
      const long g = tile_at;
      if (g >= kSlots && !test(&bars.s_full[g % kSlots], uint32_t(g / kSlots - 1) & 1)) return false;
      arrive(&bars.k_full[g % kSlots], 1);
      after(load(), [g] { k_there[g] = true; complete(&bars.k_full[g % kSlots], 1); });
      ++tile_at;
      return true;
    }
    if (taken < published && taken < long(units.size())) {
      const Unit& u = units[taken];
      if (u.cnt > 0) {
        const long un = unit_at + 1;
        if (un >= 2 && !test(&bars.q_empty[un % 2], uint32_t(un / 2 - 1) & 1)) return false;
        ++unit_at;
        arrive(&bars.q_full[un % 2], 1);
        after(load(), [un] { q_there[un] = true; complete(&bars.q_full[un % 2], 1); });
        tile_end += u.T;
      }
      arrive(&bars.sched_empty[taken % kSched]);
      ++taken;
      return true;
    }
    return false;
  });
  // V producer (the tiles of the units that the K producer has begun)
  static long v_at;
  v_at = 0;
  actors.push_back([load] {
    const long g = v_at;
    if (g >= tile_end || (g >= kSlots && !test(&bars.v_empty[g % kSlots], uint32_t(g / kSlots - 1) & 1))) return false;
    ++v_at;
    arrive(&bars.v_full[g % kSlots], 1);
    after(load(), [g] { v_there[g] = true; complete(&bars.v_full[g % kSlots], 1); });
    return true;
  });
  // softmax: tile after tile
  static long s_at;
  s_at = 0;
  actors.push_back([=, &rng] {
    const long g = s_at;
    if (g >= long(n_tiles) || !test(&bars.s_full[g % kSlots], uint32_t(g / kSlots) & 1)) return false;
    ++s_at;
    after(200 + long(rng() % uint32_t(softmax_max)), [g] { p_there[g] = true; arrive(&bars.p_full[g % kSlots]); });
    return true;
  });
  // epilogue
  static long o_at;
  o_at = 0;
  actors.push_back([=, &rng] {
    const long u = o_at;
    if (u >= long(with_tiles.size()) || !test(&bars.o_full, uint32_t(u) & 1)) return false;
    ++o_at;
    after(300 + long(rng() % 1500u), [u] { o_read[u] = true; arrive(&bars.o_empty); });
    return true;
  });

  run_actors();
  Args<1> args{int(units.size()), nullptr};
  mma_role<false, 1>(args, &bars, kBase, 0);
  if (qk != long(n_tiles) || pv != long(n_tiles)) fail("tiles left out", pv);
}

static Unit unit_of(int T, bool second) {              // T = 0: an empty list; -1: a list that breaks its contract
  if (T <= 0) return Unit{0, 0, 0, T == 0 ? kZeroUnit : kBadList};
  return Unit{T, second ? T - 1 : T, T, 1};
}

int main(int argc, char** argv) {
  const long n_random = argc > 1 ? std::atol(argv[1]) : 1000;
  std::mt19937 rng(1);
  auto run = [&](const std::vector<int>& T, const std::vector<long>& publish, long load_min, long load_max, long softmax_max, bool second) {
    scenario = "tiles";
    for (int x : T) scenario += " " + std::to_string(x);
    scenario += ", published after";
    for (long x : publish) scenario += " " + std::to_string(x);
    std::vector<Unit> list;
    for (int x : T) list.push_back(unit_of(x, second && x > 1));
    simulate(list, publish, rng, load_min, load_max, softmax_max);
  };
  // a unit that is published when the one before has nearly or wholly run out, K tiles that come later than P
  for (int first : {1, 2, 3, 4, 5, 8})
    for (int then : {1, 2, 3, 4, 5, 8, 9})
      for (long late : {100L, 3000L, 6000L, 9000L, 12000L, 15000L, 20000L, 40000L})
        for (long load : {500L, 3000L, 20000L}) run({first, then, 4}, {0, late, late}, load, load, 800, (first + then) % 2 == 0);
  // empty and broken lists, which cost a hand-over each
  for (int zeros = 1; zeros < 6; ++zeros)
    for (long each : {1000L, 3500L, 6000L}) {
      std::vector<int> T{8};
      for (int i = 0; i < zeros; ++i) T.push_back(i % 2 ? -1 : 0);
      T.push_back(8);
      run(T, std::vector<long>(T.size(), each), 4000, 9000, 1500, true);
    }
  for (long i = 0; i < n_random; ++i) {
    const int lengths[] = {-1, 0, 0, 1, 1, 2, 3, 4, 5, 6, 8, 12};
    std::vector<int> T(1 + rng() % 12);
    std::vector<long> publish;
    for (int& x : T) { x = lengths[rng() % 12]; publish.push_back(long(rng() % (rng() % 2 ? 3000u : 20000u))); }
    const long load_min = 200 + long(rng() % 2000), load_max = load_min + long(rng() % 12000);
    run(T, publish, load_min, load_max, 300 + long(rng() % 4000), rng() % 2);
  }
  std::printf("ok\n");
  return 0;
}

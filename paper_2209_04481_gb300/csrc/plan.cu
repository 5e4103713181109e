// plan.cu -- radial planes per CTA of the tiled residual.
//
// A CTA costs a preamble and then its planes.  What the launch takes depends
// on how the CTAs fall on the SMs, so the launch of every candidate chunk is
// simulated: CTAs start in launch order (all tiles of chunk 0, then chunk 1,
// ...) on the first free slot, the first `nsm` of them on SMs of their own.
// Measured on 152 SMs with 152 x {1, 2} CTAs of 256 FP32 or 128 FP64 threads, norms
// included:
//   * two CTAs on one SM take 4.8 us per plane where one takes 2.7 (FP32), 74
//     where one takes 42 (FP64): two CTAs run at 0.57 of the rate of one;
//   * the preamble (first loads, the redundant r face at the chunk's start, and
//     the closing reduction) takes about 1.5 planes in FP32 and 0.5 in FP64,
//     and since it is latency it does not slow down beside another CTA.
// What it picks against a sweep of 1 to 16 planes (R alone, van Albada).  FP32, the
// fastest on each: 14 planes on 128 x 64 x 128 (61.5 us; 7: 65.4, 12: 81.9, 16: 68.3),
// 6 on 95 x 45 x 88 (30.8 us; 5: 39.0, 12: 39.0), 2 on 64 x 32 x 64 (16.4 us; 4: 18.6),
// 1 on 32 x 16 x 32 (12.4 us; 4: 18.5).  FP64, within 3 % of the fastest: 9 on
// 128 x 64 x 128 (1.53 ms; 7: 1.58, 12: 1.68, 16: 1.79), 12 on 95 x 45 x 88 (0.71 ms;
// 6: 0.69, 9: 0.86), 1 on 32 x 16 x 32 (60 us; 4: 172).
#include <algorithm>
#include <queue>
#include <vector>

#include "corona_internal.h"

namespace crn {
namespace {

constexpr double kSharedRate = 0.57;
constexpr double kPreamble32 = 1.5, kPreamble64 = 0.5;  // in planes
// more CTAs per slot than this leave no imbalance to trade for their preambles
constexpr long long kMaxWaves = 6;

struct Cta {
  double pre = 0.0, work = 0.0;
  bool live = false;
};
struct Sm {
  double now = 0.0;
  Cta c[2];
  double rate(int q) const {
    if (c[q].pre > 0.0) return 1.0;
    const Cta& o = c[1 - q];
    return o.live && !(o.pre > 0.0) ? kSharedRate : 1.0;
  }
  // time to the next change of state; < 0 if idle
  double step() const {
    double best = -1.0;
    for (int q = 0; q < 2; ++q) {
      if (!c[q].live) continue;
      const double t = (c[q].pre > 0.0 ? c[q].pre : c[q].work) / rate(q);
      if (best < 0.0 || t < best) best = t;
    }
    return best;
  }
};

// run time of the launch in planes, or a value above `give_up`
double simulate(int nr, long long ntiles, int nsm, int per_sm, int kc, double pre, double give_up) {
  const long long nch = (nr + kc - 1) / kc, total = nch * ntiles;
  const long long last = (nch - 1) * ntiles;
  const double rem = (double)(nr - (nch - 1) * kc);
  long long next = 0;
  auto take = [&](Cta& c) {
    c.live = next < total;
    if (!c.live) return;
    c.pre = pre;
    c.work = next >= last ? rem : (double)kc;
    ++next;
  };
  std::vector<Sm> sm((size_t)nsm);
  for (int q = 0; q < per_sm; ++q)
    for (Sm& s : sm) take(s.c[q]);
  using Event = std::pair<double, int>;
  std::priority_queue<Event, std::vector<Event>, std::greater<Event>> ev;
  for (int i = 0; i < nsm; ++i)
    if (sm[i].step() >= 0.0) ev.push({sm[i].step(), i});
  double end = 0.0;
  while (!ev.empty()) {
    const Event e = ev.top();
    ev.pop();
    Sm& s = sm[e.second];
    const double dt = e.first - s.now;
    const double r[2] = {s.rate(0), s.rate(1)};
    s.now = e.first;
    for (int q = 0; q < 2; ++q) {
      Cta& c = s.c[q];
      if (!c.live) continue;
      if (c.pre > 0.0) {
        c.pre -= dt;
        if (c.pre < 1e-9) c.pre = 0.0;
      } else {
        c.work -= dt * r[q];
        if (c.work < 1e-9) {
          end = std::max(end, e.first);
          if (end > give_up) return end;
          take(c);
        }
      }
    }
    const double t = s.step();
    if (t >= 0.0) ev.push({s.now + t, e.second});
  }
  return end;
}

}  // namespace

int choose_radial_chunk(int nr, long long ntiles, int nsm, int per_sm, bool fp64) {
  if (ntiles <= 0 || nsm <= 0) return nr;
  per_sm = std::max(1, std::min(per_sm, 2));
  int best = nr;
  double best_t = 1e300;
  for (int kc = nr; kc >= 1; --kc) {
    const long long total = (long long)((nr + kc - 1) / kc) * ntiles;
    if (kc < nr && total > kMaxWaves * nsm * per_sm) break;
    const double t = simulate(nr, ntiles, nsm, per_sm, kc, fp64 ? kPreamble64 : kPreamble32, best_t);
    if (t < best_t - 1e-9) {
      best_t = t;
      best = kc;
    }
  }
  return best;
}

}  // namespace crn

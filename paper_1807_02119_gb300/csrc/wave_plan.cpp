// Level schedule of a step list (the forward plan's steps or the reverse program's).
//
// A contraction tree of a few hundred steps is only 10 to 35 levels deep, so most steps
// can run at the same time; one after another they are bound by launch and memory latency.
// The schedule works in rounds: first every light step (a small row step) that can run
// without a heavy result, level by level, then the heavy steps that are ready, each its own
// launch.  Consecutive levels that a cluster of CTAs can hold become one launch with a
// cluster barrier between levels (k_waves); a wider level is one launch over the GPU
// (k_wave_wide).  Every step computes exactly what it computes alone.
//
// Memory: tensors are placed by first fit over their lifetimes in schedule units (a level,
// or a heavy step), so tensors used in the same level never overlap.
#include <algorithm>
#include <cstring>
#include <numeric>

#include "pk_internal.h"

namespace pk {
namespace {

struct Interval {
  int64_t off, len;
};

uint64_t align256(uint64_t x) { return (x + 255) & ~uint64_t(255); }

bool overlap(const Interval& x, const Interval& y) {
  return x.off < y.off + y.len && y.off < x.off + x.len;
}

// log2 of the lanes that share one output's sum over k: at most kWaveK terms per lane (one
// round trip for their operands) while the step has few lanes, 16 (8 of a longer sum) while
// they stay within what the GPU holds at once.
int lanes_log2(int64_t outs, int64_t K) {
  int l = 0;
  while (l < 5 && (((K >> l) > kWaveK && (outs << (l + 1)) <= (1 << 13)) ||
                   ((K >> l) > (K > 16 ? 8 : 16) && (outs << (l + 1)) <= (1 << 18))))
    ++l;
  return l;
}

uint32_t push_record(const Step& s, const std::vector<int64_t>& off, std::vector<uint8_t>& blob, int lanes,
                     uint32_t per = 1) {
  WaveRec r;
  std::memset(&r, 0, sizeof(r));
  r.a = s.a;
  r.b = s.b;
  r.c = s.c;
  r.R = (uint32_t)s.R;
  r.N = (uint32_t)s.N;
  r.K = (uint32_t)s.K;
  r.mul_r = div_mul(s.R, s.R * s.N);
  r.nrow = (uint8_t)s.nrow;
  r.nk = (uint8_t)s.nk;
  r.nn = (uint8_t)s.nn;
  r.lanes = (uint8_t)lanes;
  r.off_a = off[s.a];
  r.off_b = s.b >= 0 ? off[s.b] : 0;
  r.off_c = off[s.c];
  r.per = per;
  const size_t at = blob.size();
  blob.resize(at + sizeof(WaveRec) + sizeof(WaveRun) * (size_t)(s.nrow + s.nk + s.nn));
  std::memcpy(blob.data() + at, &r, sizeof(r));
  WaveRun* w = (WaveRun*)(blob.data() + at + sizeof(WaveRec));
  auto put = [&](const Run* v, int n, int64_t top) {
    for (int i = 0; i < n; ++i, ++w)
      *w = {(uint32_t)v[i].size, div_mul(v[i].size, top), (uint32_t)v[i].sa, (uint32_t)v[i].sb};
  };
  put(s.row, s.nrow, s.R);
  put(s.kr, s.nk, s.K);
  put(s.nr, s.nn, s.N);
  return (uint32_t)(at / 16);
}

}  // namespace

int64_t first_fit(const std::vector<int64_t>& elems, const std::vector<int32_t>& born,
                  const std::vector<int32_t>& dies, std::vector<int64_t>& off) {
  const int32_t n = (int32_t)elems.size();
  std::vector<int32_t> ord(n);
  std::iota(ord.begin(), ord.end(), 0);
  std::sort(ord.begin(), ord.end(), [&](int32_t x, int32_t y) {
    return elems[x] != elems[y] ? elems[x] > elems[y] : x < y;
  });
  struct Placed {
    int64_t off, end;
    int32_t born, dies;
  };
  std::vector<Placed> placed;   // by offset
  off.assign(n, 0);
  int64_t top = 0;
  for (int32_t t : ord) {
    const int64_t len = (elems[t] + 63) / 64 * 64;
    int64_t at = 0;
    for (const Placed& p : placed) {
      if (p.dies < born[t] || dies[t] < p.born) continue;
      if (at + len <= p.off) break;
      at = std::max(at, p.end);
    }
    off[t] = at;
    const Placed mine{at, at + len, born[t], dies[t]};
    placed.insert(std::upper_bound(placed.begin(), placed.end(), mine,
                                   [](const Placed& x, const Placed& y) { return x.off < y.off; }),
                  mine);
    top = std::max(top, at + len);
  }
  return top;
}

bool wave_light(const Step& s, const pk_tuning& tune) {
  // the top of pk_tuning's ranges leaves K and the outputs to the level kernels' own limits
  if (s.kernel != KROWS || s.K > (tune.seq_k == 2048 ? kWaveOuts : tune.seq_k)) return false;
  const int64_t outs = s.R * s.N, work = outs * s.K;
  if (outs > (tune.seq_outs == 65536 ? kWaveOuts : tune.seq_outs)) return false;
  // K > 32: more work than that still runs better here, where lanes share a sum, than on the
  // thread-per-output kernel (the row kernel's registers hold 32 terms)
  if (work > (s.K > 32 ? 16 * tune.seq_work : tune.seq_work)) return false;
  // the kernels' divisions y / d as umulhi(y, ceil(2^32 / d)) are exact while y d < 2^32
  if (s.N > 1 && outs * s.R >= ((int64_t)1 << 32)) return false;
  auto exact = [](const Run* r, int n) {
    int64_t y = 1, d = 1;
    for (int i = 0; i < n; ++i) {
      y *= r[i].size;
      if (i + 1 < n) d = std::max(d, r[i].size);
    }
    return y * d < ((int64_t)1 << 32);
  };
  return exact(s.row, s.nrow) && exact(s.kr, s.nk) && exact(s.nr, s.nn);
}

void wave_schedule(const std::vector<Step>& steps, int32_t n_tens, const pk_tuning& tune, int32_t heavy,
                   bool breadth, const std::vector<std::pair<int32_t, int32_t>>* extra, int32_t first_tail,
                   std::vector<WaveUnit>& units) {
  const int32_t n = (int32_t)steps.size();
  units.clear();
  std::vector<int32_t> prod(n_tens, -1), need(n, 0);
  std::vector<std::vector<int32_t>> next(n);
  for (int32_t i = 0; i < n; ++i) prod[steps[i].c] = i;
  auto edge = [&](int32_t from, int32_t to) {
    next[from].push_back(to);
    ++need[to];
  };
  for (int32_t i = 0; i < n; ++i) {
    if (prod[steps[i].a] >= 0) edge(prod[steps[i].a], i);
    if (steps[i].b >= 0 && prod[steps[i].b] >= 0) edge(prod[steps[i].b], i);
  }
  if (extra)
    for (const auto& e : *extra) edge(e.first, e.second);
  // steps from first_tail on come last, one after another
  for (int32_t i = 0; i < first_tail && first_tail < n; ++i) edge(i, first_tail);
  for (int32_t i = first_tail + 1; i < n; ++i) edge(i - 1, i);
  std::vector<char> light(n);
  std::vector<int32_t> ready_l, ready_h;
  auto add = [&](int32_t i) { (light[i] ? ready_l : ready_h).push_back(i); };
  for (int32_t i = 0; i < n; ++i) light[i] = i < first_tail && wave_light(steps[i], tune) && !((heavy & kHeavyTc64) && tc64_step(steps[i])) &&
               !((heavy & kHeavyTc) && steps[i].tc);
  for (int32_t i = 0; i < n; ++i)
    if (need[i] == 0) add(i);
  auto finish = [&](int32_t i) {
    for (int32_t j : next[i])
      if (--need[j] == 0) add(j);
  };
  while (!ready_l.empty() || !ready_h.empty()) {
    while (!ready_l.empty()) {
      std::vector<int32_t> lev;
      lev.swap(ready_l);
      std::sort(lev.begin(), lev.end());
      for (int32_t i : lev) finish(i);
      units.push_back({false, std::move(lev)});
    }
    std::vector<int32_t> hs;
    hs.swap(ready_h);
    std::sort(hs.begin(), hs.end());
    if (!breadth && hs.size() > 1) {
      ready_h.assign(hs.begin() + 1, hs.end());
      hs.resize(1);
    }
    for (int32_t i : hs) {
      units.push_back({true, {i}});
      finish(i);
    }
  }
}

int64_t wave_layout(const std::vector<Step>& steps, const std::vector<int64_t>& elems,
                    const std::vector<char>& pinned, const std::vector<WaveUnit>& units,
                    std::vector<int64_t>& off) {
  const int32_t n_tens = (int32_t)elems.size();
  std::vector<int32_t> born(n_tens, -1), dies(n_tens, -1);
  for (int32_t u = 0; u < (int32_t)units.size(); ++u)
    for (int32_t i : units[u].steps) {
      born[steps[i].c] = u;
      dies[steps[i].c] = std::max(dies[steps[i].c], u);
      dies[steps[i].a] = std::max(dies[steps[i].a], u);
      if (steps[i].b >= 0) dies[steps[i].b] = std::max(dies[steps[i].b], u);
    }
  for (int32_t t = 0; t < n_tens; ++t)
    if (pinned[t]) dies[t] = (int32_t)units.size();
  return first_fit(elems, born, dies, off);
}

void wave_hazards(const std::vector<Step>& steps, const std::vector<int64_t>& elems,
                  const std::vector<int64_t>& off, std::vector<std::pair<int32_t, int32_t>>& edges) {
  edges.clear();
  const int32_t n = (int32_t)steps.size();
  auto iv = [&](int32_t t) { return Interval{off[t], elems[t]}; };
  for (int32_t j = 0; j < n; ++j) {
    const Interval w = iv(steps[j].c);
    for (int32_t i = 0; i < j; ++i) {
      const Step& s = steps[i];
      // j overwrites what i reads or wrote, or reads where i wrote later than its operand
      bool hit = overlap(w, iv(s.a)) || (s.b >= 0 && overlap(w, iv(s.b))) || overlap(w, iv(s.c));
      if (!hit && steps[j].a != s.c) hit = overlap(iv(s.c), iv(steps[j].a));
      if (!hit && steps[j].b >= 0 && steps[j].b != s.c) hit = overlap(iv(s.c), iv(steps[j].b));
      if (hit) edges.push_back({i, j});
    }
  }
}

bool wave_check(const std::vector<Step>& steps, const std::vector<int64_t>& elems,
                const std::vector<char>& pinned, const WaveProgram& w, std::string& err) {
  // replay of the units over the arena: every step reads what its producer wrote, no step of
  // a unit writes where another step of the unit reads or writes
  const int32_t n_tens = (int32_t)elems.size();
  std::vector<int32_t> when(n_tens, -1);   // unit that wrote the tensor (initial: -1)
  std::vector<char> init(n_tens, 1), alive(n_tens, 0), done(steps.size(), 0);
  for (const Step& s : steps) init[s.c] = 0;
  for (int32_t t = 0; t < n_tens; ++t) {
    if (w.off[t] < 0 || w.off[t] + elems[t] > w.arena_elems || w.off[t] % 64 != 0) {
      err = "level schedule: tensor " + std::to_string(t) + " outside the arena";
      return false;
    }
    alive[t] = init[t];
  }
  auto hits = [&](int32_t x, int32_t y) {
    return overlap({w.off[x], elems[x]}, {w.off[y], elems[y]});
  };
  std::vector<int32_t> written;
  for (int32_t t = 0; t < n_tens; ++t)
    if (init[t]) written.push_back(t);
  for (size_t i = 0; i < written.size(); ++i)
    for (size_t j = 0; j < i; ++j)
      if (hits(written[i], written[j]) && elems[written[i]] > 0) {
        err = "level schedule: initial tensors overlap";
        return false;
      }
  for (int32_t u = 0; u < (int32_t)w.units.size(); ++u) {
    const std::vector<int32_t>& us = w.units[u].steps;
    for (int32_t i : us) {
      const Step& s = steps[i];
      for (int32_t t : {s.a, s.b})
        if (t >= 0 && (!alive[t] || (!init[t] && when[t] >= u))) {
          err = "level schedule: step " + std::to_string(i) + " reads a tensor that is not there";
          return false;
        }
      for (int32_t j : us) {
        const Step& o = steps[j];
        if (hits(s.c, o.a) || (o.b >= 0 && hits(s.c, o.b)) || (i != j && hits(s.c, o.c))) {
          err = "level schedule: step " + std::to_string(i) + " writes what step " + std::to_string(j) +
                " of its level uses";
          return false;
        }
      }
    }
    for (int32_t i : us) {   // results end the tensors they overwrite
      for (int32_t t : written)
        if (alive[t] && hits(steps[i].c, t)) alive[t] = 0;
      done[i]++;
      when[steps[i].c] = u;
    }
    for (int32_t i : us) {
      alive[steps[i].c] = 1;
      written.push_back(steps[i].c);
    }
  }
  for (size_t i = 0; i < steps.size(); ++i)
    if (done[i] != 1) {
      err = "level schedule: step " + std::to_string(i) + " not run exactly once";
      return false;
    }
  for (int32_t t = 0; t < n_tens; ++t)
    if (pinned[t] && !alive[t]) {
      err = "level schedule: result tensor " + std::to_string(t) + " overwritten";
      return false;
    }
  for (const auto& stages : w.stages) {   // stages cover the units in order
    size_t u = 0;
    for (const WaveStage& st : stages)
      for (int32_t i = 0; i < st.units; ++i, ++u)
        if (u >= w.units.size() || (!w.units[u].heavy && st.kind == WaveStage::STEP)) {
          err = "level schedule: stages do not cover the units";
          return false;
        }
    if (u != w.units.size()) {
      err = "level schedule: stages do not cover the units";
      return false;
    }
  }
  return true;
}

void wave_stages(const std::vector<Step>& steps, const pk_tuning& tune, int32_t heavy, bool shared, WaveProgram& w) {
  // records, items and level table of all levels in order
  std::vector<uint8_t> recs;
  std::vector<WaveItem> items;
  const size_t nu = w.units.size();
  std::vector<uint32_t> lev(nu + 1, 0), rec_at(nu + 1, 0);   // first item / record byte of a unit
  std::vector<int64_t> weight(nu, 0);   // a unit's items, weighed by their terms per lane
  for (size_t u = 0; u < nu; ++u) {
    lev[u] = (uint32_t)items.size();
    rec_at[u] = (uint32_t)recs.size();
    const Step& s0 = steps[w.units[u].steps[0]];
    if (w.units[u].heavy && (!wave_light(s0, tune) || ((heavy & kHeavyTc) && s0.tc))) continue;
    for (int32_t i : w.units[u].steps) {
      const int64_t outs = steps[i].R * steps[i].N;
      const int lg = shared ? lanes_log2(outs, steps[i].K) : 0;
      const uint32_t at = push_record(steps[i], w.off, recs, lg);
      const int64_t lanes = outs << lg;
      for (int64_t c = 0; c * 32 < lanes; ++c) items.push_back({at, (uint32_t)c});
      weight[u] += (lanes + 31) / 32 * std::max<int64_t>(4, steps[i].K / (lanes / outs));
    }
  }
  lev[nu] = (uint32_t)items.size();
  rec_at[nu] = (uint32_t)recs.size();
  auto put = [&](const void* src, size_t n) {   // 16-byte aligned
    const size_t at = w.blob.size();
    w.blob.resize((at + n + 15) / 16 * 16, 0);
    if (n) std::memcpy(w.blob.data() + at, src, n);
    return (uint32_t)at;
  };
  if (items.size() % 2) items.push_back({0, 0});   // a stage's items end on 16 bytes
  w.blob.clear();
  put(recs.data(), recs.size());
  const uint32_t item_at = put(items.data(), sizeof(WaveItem) * items.size());
  const uint32_t lev_at = put(lev.data(), 4 * lev.size());
  w.init_off = w.blob.size();
  put(w.off.data(), 8 * (size_t)w.n_init);
  for (int fp64 = 0; fp64 < 2; ++fp64) {
    // A level costs the cluster a barrier (0.3 us) and the GPU-wide launch about 0.9 us.  FP64
    // runs at 2 multiply-adds per cycle and multiprocessor, 16 cycles per warp instruction, so
    // its levels spread over more multiprocessors, and leave the cluster, sooner.
    const int64_t per_cta = fp64 ? kWaveCtaWarps64 : kWaveCtaWarps32;
    const int64_t fused_max = kWaveMaxCtas * per_cta;
    std::vector<WaveStage>& out = w.stages[fp64];
    out.clear();
    w.n_fused[fp64] = w.n_fused_steps[fp64] = 0;
    for (size_t u = 0; u < nu;) {
      WaveStage st;
      st.step = w.units[u].steps[0];
      st.units = 1;
      if (w.units[u].heavy && (fp64 || lev[u] == lev[u + 1])) {
        st.kind = WaveStage::STEP;
        out.push_back(st);
        ++u;
        continue;
      }
      auto load = [&](size_t x) { return (weight[x] + 3) / 4; };   // in items of four terms
      int64_t most = load(u);
      size_t v = u + 1;
      st.kind = most > fused_max || w.units[u].heavy ? WaveStage::WIDE : WaveStage::FUSED;
      if (st.kind == WaveStage::FUSED)
        for (; v < nu && !w.units[v].heavy && load(v) <= fused_max; ++v) most = std::max<int64_t>(most, load(v));
      st.units = (int32_t)(v - u);
      st.items = (int32_t)(lev[v] - lev[u]);
      while (st.ctas < kWaveMaxCtas && most > st.ctas * per_cta) st.ctas *= 2;
      for (size_t x = u; x < v; ++x)
        st.steps.insert(st.steps.end(), w.units[x].steps.begin(), w.units[x].steps.end());
      const uint32_t i0 = lev[u] & ~1u, l0 = (uint32_t)u & ~3u;   // 16-byte aligned starts
      st.range.rec = rec_at[u];
      st.range.rec_bytes = rec_at[v] - rec_at[u];
      st.range.item = item_at + (uint32_t)sizeof(WaveItem) * i0;
      st.range.item_bytes = ((lev[v] - i0) * (uint32_t)sizeof(WaveItem) + 15) / 16 * 16;
      st.range.item0 = i0;
      st.first = lev[u] - i0;
      st.range.lev = lev_at + 4 * l0;
      st.range.lev_bytes = ((uint32_t)(v + 1 - l0) * 4 + 15) / 16 * 16;
      st.range.lev0 = (uint32_t)u - l0;
      if (st.steps.size() > 1) {
        w.n_fused[fp64] += 1;
        w.n_fused_steps[fp64] += (int32_t)st.steps.size();
      }
      out.push_back(st);
      u = v;
    }
  }
}

int32_t wave_batch(const Plan& p, bool shared, std::vector<uint8_t>& blob, WaveRange& range) {
  std::vector<WaveItem> items;
  std::vector<uint32_t> lev;
  blob.clear();
  range = WaveRange{};
  const WaveProgram& w = p.wave[PK_C64];   // no step of it is kept apart for the tensor cores
  for (const WaveUnit& u : w.units) {
    lev.push_back((uint32_t)items.size());
    for (int32_t i : u.steps) {
      const Step& s = p.steps[i];
      const int64_t outs = s.R * s.N;
      const int lg = shared ? lanes_log2(outs, s.K) : 0;
      const int64_t lanes = outs << lg;
      const int64_t per = std::max<int64_t>(1, (lanes + 65535) / 65536);   // at most 2048 items a step
      const uint32_t at = push_record(s, w.off, blob, lg, (uint32_t)per);
      for (int64_t c = 0; c * 32 * per < lanes; ++c) items.push_back({at, (uint32_t)c});
    }
  }
  lev.push_back((uint32_t)items.size());
  auto put = [&](const void* src, size_t n, uint32_t& at, uint32_t& len) {
    at = (uint32_t)blob.size();
    len = (uint32_t)((n + 15) / 16 * 16);
    blob.resize(at + len, 0);
    if (n) std::memcpy(blob.data() + at, src, n);
  };
  range.rec_bytes = (uint32_t)blob.size();
  put(items.data(), sizeof(WaveItem) * items.size(), range.item, range.item_bytes);
  put(lev.data(), 4 * lev.size(), range.lev, range.lev_bytes);
  return (int32_t)w.units.size();
}

void plan_waves(Plan& p, bool compact, bool one) {
  const int32_t n = (int32_t)p.tensors.size(), ns = (int32_t)p.steps.size();
  std::vector<int64_t> elems(n);
  std::vector<char> pinned(n, 0);
  for (int32_t t = 0; t < n; ++t) elems[t] = p.tensors[t].elems;
  pinned[p.final_tensor] = 1;
  p.tc64_bytes = 0;
  for (const Step& s : p.steps)
    if (p.use_tc64 && !compact && tc64_step(s))
      p.tc64_bytes = std::max<int64_t>(p.tc64_bytes, tc64_scratch(s.Bsz, s.M, s.N, s.K).bytes);
  const int32_t tail = p.conv.empty() && p.tail.empty() ? ns : p.tail_first;
  int64_t limit = p.arena_elems;   // twice that up to 1 GiB, a quarter more up to 16 GiB
  if (limit <= (1 << 25))
    limit = 2 * limit + (1 << 12);
  else if (limit <= (1 << 30) / 5 * 4)
    limit += limit / 4;
  for (int32_t prec : {PK_C128, PK_C64, PK_SPLIT}) {
    WaveProgram& w = p.wave[prec];
    w = WaveProgram();
    w.n_init = p.n_init;
    const int32_t heavy = prec == PK_SPLIT ? kHeavyTc : prec == PK_C128 && p.tc64_bytes > 0 ? kHeavyTc64 : 0;
    // breadth first over the heavy steps has the fewest rounds; one heavy step at a time needs
    // about the memory of the steps' own order.  The widening records of a complex128 tail
    // address the steps' own offsets, so such plans keep them, and so do plans that must stay
    // within a memory limit: their schedule follows the offsets' reuse.
    for (int breadth = 1; breadth >= 0 && !compact && tail == ns; --breadth) {
      wave_schedule(p.steps, n, p.tuning, heavy, breadth != 0, nullptr, ns, w.units);
      w.arena_elems = wave_layout(p.steps, elems, pinned, w.units, w.off);
      if (w.arena_elems <= limit) break;
      w.off.clear();
    }
    if (w.off.empty()) {
      for (int32_t t = 0; t < n; ++t) w.off.push_back(p.tensors[t].offset);
      w.arena_elems = p.arena_elems;
      std::vector<std::pair<int32_t, int32_t>> edges;
      wave_hazards(p.steps, elems, w.off, edges);
      wave_schedule(p.steps, n, p.tuning, heavy, false, &edges, tail, w.units);
    }
    // complex64 sums keep the steps' own order, a lane each (wave.cuh); the exact residues, whose
    // sums do not depend on it, share them on the same units and offsets
    if (prec == PK_C64) {
      p.wave[kWaveExact] = w;
      wave_stages(p.steps, p.tuning, heavy, true, p.wave[kWaveExact]);
    }
    wave_stages(p.steps, p.tuning, heavy, prec != PK_C64, w);
  }
  // workspace: [recipes | slots | conv | every schedule's level records] uploaded, then the
  // device's own state.  A launch in any precision after any upload finds its own records;
  // schedules with equal ones (as a rule those of small plans) share them.
  uint64_t off = p.off_wave[0];
  for (int i = 0; i < 4; ++i) {
    int same = 0;
    while (same < i && p.wave[same].blob != p.wave[i].blob) ++same;
    p.off_wave[i] = one ? p.off_wave[0] : same < i ? p.off_wave[same] : off;
    off = align256(std::max<uint64_t>(off, p.off_wave[i] + p.wave[i].blob.size()));
  }
  p.off_records = off;
  p.off_meta = off;
  off = align256(off + 16ull * p.n_meta);
  p.off_counter = off;
  off = align256(off + 4ull * std::max<int32_t>(1, ns));
  p.off_result = off;
  off = align256(off + 32ull * (uint64_t)p.n_slices + 32);
  p.off_scratch = off;
  off = align256(off + 16ull * (uint64_t)std::max<int64_t>(1, p.splitk_partials));
  p.off_arena = off;
  p.off_tail = align256(p.off_arena + 8ull * (uint64_t)p.ws_elems());
}

}  // namespace pk

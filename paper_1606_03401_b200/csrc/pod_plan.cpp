// Host side of the pod kernel: sizes, and the schedule of phases with the operand slots worked out.
#include <algorithm>
#include <cstring>
#include <unordered_map>

#include "pod.hpp"

namespace mebptt {
namespace pod {

namespace {
inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
inline int up_to(int v, int m) { return (v + m - 1) / m * m; }
inline int slices(int k) { return ceil_div(k, 128); }   // FMA: a warp takes 128 elements of the contraction index at a time
}  // namespace

size_t packed_elems(const Config& c, int l) { return (size_t)c.T * 4 * c.U * c.pitch_w(l); }
size_t packed_readout_elems(const Config& c) { return (size_t)c.T * c.op * c.pitch_r(); }

// The pod size and the batch rows per pod with the least estimated time.  Rows are cheap until the
// arithmetic of a phase shows beside its fixed part, CTAs until the pushes to all of them do; pods
// that do not fit the device at once take turns.  The tensor cores want their weights in shared memory;
// the FMA path can read them from the L2, which then bounds it.
Config choose_config(const Layout& y, const team::DeviceFacts& dev) {
  Config best;
  const int esz = (int)y.esz;
  if (y.L > kMaxLayers || (y.dtype == MEBPTT_BF16 && !y.tensor_cores)) return best;
  // a thread's offsets from the start of the stages (dz, h, dy, carried dz) and of a step of x have 32 bits (a rule on the descriptor:
  // how much a plan keeps must not choose the kernel, and with it the order of sums)
  const int64_t bh = (int64_t)y.B * y.H, steps = std::max(walked_chunk_steps(y.B, y.t), 2);
  if ((y.L * (steps + 4) * bh * 20 + (int64_t)steps * y.B * y.O * 4) >> 32 || ((int64_t)y.B * y.I) >> 31) return best;
  for (int lt = 0; lt <= 4; ++lt)
    for (int nb = 1; nb <= 8; nb *= 2) {
      Config c;
      c.T = 1 << lt; c.nb = nb; c.pods = ceil_div(y.B, nb);
      const int fit = std::min(dev.clusters[lt], dev.sms >> lt);
      if (fit < 1 || c.T > y.H || (nb > 1 && nb >= 2 * y.B)) continue;
      c.mma = y.dtype == MEBPTT_BF16;
      c.planes = 3;
      c.U = ceil_div(y.H, c.T); c.up = up_to(c.U, 4);
      c.kx = up_to(y.I, c.mma ? 16 : 4); c.kh = up_to(c.T * c.up, c.mma ? 32 : 4);
      c.rows_o = ceil_div(y.O, c.T); c.op = up_to(c.rows_o, 4);
      c.extra = c.mma ? 8 : 0;
      if (y.L * c.up * nb > kThreads || c.op * nb > kThreads || ceil_div(ceil_div(y.I, 4), c.T) * nb > kThreads) continue;
      int64_t weights = (int64_t)c.op * c.pitch_r() * esz;
      for (int l = 0; l < y.L; ++l) weights += (int64_t)4 * c.U * c.pitch_w(l) * esz;
      // parts of the contractions
      const int ng = ceil_div(c.U, 8);
      // a power of two; a piece of work has a fixed part, so none is cut below 8 steps of the tensor cores
      auto parts = [&](int groups, int steps) {
        int n = 1;
        while (2 * n <= (c.mma ? steps / 8 : steps) && 2 * n * groups <= kWarps) n *= 2;
        return n;
      };
      for (int l = 0; l < y.L; ++l)
        c.ns_f[l] = c.mma ? parts(ng, (kin(c, l) + c.kh) / 16) : parts(c.U, slices(kin(c, l)) + slices(c.kh));
      c.ns_r = c.mma ? parts(ceil_div(c.op, 16), c.kh / 16) : parts(c.op / 4, slices(c.kh));
      c.ns_b = c.mma ? 1 : c.kh <= kThreads / 4 ? 4 : c.kh <= kThreads / 2 ? 2 : 1;
      auto lg = [](int v) { int n = 0; while (1 << n < v) ++n; return n; };
      c.lg_f0 = lg(c.ns_f[0]); c.lg_f1 = y.L > 1 ? lg(c.ns_f[1]) : 0; c.lg_r = lg(c.ns_r); c.lg_b = lg(c.ns_b);
      c.works_f0 = (c.mma ? ng : c.U) << c.lg_f0; c.works_f1 = (c.mma ? ng : c.U) << c.lg_f1; c.works_r = ceil_div(c.op, c.mma ? 16 : 4) << c.lg_r;
      // the operand area
      c.pitch_x = c.mma ? (c.kx + 8) * 2 : c.kx * 4;
      c.pitch_h = c.mma ? (c.kh + 8) * 2 : c.kh * 4;
      c.x_slot = up_to(nb * c.pitch_x, 16); c.h_slot = up_to(nb * c.pitch_h, 16);
      int at = 0;
      auto take = [&](int64_t bytes) { const int r = at; at += (int)std::min<int64_t>((bytes + 15) & ~15ll, 1 << 26); return r; };
      take((int64_t)kXSlots * c.x_slot);
      c.at_h = take((int64_t)y.L * kHSlots * c.h_slot);
      c.p_slot = up_to(c.T * c.ns_b * c.U * nb * 4, 16);
      c.at_p = take((int64_t)4 * y.L * c.p_slot);
      c.dz_pitch = (up_to(4 * c.U, 16) + 8) * 2; c.dy_pitch = (up_to(c.op, 16) + 8) * 2;
      c.dz_buf = c.mma ? c.planes * nb * c.dz_pitch : 4 * c.U * nb * 4;
      c.dy_buf = c.mma ? c.planes * nb * c.dy_pitch : c.op * nb * 4;
      c.dz_buf = up_to(c.dz_buf, 16); c.dy_buf = up_to(c.dy_buf, 16);
      c.at_dz = take((int64_t)2 * y.L * c.dz_buf);
      c.at_dy = take((int64_t)2 * c.dy_buf);
      int64_t red = c.mma ? (int64_t)ceil_div(c.op, 16) * 16 * c.ns_r * nb * 4 : (int64_t)c.op * c.ns_r * nb * 4;
      for (int l = 0; l < y.L; ++l) red += c.red_f(l);
      c.red_bytes = (int)std::min<int64_t>((red + 15) & ~15ll, 1 << 26);
      c.at_red = take((int64_t)2 * c.red_bytes);
      c.at_dummy = take(64);
      c.at_map = take((int64_t)c.kh * 8);
      if (at / 16 >= kNone) continue;
      c.at_w = at;
      const int fixed = kWindows * kWindow * (int)sizeof(Task) + 1024;
      const int64_t left = team::kSmemMax - fixed - at;
      if (left < 0) continue;
      c.resident = weights <= left;
      if (c.mma && !c.resident) continue;
      c.smem = fixed + at + (c.resident ? (int)weights : 0);
      const int waves = ceil_div(c.pods, fit);
      const double active = (double)std::min(c.pods, fit) * c.T;
      // (fitted to a scan of T and nb over four problems: a phase's fixed part is some 4500 cycles, whatever it does)
      double cyc_f = 0, cyc_b = 0;
      for (int l = 0; l < y.L; ++l) {
        const int kk = kin(c, l) + c.kh, nc = l ? kk : c.kh;
        if (c.mma) {
          cyc_f += ceil_div(ng * c.ns_f[l], kWarps) * (ceil_div(kk / 16, c.ns_f[l]) * 45.0 + 400.0);
          cyc_b += ceil_div(nc / 32, kWarps) * (ceil_div(4 * c.U, 16) * c.planes * 45.0 + 600.0);
        } else {
          const int its = slices(kin(c, l)) + slices(c.kh);
          double f = std::max(1.2 * c.U * its * (4.0 * nb + 16.0), ceil_div(c.U * c.ns_f[l], kWarps) * (ceil_div(its, c.ns_f[l]) * 120.0 + 300.0));
          double b = ceil_div(nc * c.ns_b, kThreads) * (double)ceil_div(4 * c.U, c.ns_b) * std::max(16.0, (3.0 + nb) * kWarps / 4) + 400.0;
          if (!c.resident) {
            const double bf = 4.0 * c.U * kk * esz, bb = 4.0 * c.U * nc * esz;
            f = std::max(f, std::max(bf / 40.0, bf * active / 5000.0));
            b = std::max(b, std::max(bb / 40.0, bb * active / 5000.0));
          }
          cyc_f += f * (1.0 + 0.17 * nb); cyc_b += b * (1.0 + 0.17 * nb);
        }
      }
      c.cycles = waves * (3 * (4400.0 + 20.0 * c.T) + 2 * cyc_f + cyc_b);
      c.ok = true;
      if (!best.ok || c.cycles < best.cycles) best = c;
    }
  return best;
}

namespace {

struct Item {                    // a task before its slots are known
  Task t;
  int64_t in = 0, out = 0;       // versions of the states it reads and writes (0: the caller's, else 1 + index of the operation)
};
using Key = int64_t;             // an operand vector: x_k, or h of a layer in some version
inline bool has_products(const Task& t) { return t.kind == FWD || t.kind == READ || t.kind == BWD || t.kind == DHA || t.kind == CARRY; }
inline Key key_x(int64_t k) { return k << 8 | 255; }
inline Key key_h(int l, int64_t version) { return version << 8 | l; }

struct Slot { Key key = -1; int read = -9, pushed = -9; };

struct Builder {
  const Layout& y;
  const Config& c;
  Schedule& s;

  // ---- phases: each task in the earliest one after everything it depends on ----
  std::vector<std::vector<Item>> open;
  std::vector<uint32_t> taken;             // classes in a phase: bit l its F or B, 16 R, 17 D
  int64_t base = 0, top = -1, n_open = 0;
  std::vector<int64_t> cell, named, state, version, b_phase, d_phase;   // phases of B(l, k) at [l][k & 3], of D(k) at [k & 3]
  int core = 0;

  Builder(const Layout& y_, const Config& c_, Schedule& s_)
      : y(y_), c(c_), s(s_), cell((size_t)y_.arena_units, -1), named((size_t)4 * y_.L, -1),
        state((size_t)(y_.arena_units + 5) * y_.L, -1), version((size_t)y_.arena_units + 5, 0), b_phase((size_t)4 * y_.L, -1),
        d_phase(4, -1) {
  }
  size_t slot_of(int32_t loc) const {
    return loc >= 0 ? (size_t)loc + 5
                    : loc == MEBPTT_LOC_INIT ? 0 : loc == MEBPTT_LOC_PING ? 1 : loc == MEBPTT_LOC_PONG ? 2 : 3 + (size_t)core;
  }
  uint32_t address(int32_t loc) const {
    switch (loc) {
      case MEBPTT_LOC_INIT: return (uint32_t)y.blk_init;
      case MEBPTT_LOC_PING: return (uint32_t)y.blk_ping;
      case MEBPTT_LOC_PONG: return (uint32_t)y.blk_pong;
      case MEBPTT_LOC_CORE: return (uint32_t)y.blk_core[core];
      default: return (uint32_t)loc * (uint32_t)y.loc_blocks;
    }
  }
  int units(int32_t loc, int fmt) const {
    if (loc < 0) return 1;
    const int blocks = fmt == MEBPTT_FMT_HIDDEN ? y.unit_blocks : y.unit_blocks + 4 * y.L + (fmt == MEBPTT_FMT_INTERNAL ? y.unit_blocks : 0);
    return (blocks * y.parts + y.loc_blocks - 1) / y.loc_blocks;
  }
  template <class F> void cells(int32_t loc, int n, int l, F f) {
    if (loc >= 0) { for (int i = 0; i < n && (size_t)(loc + i) < cell.size(); ++i) f(cell[(size_t)(loc + i)]); }
    else if (loc != MEBPTT_LOC_INIT) f(named[(slot_of(loc) - 1) * (size_t)y.L + (size_t)l]);
  }
  int64_t last_touch(int32_t loc, int n, int l) {
    int64_t p = -1;
    cells(loc, n, l, [&](int64_t& v) { p = std::max(p, v); });
    return p;
  }
  void touch(int32_t loc, int n, int l, int64_t phase) {
    cells(loc, n, l, [&](int64_t& v) { v = std::max(v, phase); });
  }
  int64_t place(const Item& it, int64_t after) {
    const uint32_t bit = 1u << (it.t.kind == READ ? 16 : it.t.kind == DHA ? 17 : it.t.layer);
    int64_t p = std::max(after + 1, base);
    for (;; ++p) {
      const size_t i = (size_t)(p - base);
      if (i >= open.size()) { open.resize(i + 1); taken.resize(i + 1, 0); }
      if (taken[i] & bit) continue;
      taken[i] |= bit;
      open[i].push_back(it);
      break;
    }
    top = std::max(top, p);
    ++n_open;
    return p;
  }
  void forward(const mebptt_op& op, int64_t index) {
    const uint32_t src = address(op.src);
    const size_t si = slot_of(op.src);
    if (op.dst == MEBPTT_LOC_CORE) core ^= 1;   // (never the source as well: a valid tape does not read what it writes)
    const size_t so = slot_of(op.dst);
    const int n = units(op.dst, op.dst_fmt), n_src = units(op.src, MEBPTT_FMT_HIDDEN);
    const int64_t arena_free = op.dst >= 0 ? last_touch(op.dst, n, 0) : -1, from = version[si];
    int64_t below = -1, last = -1;
    for (int l = 0; l < y.L; ++l) {
      Item it;
      it.t = Task{};
      it.t.kind = FWD; it.t.layer = (uint8_t)l; it.t.k = (int32_t)op.k; it.t.src = src; it.t.dst = address(op.dst);
      if (op.dst_fmt != MEBPTT_FMT_HIDDEN) it.t.flags |= GATES;
      if (op.dst_fmt == MEBPTT_FMT_INTERNAL) it.t.flags |= COPY_IN;
      if (l == 0) it.t.flags |= COUNT;
      it.in = from; it.out = index + 1;
      const int64_t free_at = op.dst >= 0 ? arena_free : last_touch(op.dst, n, l);
      const int64_t p = place(it, std::max(std::max(state[si * y.L + l], below), free_at));
      state[so * y.L + l] = p;
      below = p;
      last = std::max(last, p);
      if (op.dst < 0) touch(op.dst, n, l, p);
      if (op.dst < 0 && l > 0) touch(op.dst, n, l - 1, p);
      if (op.src < 0) touch(op.src, n_src, l, p);
    }
    version[so] = index + 1;
    if (op.dst >= 0) touch(op.dst, n, 0, last);
    if (op.src >= 0) touch(op.src, n_src, 0, last);
  }
  void backward(const mebptt_op& op) {
    const int sidx = (int)((op.k - 1) % y.S), q = (int)(op.k & 3), L = y.L;
    const size_t si = slot_of(op.src);
    Item r;
    r.t = Task{};
    r.t.kind = READ; r.t.layer = (uint8_t)(L - 1); r.t.k = (int32_t)op.k; r.t.sidx = (uint16_t)sidx; r.t.src = address(op.src);
    r.in = version[si];
    // dy takes the place of dy_{k+2}; its shares that of the ones the top layer used at step k + 2
    const int64_t pr = place(r, std::max(state[si * L + L - 1], d_phase[(size_t)((q + 2) & 3)]));
    Item dh;
    dh.t = r.t;
    dh.t.kind = DHA;
    int64_t above = place(dh, std::max(pr, b_phase[(size_t)(L - 1) * 4 + ((q + 2) & 3)])), last = above;
    d_phase[(size_t)q] = above;
    for (int l = L - 1; l >= 0; --l) {
      Item b;
      b.t = Task{};
      b.t.kind = BWD; b.t.layer = (uint8_t)l; b.t.k = (int32_t)op.k; b.t.sidx = (uint16_t)sidx; b.t.src = address(op.src);
      int64_t after = std::max(std::max(state[si * L + l], above), b_phase[(size_t)l * 4 + ((q + 1) & 3)]);
      // its shares for the layer below take the place of those of step k + 2
      if (l > 0) after = std::max(after, b_phase[(size_t)(l - 1) * 4 + ((q + 2) & 3)]);
      if (op.dst_fmt == MEBPTT_FMT_INTERNAL) {
        b.t.dst = b.t.src + (uint32_t)((y.unit_blocks + 4 * y.L) * y.parts);
      } else {
        b.t.dst = address(op.aux);
        after = std::max(after, state[slot_of(op.aux) * L + l]);
      }
      if (op.k == y.t) b.t.flags |= FIRST;
      if (op.k == y.t || sidx == y.S - 1) b.t.flags |= OPEN;
      if (sidx == 0) b.t.flags |= CLOSE;
      if (l == L - 1) b.t.flags |= COUNT;
      const int64_t p = place(b, after);
      b_phase[(size_t)l * 4 + q] = p;
      above = p;
      last = std::max(last, p);
    }
    for (int l = 0; l < (op.src < 0 ? L : 1); ++l) touch(op.src, units(op.src, op.dst_fmt), l, last);
    if (op.dst_fmt != MEBPTT_FMT_INTERNAL)
      for (int l = 0; l < (op.aux < 0 ? L : 1); ++l) touch(op.aux, units(op.aux, MEBPTT_FMT_HIDDEN), l, last);
  }

  // ---- slots: phase by phase, loads put into the phase before the one that needs them ----
  struct Pools { std::vector<Slot> x, h; };   // h: [L][kHSlots]
  std::unordered_map<Key, std::vector<int>> uses;
  int64_t next_use(Key k, int phase) const {   // first use after `phase`; far away: none
    const auto it = uses.find(k);
    if (it == uses.end()) return (int64_t)1 << 40;
    const auto u = std::upper_bound(it->second.begin(), it->second.end(), phase);
    return u == it->second.end() ? (int64_t)1 << 40 : *u;
  }
  // A slot of the pool that can be pushed to in emitted phase e and is not needed in phase `cur` itself:
  // the one whose content is needed last.
  int victim(const Slot* pool, int n, int e, int cur, int phase) const {
    int best = -1;
    int64_t far = -1;
    for (int i = 0; i < n; ++i) {
      if (pool[i].read >= e || pool[i].pushed >= e || pool[i].read == cur) continue;
      const int64_t u = pool[i].key < 0 ? (int64_t)1 << 41 : next_use(pool[i].key, phase);
      if (u > far) { far = u; best = i; }
    }
    return best;
  }
  static int find(const Slot* pool, int n, Key k) {
    for (int i = 0; i < n; ++i) if (pool[i].key == k) return i;
    return -1;
  }
  static uint16_t u16(int bytes) { return (uint16_t)(bytes / 16); }

  void close(int chunk) {
    uses.clear();
    for (size_t p = 0; p < open.size(); ++p)
      for (const Item& it : open[p]) {
        const Task& t = it.t;
        if (t.kind == FWD) {
          uses[t.layer == 0 ? key_x(t.k) : key_h(t.layer - 1, it.out)].push_back((int)p);
          uses[key_h(t.layer, it.in)].push_back((int)p);
        } else if (t.kind == READ) {
          uses[key_h(t.layer, it.in)].push_back((int)p);
        }
      }
    std::vector<std::vector<Task>> out;
    // the launch's first backward operations lack the shares of the step after: from its carried dz
    {
      std::vector<Task> z;
      uint32_t seen = 0;
      for (const std::vector<Item>& ph : open)
        for (const Item& it : ph)
          if (it.t.kind == BWD && !(seen >> it.t.layer & 1)) {
            seen |= 1u << it.t.layer;
            if (it.t.flags & FIRST) continue;
            Task t = it.t;
            t.kind = CARRY; t.flags = 0;
            t.sidx = (it.t.flags & OPEN) ? kNone : (uint16_t)(it.t.sidx + 1);   // the stage still holds a step of the same chunk
            z.push_back(t);
          }
      if (!z.empty()) out.push_back(z);
    }
    Pools pools;
    pools.x.resize(kXSlots);
    pools.h.resize((size_t)y.L * kHSlots);
    for (size_t p = 0; p < open.size(); ++p) {
      std::vector<Item> rest(open[p]);
      while (!rest.empty()) {
        const int e = (int)out.size();                          // the phase being put together
        Pools q = pools;
        std::vector<Task> now, loads;
        std::vector<Item> later;
        bool gap = false;                                       // a phase of loads has to come first
        auto loaded = [&](const Task& l) {                      // its class is taken in the phase before
          auto same = [&](const Task& o) { return o.kind == l.kind && (l.kind == LOAD_X || o.layer == l.layer); };
          for (const Task& o : out.back()) if (same(o)) return true;
          for (const Task& o : loads) if (same(o)) return true;
          return out.back().size() + loads.size() >= (size_t)kPhaseTasks;
        };
        auto operand = [&](Slot* pool, int n, Key key, const Task& load, int slot0, int bytes, int& at) {
          int i = find(pool, n, key);
          if (i < 0) {
            i = e > 0 && !loaded(load) ? victim(pool, n, e - 1, e, (int)p - 1) : -1;
            if (i < 0) { gap = true; return; }
            Task l = load;
            l.so = u16(slot0 + i * bytes);
            loads.push_back(l);
            pool[i].key = key;
            pool[i].pushed = e - 1;
          }
          pool[i].read = e;
          at = slot0 + i * bytes;
        };
        for (size_t j = 0; j < rest.size() && !gap; ++j) {
          const Item& it = rest[j];
          Task t = it.t;
          const int l = t.layer;
          Slot* hl = q.h.data() + (size_t)l * kHSlots;
          int a = -1, b = -1;
          Task load{};
          load.layer = (uint8_t)l;
          if (t.kind == FWD && l == 0) {
            load.kind = LOAD_X; load.k = t.k;
            operand(q.x.data(), kXSlots, key_x(t.k), load, c.slot_x(0), c.x_slot, a);
          } else if (t.kind == FWD) {
            load.kind = LOAD_H; load.layer = (uint8_t)(l - 1); load.src = t.dst;
            operand(hl - kHSlots, kHSlots, key_h(l - 1, it.out), load, c.slot_h(l - 1, 0), c.h_slot, a);
            load.layer = (uint8_t)l;
          }
          if (gap) break;
          if (t.kind == FWD || t.kind == READ) {
            load.kind = LOAD_H; load.src = t.src;
            operand(hl, kHSlots, key_h(l, it.in), load, c.slot_h(l, 0), c.h_slot, b);
            if (gap) break;
          }
          t.sa = a < 0 ? kNone : u16(a);
          t.sb = b < 0 ? kNone : u16(b);
          now.push_back(t);
          later.push_back(it);
        }
        if (gap) {                                              // what was found room for stays
          if (!loads.empty()) {
            out.back().insert(out.back().end(), loads.begin(), loads.end());
            pools = q;
          }
          out.emplace_back();
          continue;
        }
        // results, once it is known what the phase reads; a task whose result finds no room waits for another phase
        std::vector<Item> wait;
        std::vector<Task> done;
        for (size_t j = 0; j < now.size(); ++j) {
          Task& t = now[j];
          const Item& it = later[j];
          const int l = t.layer;
          t.so = kNone;
          if (t.kind == FWD) {
            const Key key = key_h(l, it.out);
            if (next_use(key, (int)p) < (int64_t)1 << 40) {
              const int i = victim(q.h.data() + (size_t)l * kHSlots, kHSlots, e, e, (int)p);
              if (i < 0) { wait.push_back(it); continue; }
              Slot& sl = q.h[(size_t)l * kHSlots + (size_t)i];
              sl.key = key; sl.pushed = e;
              t.so = u16(c.slot_h(l, i));
            }
          }
          done.push_back(t);
        }
        if (done.empty()) { out.emplace_back(); continue; }     // every slot was read or written just now: a phase of nothing in between
        if (!loads.empty()) out.back().insert(out.back().end(), loads.begin(), loads.end());
        out.push_back(done);
        pools = q;
        rest = wait;
      }
    }
    team::Launch g;
    g.task0 = s.tasks.size();
    auto pad = [&] { while (s.tasks.size() % kWindow) s.tasks.push_back(Task{}); };
    for (std::vector<Task>& ph : out) {
      if (ph.empty()) ph.push_back(Task{});                     // keeps its place as an empty phase
      std::stable_sort(ph.begin(), ph.end(), [](const Task& u, const Task& v) { return has_products(u) > has_products(v); });
      Header h{};
      h.n = (uint8_t)ph.size();
      int rot = 0;
      for (size_t i = 0; i < ph.size(); ++i) {
        Task& t = ph[i];
        if (t.flags & COUNT) ++(t.kind == FWD ? g.fwd_ops : g.bwd_ops);
        const int l = t.layer, L = y.L;
        const uint32_t at = (uint32_t)(i + 1), nib = at << (4 * l);
        h.products += has_products(t);
        t.rot = (uint8_t)(rot & (kWarps - 1));
        switch (t.kind) {
          case FWD: {
            h.main |= nib; h.sums = 1; h.n_h += t.so != kNone;
            int red = c.at_red;
            for (int j = 0; j < l; ++j) red += c.red_f(j);
            t.red = u16(red); t.w = (uint32_t)c.w_at(l);
            rot += (c.mma ? ceil_div(c.U, 8) : c.U) * (l ? c.ns_f[1] : c.ns_f[0]);
            break;
          }
          case READ: {
            h.r = (uint8_t)at; h.sums = 1;
            int red = c.at_red;
            for (int j = 0; j < L; ++j) red += c.red_f(j);
            t.red = u16(red); t.w = (uint32_t)c.w_at(L); t.so = u16(c.at_dy + (t.k & 1) * c.dy_buf);
            rot += ceil_div(c.op, c.mma ? 16 : 4) * c.ns_r;
            break;
          }
          case BWD: {
            const bool own = !(t.flags & CLOSE), below = l > 0;
            h.main |= nib; h.bwd |= nib; h.cells = 1; h.n_p += own + below;
            t.sa = u16(c.share_slot(l, 0, t.k & 1)); t.sb = u16(c.share_slot(l, 1, t.k & 1));
            t.so = u16(c.share_slot(l, 0, (t.k - 1) & 1));
            t.red = below ? u16(c.share_slot(l - 1, 1, t.k & 1)) : t.so;
            t.w = (uint32_t)(c.w_at(l) + (below ? 0 : kin(c, l)));
            t.cols = (uint16_t)((own + below) * c.kh);
            rot += t.cols / 32;
            break;
          }
          case CARRY:
            h.carry |= nib; h.cells = 1; ++h.n_p;
            t.so = t.red = u16(c.share_slot(l, 0, t.k & 1));
            t.w = (uint32_t)(c.w_at(l) + kin(c, l));
            t.cols = (uint16_t)c.kh;
            rot += t.cols / 32;
            break;
          case DHA:   // (dy was left by other threads: the barrier before the products)
            h.cells = 1; ++h.n_p;
            t.sa = u16(c.at_dy + (t.k & 1) * c.dy_buf); t.so = t.red = u16(c.share_slot(L - 1, 1, t.k & 1));
            t.w = (uint32_t)c.w_at(L);
            t.cols = (uint16_t)c.kh;
            rot += t.cols / 32;
            break;
          case LOAD_H: h.load |= nib; ++h.n_h; break;
          case LOAD_X: h.x = (uint8_t)at; ++h.n_x; break;
          default: break;
        }
      }
      if (s.tasks.size() % kWindow + ph.size() + 1 > (size_t)kWindow) pad();
      Task rec;
      memcpy(&rec, &h, sizeof rec);
      s.tasks.push_back(rec);
      s.tasks.insert(s.tasks.end(), ph.begin(), ph.end());
      ++g.phases;
    }
    pad();
    g.ntasks = s.tasks.size() - g.task0;
    g.chunk = chunk;
    s.launches.push_back(g);
    open.clear();
    taken.clear();
    n_open = 0;
    base = top + 1;
  }
};

}  // namespace

// A launch ends with its chunk, or when as many tasks are open as leave room for the records they become:
// with headers, loads and padding up to seven times as many (0.99 of that over some thousand problems), and
// where it is more, launches of fewer tasks.
void build_schedule(const Layout& y, const Plan* p, const Config& c, size_t room, Schedule& s) {
  for (int64_t most = (int64_t)team::kMaxLaunchTasks / 7;; most = std::min<int64_t>(most / 2, (int64_t)room / 8)) {
    s = Schedule{};
    Builder w(y, c, s);
    int64_t index = 0;
    for (const mebptt_op& op : p->tape) {
      if (op.kind == MEBPTT_OP_FWD) {
        w.forward(op, index);
      } else {
        w.backward(op);
        if ((op.k - 1) % y.S == 0) w.close((int)((op.k - 1) / y.S));
      }
      ++index;
      if (w.n_open > most) w.close(-1);
    }
    size_t largest = 0;
    for (const team::Launch& g : s.launches) largest = std::max(largest, g.ntasks);
    if (largest <= room || most == 0) return;
  }
}

}  // namespace pod
}  // namespace mebptt

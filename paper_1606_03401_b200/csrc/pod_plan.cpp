// Host side of the pod kernel: sizes, and the schedule of phases with the operand slots worked out.
#include <algorithm>
#include <unordered_map>

#include "pod.hpp"

namespace mebptt {
namespace pod {

namespace {
inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
inline int pad16(int v) { return (v + 15) & ~15; }
inline int slices(int k) { return ceil_div(k, 128); }
}  // namespace

int slot_x(const Config& c, int i) { return i * c.x_slot; }
int slot_h(const Layout& y, const Config& c, int l, int i) { (void)y; return kXSlots * c.x_slot + (l * kHSlots + i) * c.h_slot; }
int slot_dz(const Layout& y, const Config& c, int l, int i) {
  return kXSlots * c.x_slot + y.L * kHSlots * c.h_slot + (l * kDzSlots + i) * c.dz_slot;
}
int slot_dy(const Layout& y, const Config& c, int i) {
  return kXSlots * c.x_slot + y.L * (kHSlots * c.h_slot + kDzSlots * c.dz_slot) + i * c.dy_slot;
}

// The pod size and the batch rows per pod with the least estimated time.  Rows are cheap until the
// arithmetic of a phase shows beside its fixed part, CTAs until the pushes to all of them do; pods
// that do not fit the device at once take turns.
Config choose_config(const Layout& y, int sms, const int* max_clusters) {
  const team::Dims d = team::dims(y);
  Config best;
  for (int lt = 0; lt <= 4; ++lt)
    for (int nb = 1; nb <= 8; nb *= 2) {
      Config c;
      c.T = 1 << lt; c.nb = nb; c.pods = ceil_div(y.B, nb);
      const int fit = std::min(max_clusters[lt], sms >> lt);
      if (fit < 1 || c.T > y.H) continue;
      const int u = ceil_div(y.H, c.T), gb = ceil_div(u, 4), gr = ceil_div(d.groups_o, c.T), esz = (int)y.esz;
      auto parts = [](int groups, int its) { return std::max(1, std::min(its, kWarps / std::max(1, groups))); };
      c.x_slot = pad16(nb * d.ip[0]); c.h_slot = pad16(nb * d.hp); c.dz_slot = pad16(nb * d.gp); c.dy_slot = pad16(nb * ((y.O + 7) & ~7));
      c.slot_floats = kXSlots * c.x_slot + y.L * (kHSlots * c.h_slot + kDzSlots * c.dz_slot) + kDySlots * c.dy_slot;
      if (c.slot_floats / 16 >= kNone) continue;
      c.ns_r = parts(gr, slices(d.hp));
      int sum_f = 0, sum_b = 0, most = gr * c.ns_r;
      double cyc_f = 0, cyc_b = 0;
      int64_t bytes_f[team::kMaxLayers], bytes_b[team::kMaxLayers], bytes_r = (int64_t)gr * 4 * d.hp * esz, all = bytes_r;
      for (int l = 0; l < y.L; ++l) {
        const int its_f = slices(d.ip[l]) + slices(d.hp), its_b = slices(d.gp) + slices(d.kb[l] - d.gp);
        c.ns_f[l] = parts(u, its_f); c.ns_b[l] = parts(gb, its_b);
        sum_f += u * c.ns_f[l]; sum_b += gb * c.ns_b[l];
        most = std::max(most, std::max(u * c.ns_f[l], gb * c.ns_b[l]));
        bytes_f[l] = (int64_t)u * 4 * d.kf[l] * esz; bytes_b[l] = (int64_t)gb * 4 * d.kb[l] * esz;
        all += bytes_f[l] + bytes_b[l];
      }
      // room for a phase of the wavefront over all layers in both directions, with the readout
      c.red_floats = std::max(most, sum_f + sum_b + gr * c.ns_r) * nb * 4;
      const int fixed = kWindows * kWindow * (int)sizeof(Task) + 2048;
      int64_t left = team::kSmemMax - fixed - ((int64_t)c.slot_floats + 2 * c.red_floats) * 4;
      if (left < 0) continue;
      int64_t held = 0;
      auto keep = [&](int bit, int64_t bytes) {
        if (bytes <= left) { c.resident |= 1ull << bit; left -= bytes; held += bytes; }
      };
      for (int l = 0; l < y.L; ++l) keep(2 * l, bytes_f[l]);
      for (int l = 0; l < y.L; ++l) keep(2 * l + 1, bytes_b[l]);
      keep(63, bytes_r);
      c.smem = fixed + (c.slot_floats + 2 * c.red_floats) * 4 + (int)held;
      const int waves = ceil_div(c.pods, fit);
      const double active = (double)std::min(c.pods, fit) * c.T;
      auto cycles = [&](int groups, int its, int k, int ns, bool res) {
        const double through = (double)groups * its * (4.0 * nb + 4.0 * esz);
        const double chain = (double)ceil_div(groups * ns, kWarps) * (ceil_div(its, ns) * 70.0 + 100.0);
        double t = std::max(through, chain);
        if (!res) {
          const double bytes = (double)groups * 4 * k * esz;
          t = std::max(t, std::max(bytes / 40.0, bytes * active / 2500.0));
        }
        return t;
      };
      for (int l = 0; l < y.L; ++l) {
        cyc_f += cycles(u, slices(d.ip[l]) + slices(d.hp), d.kf[l], c.ns_f[l], c.resident >> (2 * l) & 1);
        cyc_b += cycles(gb, slices(d.gp) + slices(d.kb[l] - d.gp), d.kb[l], c.ns_b[l], c.resident >> (2 * l + 1) & 1);
      }
      const double push = 25.0 * c.T;   // what a thread spends on sending a value to every CTA
      c.cycles = waves * (3 * (1100.0 + (c.T > 1 ? 300.0 : 0.0) + push) + 2 * cyc_f + cyc_b +
                          cycles(gr, slices(d.hp), d.hp, c.ns_r, c.resident >> 63 & 1));
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
inline Key key_x(int64_t k) { return k << 8 | 255; }
inline Key key_h(int l, int64_t version) { return version << 8 | l; }

struct Slot { Key key = -1; int read = -9, pushed = -9; };

struct Builder {
  const Layout& y;
  const Config& c;
  const team::Dims d;
  Schedule& s;

  // ---- phases: each task in the earliest one after everything it depends on ----
  std::vector<std::vector<Item>> open;
  std::vector<int> red;
  int64_t base = 0, top = -1, n_open = 0;
  std::vector<int64_t> cell, named, state, version, b_phase;   // b_phase: [L][4], phase of B(l, k) at k & 3
  int core = 0;
  uint32_t at_ping, at_pong, at_core[2], at_arena, loc_step;

  Builder(const Layout& y_, const Config& c_, Schedule& s_)
      : y(y_), c(c_), d(team::dims(y_)), s(s_), cell((size_t)y_.arena_units, -1), named((size_t)4 * y_.L, -1),
        state((size_t)(y_.arena_units + 5) * y_.L, -1), version((size_t)y_.arena_units + 5, 0), b_phase((size_t)4 * y_.L, -1) {
    at_ping = (uint32_t)(y.off_ping >> 8); at_pong = (uint32_t)(y.off_pong >> 8);
    at_core[0] = (uint32_t)(y.off_core >> 8); at_core[1] = (uint32_t)(y.off_core2 >> 8);
    at_arena = (uint32_t)(y.off_arena >> 8); loc_step = (uint32_t)(y.loc_bytes >> 8);
  }
  size_t slot_of(int32_t loc) const {
    return loc >= 0 ? (size_t)loc + 5
                    : loc == MEBPTT_LOC_INIT ? 0 : loc == MEBPTT_LOC_PING ? 1 : loc == MEBPTT_LOC_PONG ? 2 : 3 + (size_t)core;
  }
  uint32_t address(int32_t loc) const {
    switch (loc) {
      case MEBPTT_LOC_INIT: return team::kInit;
      case MEBPTT_LOC_PING: return at_ping;
      case MEBPTT_LOC_PONG: return at_pong;
      case MEBPTT_LOC_CORE: return at_core[core];
      default: return at_arena + (uint32_t)loc * loc_step;
    }
  }
  int units(int32_t loc, int fmt) const {
    if (loc < 0) return 1;
    const size_t bytes = fmt == MEBPTT_FMT_HIDDEN ? y.unit : fmt == MEBPTT_FMT_INTERNAL ? y.rec : y.rec_in;
    return (int)((bytes + y.loc_bytes - 1) / y.loc_bytes);
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
  int red_of(const Task& t) const {
    const int u = ceil_div(y.H, c.T);
    const int w = t.kind == FWD ? u * c.ns_f[t.layer] : t.kind == READ ? ceil_div(d.groups_o, c.T) * c.ns_r : ceil_div(u, 4) * c.ns_b[t.layer];
    return w * c.nb * 4;
  }
  int64_t place(const Item& it, int64_t after) {
    int64_t p = std::max(after + 1, base);
    for (;; ++p) {
      const size_t i = (size_t)(p - base);
      if (i >= open.size()) { open.resize(i + 1); red.resize(i + 1, 0); }
      const int need = red_of(it.t);
      if (open[i].size() < team::kMaxPhaseTasks && red[i] + need <= c.red_floats) {
        red[i] += need;
        open[i].push_back(it);
        break;
      }
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
    // dy takes the place of dy_{k+4}
    int64_t above = place(r, std::max(state[si * L + L - 1], b_phase[(size_t)(L - 1) * 4 + q])), last = above;
    for (int l = L - 1; l >= 0; --l) {
      Item b;
      b.t = Task{};
      b.t.kind = BWD; b.t.layer = (uint8_t)l; b.t.k = (int32_t)op.k; b.t.sidx = (uint16_t)sidx; b.t.src = address(op.src);
      int64_t after = std::max(std::max(state[si * L + l], above), b_phase[(size_t)l * 4 + ((q + 1) & 3)]);
      // dz_k takes the place of dz_{k+2}, which the layer below has to have read
      if (l > 0) after = std::max(after, b_phase[(size_t)(l - 1) * 4 + ((q + 2) & 3)]);
      if (op.dst_fmt == MEBPTT_FMT_INTERNAL) {
        b.t.dst = b.t.src + (uint32_t)(y.rec_in >> 8);
      } else {
        b.t.dst = address(op.aux);
        after = std::max(after, state[slot_of(op.aux) * L + l]);
      }
      if (sidx == 0) b.t.flags |= CARRY_OUT;
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
  static uint16_t u16(int floats) { return (uint16_t)(floats / 16); }

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
    Pools pools;
    pools.x.resize(kXSlots);
    pools.h.resize((size_t)y.L * kHSlots);
    std::vector<int64_t> dz((size_t)y.L * kDzSlots, -1);       // step whose dz lies in a slot
    for (size_t p = 0; p < open.size(); ++p) {
      std::vector<Item> rest(open[p]);
      while (!rest.empty()) {
        const int e = (int)out.size();                          // the phase being put together
        Pools q = pools;
        std::vector<int64_t> qdz = dz;
        std::vector<Task> now, loads;
        std::vector<Item> later;
        bool gap = false;                                       // a phase of loads has to come first
        auto operand = [&](Slot* pool, int n, Key key, const Task& load, int slot0, int floats, int& at) {
          int i = find(pool, n, key);
          if (i < 0) {
            i = e > 0 ? victim(pool, n, e - 1, e, (int)p - 1) : -1;
            if (i < 0 || (e > 0 && out.back().size() + loads.size() >= (size_t)kPhaseTasks)) { gap = true; return; }
            Task l = load;
            l.so = u16(slot0 + i * floats);
            loads.push_back(l);
            pool[i].key = key;
            pool[i].pushed = e - 1;
          }
          pool[i].read = e;
          at = slot0 + i * floats;
        };
        for (size_t j = 0; j < rest.size() && !gap; ++j) {
          const Item& it = rest[j];
          Task t = it.t;
          const int l = t.layer;
          Slot* hl = q.h.data() + (size_t)l * kHSlots;
          int a = 0, b = 0;
          Task load{};
          load.layer = (uint8_t)l;
          if (t.kind == FWD || t.kind == READ) {
            if (t.kind == FWD && l == 0) {
              load.kind = LOAD_X; load.k = t.k;
              operand(q.x.data(), kXSlots, key_x(t.k), load, slot_x(c, 0), c.x_slot, a);
            } else if (t.kind == FWD) {
              load.kind = LOAD_H; load.layer = (uint8_t)(l - 1); load.src = t.dst;
              operand(hl - kHSlots, kHSlots, key_h(l - 1, it.out), load, slot_h(y, c, l - 1, 0), c.h_slot, a);
              load.layer = (uint8_t)l;
            }
            if (gap) break;
            load.kind = LOAD_H; load.src = t.src;
            operand(hl, kHSlots, key_h(l, it.in), load, slot_h(y, c, l, 0), c.h_slot, b);
            if (gap) break;
            if (t.kind == READ) { a = b; b = -1; }
          } else {
            const int par = (t.k + 1) & 1;
            if (qdz[(size_t)l * kDzSlots + par] != t.k + 1) {
              if (e == 0 || out.back().size() + loads.size() >= (size_t)kPhaseTasks) { gap = true; break; }
              load.kind = LOAD_DZ; load.k = t.k + 1; load.sidx = (uint16_t)(t.sidx + 1);
              if (t.k == y.t || t.sidx == y.S - 1) load.flags |= CARRY;
              load.so = u16(slot_dz(y, c, l, par));
              loads.push_back(load);
              qdz[(size_t)l * kDzSlots + par] = t.k + 1;
            }
            a = slot_dz(y, c, l, par);
            b = l + 1 < y.L ? slot_dz(y, c, l + 1, t.k & 1) : slot_dy(y, c, t.k & 3);
          }
          t.sa = u16(a);
          t.sb = b < 0 ? kNone : u16(b);
          now.push_back(t);
          later.push_back(it);
        }
        if (gap) { out.emplace_back(); continue; }
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
              t.so = u16(slot_h(y, c, l, i));
            }
          } else if (t.kind == READ) {
            t.so = u16(slot_dy(y, c, t.k & 3));
          } else {
            t.so = u16(slot_dz(y, c, l, t.k & 1));
            qdz[(size_t)l * kDzSlots + (t.k & 1)] = t.k;
          }
          done.push_back(t);
        }
        if (done.empty()) { out.emplace_back(); continue; }     // every slot was read or written just now: a phase of nothing in between
        if (!loads.empty()) out.back().insert(out.back().end(), loads.begin(), loads.end());
        out.push_back(done);
        pools = q;
        dz = qdz;
        rest = wait;
      }
    }
    team::Launch g;
    g.task0 = s.tasks.size();
    auto pad = [&] { while (s.tasks.size() % kWindow) s.tasks.push_back(Task{}); };
    for (std::vector<Task>& ph : out) {
      if (ph.empty()) ph.push_back(Task{});                     // loads for nobody: keeps its place as an empty phase
      int r = 0;
      for (Task& t : ph)
        if (t.kind == FWD || t.kind == READ || t.kind == BWD) { t.red = (uint16_t)(r / 4); r += red_of(t); }
      if (s.tasks.size() % kWindow + ph.size() > (size_t)kWindow) pad();
      ph[0].n = (uint8_t)ph.size();
      s.tasks.insert(s.tasks.end(), ph.begin(), ph.end());
      ++g.phases;
    }
    pad();
    g.ntasks = s.tasks.size() - g.task0;
    g.chunk = chunk;
    s.launches.push_back(g);
    open.clear();
    red.clear();
    n_open = 0;
    base = top + 1;
  }
};

}  // namespace

void build_schedule(const Layout& y, const Plan* p, const Config& c, Schedule& s) {
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
    if (w.n_open > (int64_t)team::kMaxLaunchTasks / 6) w.close(-1);
  }
}

}  // namespace pod
}  // namespace mebptt

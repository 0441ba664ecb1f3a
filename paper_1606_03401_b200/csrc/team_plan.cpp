// Host side of the team path: how a problem is laid over the device, and the schedule of phases a
// plan's tape is turned into.  Plain C++, no CUDA.
#include <algorithm>
#include <cstring>

#include "pod.hpp"
#include "team.hpp"

namespace mebptt {
namespace team {

namespace {
inline int pad16(int v) { return (v + 15) & ~15; }
inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
}  // namespace

Dims dims(const Layout& y) {
  Dims d{};
  d.mma = y.dtype == MEBPTT_BF16 && y.tensor_cores;
  d.rpg = d.mma ? 16 : 4;
  d.gp = pad16(4 * y.H);
  d.hp = pad16(y.H);
  for (int l = 0; l < y.L && l < kMaxLayers; ++l) {
    d.ip[l] = pad16(l == 0 ? y.I : y.H);
    d.kf[l] = d.ip[l] + d.hp;
    d.kb[l] = d.gp + (l + 1 < y.L ? d.gp : pad16(y.O));
  }
  d.gf = ceil_div(4 * y.H, d.rpg);
  d.gb = ceil_div(y.H, d.rpg);
  d.gr = ceil_div(y.O, d.rpg);
  return d;
}

namespace {
// floats of pool: k staged elements a row (gradients on the tensor cores in three planes), partial sums
Need need(const Dims& d, const Config& c, int groups, int k, int ns, bool planes) {
  const int row = d.mma ? (planes ? 3 : 1) * (k + 8) / 2 : k;
  return Need{(c.nb * row + 3) & ~3, ceil_div(groups, c.T) * ns * c.nb * d.rpg};
}
}  // namespace
Need need_f(const Layout& y, const Dims& d, const Config& c, int l) { (void)y; return need(d, c, d.gf, d.kf[l], c.ns_f[l], false); }
Need need_r(const Layout& y, const Dims& d, const Config& c) { (void)y; return need(d, c, d.gr, d.hp, c.ns_r, false); }
Need need_b(const Layout& y, const Dims& d, const Config& c, int l) { (void)y; return need(d, c, d.gb, d.kb[l], c.ns_b[l], true); }

namespace {

// One task's share of a phase in clock cycles: operands from the L2 into shared memory, then what the
// arithmetic and the weights take, from shared memory or from the L2.
double task_cycles(const Config& c, const Dims& d, int groups_cta, int k, int ns, int esz, bool resident, bool planes) {
  const int nsub = ceil_div(c.rows, c.nb), rounds = ceil_div(groups_cta * ns, kWarps);
  double t;
  if (d.mma) {
    t = rounds * (ceil_div(k / 16, ns) * (planes ? 60.0 : 35.0) + 200.0);
  } else {
    const int its = ceil_div(k, 128);
    t = std::max((double)groups_cta * its * (4.0 * c.nb + 4.0 * esz), rounds * (ceil_div(its, ns) * 80.0 + 300.0));
  }
  const double ctas = (double)c.teams * c.T;
  if (!resident) {   // weights from the L2, as fast as an SM takes them in or all SMs together get them
    const double bytes = (double)groups_cta * d.rpg * k * esz;
    t = std::max(t, std::max(bytes / 45.0, bytes * ctas / 4000.0));
  }
  const double stage = (double)c.nb * k * (planes ? 4 : esz);
  return nsub * (t + 300.0 + std::max(stage / 30.0, stage * ctas / 4000.0));
}

// Fills in everything that follows from T, teams and rows; returns the estimated cycles of two
// forward operations and one backward operation, or a negative value if the shape does not fit.
double finish(const Layout& y, const Dims& d, Config& c) {
  const int uf = ceil_div(d.gf, c.T), ub = ceil_div(d.gb, c.T), ur = ceil_div(d.gr, c.T);
  const int esz = (int)y.esz, step = d.mma ? 64 : 128;   // least elements of the contraction index worth a piece of their own
  auto parts = [&](int groups, int k) { return std::max(1, std::min(ceil_div(k, step), kWarps / groups)); };
  c.ns_r = parts(ur, d.hp);
  int most = 0, sum_f = 0, sum_b = 0;
  const Need nr = need_r(y, d, c);
  for (int l = 0; l < y.L; ++l) {
    c.ns_f[l] = parts(uf, d.kf[l]);
    c.ns_b[l] = parts(ub, d.kb[l]);
    const Need f = need_f(y, d, c, l), b = need_b(y, d, c, l);
    most = std::max(most, std::max(f.a + f.red, b.a + b.red));
    sum_f += f.a + f.red;
    sum_b += b.a + b.red;
  }
  most = std::max(most, nr.a + nr.red);
  const int want = std::max(sum_f, sum_b) + nr.a + nr.red;
  const int fixed = 2 * kTaskWindow * (int)sizeof(Task) + 256;
  const int budget = kSmemMax - fixed;
  if ((int64_t)most * 4 > budget) return -1.0;
  auto bytes_f = [&](int l) { return (int64_t)uf * d.rpg * d.kf[l] * esz; };
  auto bytes_b = [&](int l) { return (int64_t)ub * d.rpg * d.kb[l] * esz; };
  const int64_t bytes_r = (int64_t)ur * d.rpg * d.hp * esz;
  int64_t all = bytes_r;
  for (int l = 0; l < y.L; ++l) all += bytes_f(l) + bytes_b(l);
  // room for a phase of the wavefront over the layers where the weights leave it, at least for one task
  int64_t pool = std::min<int64_t>((int64_t)want * 4, std::max<int64_t>((int64_t)most * 4, budget - all));
  c.pool_floats = (int)((pool + 15) / 16) * 4;
  if ((int64_t)c.pool_floats * 4 > budget) c.pool_floats = budget / 16 * 4;
  int64_t left = budget - (int64_t)c.pool_floats * 4, held = 0;
  c.resident = 0;
  auto keep = [&](int bit, int64_t bytes) {
    if (bytes <= left) { c.resident |= 1ull << bit; left -= bytes; held += bytes; }
  };
  for (int l = 0; l < y.L; ++l) keep(2 * l, bytes_f(l));
  for (int l = 0; l < y.L; ++l) keep(2 * l + 1, bytes_b(l));
  keep(63, bytes_r);
  c.smem = fixed + c.pool_floats * 4 + (int)held;
  double cyc = 3 * 14000.0 + task_cycles(c, d, ur, d.hp, c.ns_r, esz, (c.resident >> 63) & 1, false);
  for (int l = 0; l < y.L; ++l)
    cyc += 2 * task_cycles(c, d, uf, d.kf[l], c.ns_f[l], esz, (c.resident >> (2 * l)) & 1, false) +
           task_cycles(c, d, ub, d.kb[l], c.ns_b[l], esz, (c.resident >> (2 * l + 1)) & 1, true);
  c.ok = true;
  return cyc;
}

}  // namespace

// The number of teams with the least estimated time: with more of them a team has fewer rows to stage
// and meets fewer CTAs, with fewer a CTA has fewer weights, which it can then hold.
Config choose_config(const Layout& y, int sms) {
  Config best;
  if (y.L > kMaxLayers) return best;
  const Dims d = dims(y);
  for (int teams = 1; teams <= sms / 17; ++teams) {
    const int rows = ceil_div(y.B, std::min(teams, y.B));
    for (int nb = 1; nb <= 8; nb *= 2) {   // rows taken at a time: as many as there are, if they fit
      if (nb > 1 && nb >= 2 * rows) break;
      Config c;
      c.T = sms / teams; c.rows = rows; c.teams = ceil_div(y.B, rows); c.nb = nb;
      c.cycles = finish(y, d, c);
      if (c.cycles >= 0 && (!best.ok || c.cycles < best.cycles)) best = c;
    }
  }
  return best;
}

// Shapes other tensor-core kernels could take as well go to whichever is estimated faster, by the clock
// cycles of two forward operations and a backward one.  Step by step these take some 45 us a layer
// whatever the widths (three or four dependent launches each; measured from 160 to 1024 units), and stay
// ahead where the recurrent weights are large.  The persistent kernels for float32 storage take some
// 20 us and a launch or several a run.  Measured on both sides of the line (150 steps, input and readout as
// wide, us under HSM 20, ISM 20, MSM 30 and full memory; walked, then runs):
//   H = 192, B = 32 (estimated 29200)  3478 2606 2874 1907   3655 2712 3559 1804
//   H = 160, B = 64 (31000)            4137 3139 3413 2378   3988 2997 3841 2099
//   H = 208, B = 32 (32000)            3613 2764 2988 2079   3884 2840 3791 1850
//   H = 224, B = 32 (33200)            3787 2932 3155 2200   3759 2756 3634 1827
//   H = 176, B = 64 (34700)            4599 3505 3797 2665   4238 3142 4114 2141
bool supported(const mebptt_lstm_desc* d) {
  constexpr double kStepwise = 70000.0;   // a fifth less than measured, to be worth leaving
  constexpr double kRuns = 33000.0;
  Layout y;
  state_layout(d, y);
  if (y.tensor_path || y.L > kMaxLayers || y.t >= (1 << 30)) return false;
  const Route r = route(y);
  return r.ok && ((!y.stepwise_tc && !y.stepwise_x3) || r.cycles < (y.x3_runs ? kRuns : kStepwise * y.L));
}

Route route(const Layout& y) {
  const DeviceFacts dev = facts();
  Route r;
  r.c = choose_config(y, dev.sms);
  r.pc = pod::choose_config(y, dev);
  r.pod = r.pc.ok && (!r.c.ok || r.pc.cycles <= r.c.cycles);
  r.ok = r.pod || r.c.ok;
  r.cycles = r.pod ? r.pc.cycles : r.c.cycles;
  return r;
}

Wants wants(const Layout& y) {
  Wants s{};
  const Route r = route(y);
  if (r.pod) {
    for (int l = 0; l < y.L; ++l) s.wf[l] = pod::packed_elems(r.pc, l);
    s.wr = pod::packed_readout_elems(r.pc);
    s.rows = r.pc.nb;
  } else {
    const Dims d = dims(y);
    for (int l = 0; l < y.L; ++l) {
      s.wf[l] = (size_t)d.gf * d.rpg * d.kf[l];
      s.wb[l] = (size_t)d.gb * d.rpg * d.kb[l];
    }
    s.wr = (size_t)d.gr * d.rpg * d.hp;
    s.rows = r.c.rows;
  }
  return s;
}

namespace {

// Places each task in the earliest phase after everything it depends on.  Tasks come in the order of
// the tape, so whatever an operation must wait for has its phase already.
struct Scheduler {
  const Layout& y;
  const Config& c;
  const Dims d;
  Schedule& s;
  std::vector<std::vector<Task>> open;     // tasks by phase, from phase `base` on
  std::vector<int> used;                   // floats of the pool taken, likewise
  const size_t room;                       // records of a launch
  int64_t base = 0;                        // phases before this one belong to earlier launches
  int64_t top = -1;                        // last phase used
  // when the cells (units) of the arena were last touched; the same for ping, pong and the two cores,
  // per layer there (what lies in them always has the same format, so layers never share bytes)
  std::vector<int64_t> cell, named;
  // when the state at a location was written, per layer
  std::vector<int64_t> state;              // [location slot][L]
  std::vector<int64_t> bwd_prev;           // per layer: phase of the latest B
  int core = 0;                            // the working core alternates between two buffers

  Scheduler(const Layout& y_, const Config& c_, Schedule& s_, int64_t arena_units, size_t room_)
      : y(y_), c(c_), d(dims(y_)), s(s_), room(room_), cell((size_t)arena_units, -1), named((size_t)4 * y_.L, -1), state((size_t)(arena_units + 5) * y_.L, -1),
        bwd_prev((size_t)y_.L, -1) {
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
  int64_t* state_of(int32_t loc) {
    const size_t slot = loc >= 0 ? (size_t)loc + 5
                        : loc == MEBPTT_LOC_INIT ? 0 : loc == MEBPTT_LOC_PING ? 1 : loc == MEBPTT_LOC_PONG ? 2 : 3 + (size_t)core;
    return state.data() + slot * (size_t)y.L;
  }
  int units(int32_t loc, int fmt) const {   // cells a record takes
    if (loc < 0) return 1;
    const int blocks = fmt == MEBPTT_FMT_HIDDEN ? y.unit_blocks : y.unit_blocks + 4 * y.L + (fmt == MEBPTT_FMT_INTERNAL ? y.unit_blocks : 0);
    return (blocks * y.parts + y.loc_blocks - 1) / y.loc_blocks;
  }
  template <class F> void cells(int32_t loc, int n, int l, F f) {
    if (loc >= 0) { for (int i = 0; i < n && (size_t)(loc + i) < cell.size(); ++i) f(cell[(size_t)(loc + i)]); }
    else if (loc != MEBPTT_LOC_INIT)
      f(named[(size_t)(loc == MEBPTT_LOC_PING ? 0 : loc == MEBPTT_LOC_PONG ? 1 : 2 + core) * y.L + (size_t)l]);
  }
  int64_t last_touch(int32_t loc, int n, int l) {
    int64_t p = -1;
    cells(loc, n, l, [&](int64_t& v) { p = std::max(p, v); });
    return p;
  }
  void touch(int32_t loc, int n, int l, int64_t phase) {
    cells(loc, n, l, [&](int64_t& v) { v = std::max(v, phase); });
  }
  int64_t place(Task t, int64_t after, Need n) {
    int64_t p = std::max(after + 1, base);
    const int need = (n.a + n.red + 3) & ~3;
    for (;; ++p) {
      const size_t i = (size_t)(p - base);
      if (i >= open.size()) { open.resize(i + 1); used.resize(i + 1, 0); }
      if ((int)open[i].size() < kMaxPhaseTasks && used[i] + need <= c.pool_floats) {
        t.a_off = (uint32_t)used[i];
        t.red_off = (uint32_t)(used[i] + n.a);
        used[i] += need;
        open[i].push_back(t);
        break;
      }
    }
    top = std::max(top, p);
    return p;
  }
  // Ends a launch: everything placed so far is emitted, later tasks start in new phases.
  void close(int chunk) {
    Launch cur;
    cur.task0 = s.tasks.size();
    auto pad = [&] { while (s.tasks.size() % kTaskWindow) s.tasks.push_back(Task{}); };
    auto end = [&](int ch) {
      pad();
      cur.ntasks = s.tasks.size() - cur.task0;
      cur.chunk = ch;
      s.launches.push_back(cur);
      cur = Launch{};
      cur.task0 = s.tasks.size();
    };
    for (auto& ph : open) {
      if (ph.empty()) continue;
      if (s.tasks.size() % kTaskWindow + ph.size() > (size_t)kTaskWindow) pad();
      if (s.tasks.size() > cur.task0 && s.tasks.size() - cur.task0 + kTaskWindow > room) end(-1);
      ph.back().flags |= LAST;
      s.tasks.insert(s.tasks.end(), ph.begin(), ph.end());
      ++cur.phases;
    }
    end(chunk);
    s.phases += s.launches.back().phases;
    open.clear();
    used.clear();
    base = top + 1;
  }
  void forward(const mebptt_op& op) {
    const uint32_t src = address(op.src);
    const std::vector<int64_t> in(state_of(op.src), state_of(op.src) + y.L);
    if (op.dst == MEBPTT_LOC_CORE) core ^= 1;   // (never the source as well: a valid tape does not read what it writes)
    const int n = units(op.dst, op.dst_fmt), n_src = units(op.src, MEBPTT_FMT_HIDDEN);
    const int64_t arena_free = op.dst >= 0 ? last_touch(op.dst, n, 0) : -1;   // before any layer of this operation
    int64_t below = -1, last = -1;
    int64_t* out = state_of(op.dst);
    for (int l = 0; l < y.L; ++l) {
      Task t{};
      t.kind = FWD; t.layer = (uint8_t)l; t.k = (int32_t)op.k;
      t.src = src; t.dst = address(op.dst);
      if (op.dst_fmt != MEBPTT_FMT_HIDDEN) t.flags |= GATES;
      if (op.dst_fmt == MEBPTT_FMT_INTERNAL) t.flags |= COPY_IN;
      if (l == 0) t.flags |= COUNT;
      const int64_t free_at = op.dst >= 0 ? arena_free : last_touch(op.dst, n, l);
      const int64_t p = place(t, std::max(std::max(in[(size_t)l], below), free_at), need_f(y, d, c, l));
      out[l] = p;
      below = p;
      last = std::max(last, p);
      if (op.dst < 0) touch(op.dst, n, l, p);
      if (op.dst < 0 && l > 0) touch(op.dst, n, l - 1, p);
      if (op.src < 0) touch(op.src, n_src, l, p);
    }
    if (op.dst >= 0) touch(op.dst, n, 0, last);
    if (op.src >= 0) touch(op.src, n_src, 0, last);
  }
  void backward(const mebptt_op& op) {
    const int sidx = (int)((op.k - 1) % y.S);
    const int64_t* in = state_of(op.src);
    Task t{};
    t.kind = READ; t.layer = (uint8_t)(y.L - 1); t.k = (int32_t)op.k; t.sidx = (uint32_t)sidx;
    t.src = address(op.src);
    int64_t above = place(t, in[y.L - 1], need_r(y, d, c)), last = above;
    for (int l = y.L - 1; l >= 0; --l) {
      Task b{};
      b.kind = BWD; b.layer = (uint8_t)l; b.k = (int32_t)op.k; b.sidx = (uint32_t)sidx;
      b.src = address(op.src);
      int64_t after = std::max(std::max(in[l], above), bwd_prev[(size_t)l]);
      if (op.dst_fmt == MEBPTT_FMT_INTERNAL) {
        b.dst = b.src + (uint32_t)((y.unit_blocks + 4 * y.L) * y.parts);
      } else {
        b.dst = address(op.aux);
        after = std::max(after, state_of(op.aux)[l]);
      }
      if (op.k == y.t || sidx == y.S - 1) b.flags |= CARRY_IN;
      if (sidx == 0) b.flags |= CARRY_OUT;
      if (l == y.L - 1) b.flags |= COUNT;
      const int64_t p = place(b, after, need_b(y, d, c, l));
      bwd_prev[(size_t)l] = p;
      above = p;
      last = std::max(last, p);
    }
    // (every layer at once: the working core is rewritten no sooner than two forward operations later)
    for (int l = 0; l < (op.src < 0 ? y.L : 1); ++l) touch(op.src, units(op.src, op.dst_fmt), l, last);
    if (op.dst_fmt != MEBPTT_FMT_INTERNAL)
      for (int l = 0; l < (op.aux < 0 ? y.L : 1); ++l) touch(op.aux, units(op.aux, MEBPTT_FMT_HIDDEN), l, last);
  }
};

}  // namespace

void build_schedule(const Layout& y, const Plan* p, const Config& c, size_t room, Schedule& s) {
  Scheduler w(y, c, s, y.arena_units, room);
  for (const mebptt_op& op : p->tape) {
    if (op.kind == MEBPTT_OP_FWD) {
      w.forward(op);
    } else {
      w.backward(op);
      if ((op.k - 1) % y.S == 0) w.close((int)((op.k - 1) / y.S));
    }
    // a tape with very many recomputations between two backward operations: do not hold it all open
    if (w.open.size() > 4 * kMaxLaunchTasks) w.close(-1);
  }
}

bool build_records(const Layout& y, const Plan* p, const Route& r, size_t room, Records& out) {
  if (room < (r.pod ? pod::kLeastRoom : (size_t)kTaskWindow)) return false;
  auto keep = [&](const auto& s) {
    out.bytes.resize(s.tasks.size() * sizeof(Task));
    memcpy(out.bytes.data(), s.tasks.data(), out.bytes.size());
    out.launches = s.launches;
  };
  if (r.pod) {
    pod::Schedule s;
    pod::build_schedule(y, p, r.pc, room, s);
    keep(s);
  } else {
    Schedule s;
    build_schedule(y, p, r.c, room, s);
    keep(s);
  }
  // (the launches copy their records to the room and read them there: one that did not fit would read what lies behind)
  for (const Launch& g : out.launches)
    if (g.ntasks > room) return false;
  return true;
}

}  // namespace team
}  // namespace mebptt

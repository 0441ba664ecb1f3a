// The pod kernel: the team path's small and middle sizes, where a phase is a fraction of a microsecond
// of arithmetic and everything else is the distance between the CTAs.
//
// A pod is a thread-block cluster that walks the tape for NB batch rows.  What a phase produces for
// the others -- h of a layer, dz, dy -- is pushed straight into the operand slots in every CTA's shared
// memory (asynchronous stores that count their bytes on the receiver's barrier), so that the next
// phase starts from shared memory; nothing crosses CTAs through global memory.  Everything else a
// task reads there (cell states, gates, carried gradients, a stored state that comes back) was
// written by the same thread, and is fetched one phase ahead.
//
// Which vector lies in which slot at which phase is decided on the host, like registers by a
// compiler: a state that is not in a slot any more when it is needed is brought back by a load task
// in the phase before.
#pragma once

#include <cstdint>
#include <vector>

#include "layout.hpp"
#include "plan.hpp"
#include "team.hpp"

namespace mebptt {
namespace pod {

using team::kThreads;
using team::kWarps;
constexpr int kWindow = 64, kWindows = 4;     // tasks fetched at a time, windows held
constexpr int kPhaseTasks = 12;
constexpr int kHSlots = 4, kXSlots = 4, kDzSlots = 2, kDySlots = 4;   // operand slots (h, dz: per layer)
constexpr uint16_t kNone = 0xffff;

enum Kind : uint8_t { NOP = 0, FWD = 1, READ = 2, BWD = 3, LOAD_H = 4, LOAD_X = 5, LOAD_DZ = 6 };
enum Flag : uint8_t {
  GATES = 1, COPY_IN = 2,   // F: what the destination keeps
  CARRY = 4,                // LOAD_DZ: from the carry buffer (else from the stage)
  CARRY_OUT = 8,            // B: leave dz in the carry buffer too
  COUNT = 16
};
struct Task {
  uint8_t kind, layer, flags, n;   // n: tasks of the phase, in its first task
  int32_t k;
  uint32_t src, dst;               // as team::Task; LOAD_H: src is the state
  uint16_t sidx, sa, sb, so;       // row block in the stages; slots of the two operand segments and of the result (16-float units)
  uint16_t red, pad[3];            // partial sums, 4-float units
};
static_assert(sizeof(Task) == 32, "Task layout");

struct Config {
  bool ok = false;
  double cycles = 0;               // estimate for two forward operations and one backward operation
  int T = 1, nb = 1, pods = 1;
  int ns_f[team::kMaxLayers] = {}, ns_b[team::kMaxLayers] = {}, ns_r = 1;
  uint64_t resident = 0;           // as team::Config
  int slot_floats = 0, red_floats = 0;   // all slots; partial sums of one phase (there are two such areas)
  int x_slot = 0, h_slot = 0, dz_slot = 0, dy_slot = 0;   // floats of one slot
  int smem = 0;
};
// first float of a slot
int slot_x(const Config& c, int i);
int slot_h(const Layout& y, const Config& c, int l, int i);
int slot_dz(const Layout& y, const Config& c, int l, int i);
int slot_dy(const Layout& y, const Config& c, int i);

Config choose_config(const Layout& y, int sms, const int* max_clusters);

struct Schedule {
  std::vector<Task> tasks;
  std::vector<team::Launch> launches;
};
void build_schedule(const Layout& y, const Plan* p, const Config& c, Schedule& s);

}  // namespace pod
}  // namespace mebptt

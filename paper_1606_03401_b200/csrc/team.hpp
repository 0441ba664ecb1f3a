// The team path: shapes and precisions the tensor-core kernels do not cover (float32 products on
// CUDA cores, GRU cores, bfloat16 widths that are no multiples of 8), run by one persistent kernel
// per chunk of time steps instead of a launch per contraction.
//
// The recurrence never mixes batch rows, so the batch is cut into groups and each group is given to
// a team of T CTAs that walks the tape by itself.  The tape is turned into tasks, and the tasks into
// phases on the host: everything in a phase is independent, and the CTAs of a team meet once per phase.
// A CTA owns hidden units of every layer; its slices of the weights stay in shared memory.
//
//   F(op, l)  forward operation of layer l: the four gates of a unit are one group of 4 weight rows
//   R(op)     readout of the top layer and dy; groups of 4 readout rows
//   B(op, l)  backward operation of layer l: dh = dz_{k+1} W_hh + (dz_k of the layer above) W_ih (or
//             dy W_out), then the gate derivatives; groups of 4 units (rows of the transposed weights)
//
// Weight, bias and input gradients are contractions over a whole chunk of S steps (from stages the
// B tasks fill), between two launches of the persistent kernel.
#pragma once

#include <cstdint>
#include <vector>

#include "layout.hpp"
#include "plan.hpp"

namespace mebptt {
namespace team {

constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kSmemMax = 227 * 1024;
constexpr int kTaskWindow = 64;        // tasks a CTA fetches at a time; no phase straddles two windows
constexpr int kMaxPhaseTasks = 8;
constexpr int kMaxLayers = 16;

enum TaskKind : uint8_t { NOP = 0, FWD = 1, READ = 2, BWD = 3 };
enum TaskFlag : uint8_t {
  LAST = 1,        // ends its phase
  GATES = 2,       // F: the destination keeps the gates
  COPY_IN = 4,     // F: ... and a copy of the input state
  CARRY_IN = 8,    // B: dz_{k+1} of this layer lies in the carry buffer
  CARRY_OUT = 16,  // B: leave dz_k in the carry buffer too (first step of a chunk)
  COUNT = 32       // F of layer 0 / B of the top layer: counts as an operation
};
struct Task {
  uint8_t kind, layer, flags, pad0;
  int32_t k;
  uint32_t src;    // F: input state; R, B: record of step k.  blocks from the start of the team's states
  uint32_t dst;    // F: record written; B: state k-1 (whole-state block)
  uint32_t sidx;   // row block of step k in the stages
  uint32_t a_off, red_off, pad1;   // this task's share of the phase pool, in floats
};
static_assert(sizeof(Task) == 32, "Task layout");

// Sizes that follow from the shape alone.  A group is what a warp forms at a time: 4 weight rows on FMA
// (a unit's gates, 4 units of the transposed weights, 4 readout rows), 16 on the tensor cores.
struct Dims {
  bool mma;             // bfloat16 storage, tensor cores not forbidden
  int rpg;              // rows of a group
  int kf[kMaxLayers];   // row length of the packed forward weights (input part and recurrent part padded)
  int ip[kMaxLayers];   // padded input part of it
  int kb[kMaxLayers];   // row length of the transposed weights: 4H (recurrent), then 4H of the layer above or O
  int gp;               // padded 4H
  int hp;               // padded H: row length of the readout weights
  int gf, gb, gr;       // groups of forward rows, of units, of readout rows
};
Dims dims(const Layout& y);

struct Config {
  bool ok = false;
  double cycles = 0;                        // estimate for two forward operations and one backward operation
  int T = 1, teams = 1, rows = 1, nb = 1;   // CTAs per team, teams, batch rows per team, rows taken at a time
  int ns_f[kMaxLayers] = {}, ns_b[kMaxLayers] = {}, ns_r = 1;   // parts the contraction index is cut into
  int pool_floats = 0;                      // shared memory for a phase's operands and partial sums
  uint64_t resident = 0;                    // bit 2l: F(l) weights in shared memory, 2l+1: B(l), 63: readout
  int smem = 0;
};
// What a phase's pool holds for one task, in floats: staged operand rows and partial sums.
struct Need { int a, red; };
Need need_f(const Layout& y, const Dims& d, const Config& c, int l);
Need need_r(const Layout& y, const Dims& d, const Config& c);
Need need_b(const Layout& y, const Dims& d, const Config& c, int l);

Config choose_config(const Layout& y, int sms);

// What a configuration needs to know of the device: SMs, and clusters of 1, 2, .. 16 CTAs (a whole SM each)
// that are resident at once.  These are a B200's, and on a device with as many SMs they are not asked for: the
// same problem then takes the same kernels, with the same bits, on every one of them, and in a count made
// without a device.  A part of a device (fewer SMs) is asked.
struct DeviceFacts { int sms = 148; int clusters[5] = {148, 74, 33, 15, 7}; };
DeviceFacts facts();

// The kernel a problem goes to: the pod kernel (pod.hpp) or the walking kernel, whichever is estimated
// faster.  It depends on the descriptor alone, not on the plan.
struct Route;

struct Launch {          // one launch of the persistent kernel
  size_t task0 = 0, ntasks = 0;   // a whole number of windows
  int phases = 0;
  int fwd_ops = 0, bwd_ops = 0;   // operations it executes
  int chunk = -1;                 // >= 0: this chunk of S steps is complete afterwards
};
struct Schedule {
  std::vector<Task> tasks;
  std::vector<Launch> launches;
  int64_t phases = 0;
};
// room: records a launch may have (a whole number of windows)
void build_schedule(const Layout& y, const Plan* p, const Config& c, size_t room, Schedule& s);

}  // namespace team
}  // namespace mebptt

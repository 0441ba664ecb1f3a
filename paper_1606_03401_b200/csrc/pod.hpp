// The pod kernel: the team path's small and middle sizes, where a phase is a fraction of a microsecond
// of arithmetic and everything else is the distance between the CTAs and the instructions in front of
// and behind it.
//
// A pod is a thread-block cluster of T CTAs that walks the tape for NB batch rows.  CTA r owns U hidden
// units of every layer: their four gate rows of [W_ih | W_hh], U rows of carried state, a share of the
// readout rows.  One copy of a CTA's weights, in shared memory, serves both directions:
//
//   F(op, l)  z of the own units from all of the input and of h_{k-1}, which every CTA holds: h_k of the
//             own units is pushed to all CTAs
//   B(op, l)  dz_k of the own units, whose products with the own weight rows are shares of dh_{k-1} (and
//             of the gradient of the layer below) for all units: each is pushed to the unit's owner, who
//             adds the T shares in rank order
//   R(op)     readout rows of the CTA, dy;  D(op)  their shares of the gradient entering the top layer
//   Z(l)      B without the cell part, from the carried dz of the chunk after: at the start of a launch
//
// Pushes are asynchronous stores into the other CTAs' shared memory that count their bytes on the
// receiver's barrier.  Nothing crosses CTAs through global memory; what a task reads there was written
// by the same thread, and is fetched one phase ahead.  Which state lies in which slot of shared memory
// at which phase is decided on the host, like registers by a compiler: a state that is no longer there
// when it is needed comes back by a load task in the phase before.
#pragma once

#include <cstdint>
#include <vector>

#include "layout.hpp"
#include "plan.hpp"
#include "team.hpp"

#ifdef __CUDACC__
#define MEBPTT_BOTH __host__ __device__
#else
#define MEBPTT_BOTH
#endif

namespace mebptt {
namespace pod {

using team::kThreads;
using team::kWarps;
constexpr int kMaxLayers = 7;     // (an eighth place in the index words stays free)
constexpr int kWindow = 64, kWindows = 4;     // records fetched at a time, windows held
constexpr int kHSlots = 4, kXSlots = 4;       // h of a layer; x

enum Kind : uint8_t { NOP = 0, FWD = 1, READ = 2, BWD = 3, LOAD_H = 4, LOAD_X = 5, DHA = 6, CARRY = 7 };
enum Flag : uint8_t {
  GATES = 1, COPY_IN = 2,   // F: what the destination keeps
  FIRST = 4,                // B: nothing comes from step k + 1
  OPEN = 8,                 // B: the chunk's last step: h_k goes to the stage as well
  CLOSE = 16,               // B: the chunk's first step: dz_k goes to the carry buffer, no share for step k - 1
  COUNT = 32
};
// A phase: a header, then its tasks, those with products first.  At most one F or B, one load and one Z
// per layer, one R, one D and one LOAD_X in a phase.  Everything that is the same for all CTAs is worked
// out here: an instruction saved in a phase is saved a thousand times.
struct Header {
  uint8_t n;                // tasks; 0: nothing but padding up to the next window
  uint8_t cells;            // has B, Z or D: what other threads left has to be waited for before the products
  uint8_t sums;             // has F or R: partial sums are read after the products
  uint8_t n_h;              // pushes every CTA receives of: h,
  uint8_t n_p, n_x;         // shares, x
  uint8_t r, x;             // 1 + index of the READ, LOAD_X task; 0: none
  uint8_t products;         // tasks with products
  uint8_t pad[3];
  uint32_t main, load, carry;   // 4 bits per layer: 1 + index of its F or B, of its load, of its Z
  uint32_t bwd;             // 4 bits per layer: 1 + index of its B
  uint32_t pad2;
};
struct Task {
  uint8_t kind, layer, flags, rot;   // rot: warp that takes the first piece of the products
  int32_t k;
  uint32_t src, dst;        // F: input state, record written; B: record of step k, state k-1; LOAD_H: the state.  Blocks from the start of the pod's states
  // 16-byte units of the operand area:
  //   F: sa input, sb h slot, so slot of the result (or kNone), red partial sums     R: sb, red; so dy
  //   B: sa, sb shares received from step k + 1 and from above; so, red where shares for step k - 1 and for below are sent
  //   Z: so as B    D: sa dy, so    loads: so
  uint16_t sidx, sa, sb, so;
  uint32_t w;               // first weight of the products, elements from the start of the CTA's weights
  uint16_t red, cols;       // cols: B, Z, D: columns of the products
};
static_assert(sizeof(Header) == 32 && sizeof(Task) == 32, "records");
constexpr uint16_t kNone = 0xffff;
constexpr int kPhaseTasks = 14;

struct Config {
  bool ok = false;
  double cycles = 0;        // estimate for two forward operations and one backward operation
  int T = 1, nb = 1, pods = 1;
  int U = 0, up = 0;        // units per CTA, the same padded to 4
  int kx = 0, kh = 0;       // padded widths of x and of h (units in the order of their owners, `up` each)
  int rows_o = 0, op = 0;   // readout rows per CTA, the same padded to 4
  int extra = 0;            // elements added to a row of weights against bank conflicts
  int ns_f[kMaxLayers] = {}, ns_r = 1, ns_b = 1;   // parts the contraction index is cut into; shares a CTA sends per unit
  int works_f0 = 0, works_f1 = 0, works_r = 0;     // pieces of work of F and R
  int lg_f0 = 0, lg_f1 = 0, lg_r = 0, lg_b = 0;    // their logarithms (all layers but the first are alike)
  bool mma = false;         // bfloat16 weights on the tensor cores (else FMA on widened values)
  bool resident = false;    // the weights fit in shared memory
  int planes = 1;           // mma: bfloat16 planes a float32 gradient is split into
  // byte offsets from the start of the operand area, and sizes
  int x_slot = 0, h_slot = 0, pitch_x = 0, pitch_h = 0;   // pitches: bytes of one batch row
  int at_h = 0, at_p = 0, p_slot = 0, at_dz = 0, dz_buf = 0, dz_pitch = 0, at_dy = 0, dy_buf = 0, dy_pitch = 0;
  int at_red = 0, red_bytes = 0, at_dummy = 0, at_map = 0, at_w = 0;
  int smem = 0;
  int red_f(int l) const { return (mma ? (U + 7) / 8 * 8 : U) * (l ? ns_f[1] : ns_f[0]) * nb * 16; }   // bytes of F(l)'s partial sums
  int share_slot(int l, int above, int par) const { return at_p + ((l * 2 + above) * 2 + par) * p_slot; }
  int w_at(int l) const { return l ? 4 * U * pitch_w(0) + (l - 1) * 4 * U * pitch_w(1) : 0; }   // elements; l = L: readout
  MEBPTT_BOTH int pitch_w(int l) const { return (l ? kh : kx) + kh + extra; }   // elements of a row of layer l's weights
  MEBPTT_BOTH int pitch_r() const { return kh + extra; }
  MEBPTT_BOTH int slot_x(int i) const { return i * x_slot; }
  MEBPTT_BOTH int slot_h(int l, int i) const { return at_h + (l * kHSlots + i) * h_slot; }
};
inline int kin(const Config& c, int l) { return l ? c.kh : c.kx; }

Config choose_config(const Layout& y, const team::DeviceFacts& dev);
// elements of the packed weights: layer l, readout
size_t packed_elems(const Config& c, int l);
size_t packed_readout_elems(const Config& c);

}  // namespace pod

struct team::Route {
  bool ok = false;
  bool pod = false;      // the pod kernel with pc, else the walking kernel with c
  double cycles = 0;
  Config c;
  pod::Config pc;
};
namespace team {
Route route(const Layout& y);
// The schedule of a plan for the kernel that serves it, as the 32-byte records that kernel reads; false if a
// launch does not fit the room there is for one.
struct Records { std::vector<unsigned char> bytes; std::vector<Launch> launches; };
bool build_records(const Layout& y, const Plan* p, const Route& r, size_t room, Records& out);
}  // namespace team

namespace pod {

struct Schedule {
  std::vector<Task> tasks;   // records
  std::vector<team::Launch> launches;
};
// room: records a launch may have (a whole number of windows; at least kLeastRoom)
constexpr size_t kLeastRoom = 4 * kWindow;
void build_schedule(const Layout& y, const Plan* p, const Config& c, size_t room, Schedule& s);

}  // namespace pod
}  // namespace mebptt

// The environment switches the library reads, all in one place.  None of them is part of the
// interface: they are aids for measuring and for verifying that two ways of doing the same thing
// give the same bits, read once per process.
//
//   MEBPTT_NO_PDL=1           launch without programmatic stream serialization
//   MEBPTT_NO_OVERLAP=1       weight-gradient GEMMs on the caller's stream instead of the side stream;
//                             host-buffer inputs copied in front of the step instead of beside it
//   MEBPTT_PRIORITY=1         the step on a stream of the library's, of the most urgent priority, instead
//                             of the caller's stream itself
//   MEBPTT_NO_ZX_AHEAD=1      input projections in the step's stream, when a run needs them, instead of a
//                             window ahead on a stream of their own
//   MEBPTT_NO_SPLITK=1        no contraction is split along K (other rounding on the step-by-step paths)
//   MEBPTT_STEPWISE_PER_OP=1  step-by-step paths operation by operation instead of in runs (same bits)
//   MEBPTT_PLAN_SCAN=1        the planner scans every split point instead of walking convex columns
//                             (same tables)
//   MEBPTT_RUN_SMS=n          runs of one bfloat16 layer as on a device that keeps n CTAs resident (same bits)
//   MEBPTT_RUN_CLUSTER=n      likewise, on one that has no clusters of more than n CTAs (same bits from 513 units on)
//   MEBPTT_DEBUG=1            failed CUDA calls are named on stderr
#pragma once

#include <cstdlib>

namespace mebptt {
namespace env {

inline bool flag(const char* name) {
  const char* v = getenv(name);
  return v != nullptr && v[0] != '\0' && !(v[0] == '0' && v[1] == '\0');
}
// 0 when the variable is not set
inline int count(const char* name) {
  const char* v = getenv(name);
  return v ? atoi(v) : 0;
}
inline bool no_pdl() { static const bool v = flag("MEBPTT_NO_PDL"); return v; }
inline bool no_overlap() { static const bool v = flag("MEBPTT_NO_OVERLAP"); return v; }
inline bool priority() { static const bool v = flag("MEBPTT_PRIORITY"); return v; }
inline bool no_zx_ahead() { static const bool v = flag("MEBPTT_NO_ZX_AHEAD"); return v; }
inline bool no_splitk() { static const bool v = flag("MEBPTT_NO_SPLITK"); return v; }
inline bool stepwise_per_op() { return flag("MEBPTT_STEPWISE_PER_OP"); }   // read per call: tests switch it
inline bool plan_scan() { return flag("MEBPTT_PLAN_SCAN"); }               // likewise
inline int run_sms() { static const int v = count("MEBPTT_RUN_SMS"); return v; }
inline int run_cluster() { static const int v = count("MEBPTT_RUN_CLUSTER"); return v; }
inline bool debug() { static const bool v = flag("MEBPTT_DEBUG"); return v; }

}  // namespace env
}  // namespace mebptt

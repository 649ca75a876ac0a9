// ka_ctx.cuh -- the context behind the opaque ka_ctx handle of include/ka.h.
#pragma once

#include <string>
#include <vector>

#include "ka_internal.cuh"
#include "ka_resident.cuh"

struct ka_ctx {
  ka_params prm;
  int topo = 0, d = 0, L = 0, z = 0, m = 0, R = 0;
  int64_t N = 0, nclass = 0, nbonds = 0;
  bool pencil = false;
  cudaStream_t stream = nullptr;
  int device = 0;
  bool owns = false;
  void* buf = nullptr;
  size_t bytes = 0;
  ka::Planes pl{};
  ka::InitScratch is{};
  unsigned long long* counts_dev = nullptr;
  int* err_dev = nullptr;  // device error word of bounded device waits (0 = none), after the counts
  int* wait_mark = nullptr;  // where kernels mark it: err_dev, or (jobs of a batch) the batch's word
  std::vector<int64_t> observed;  // host copy of the counts and that word
  uint64_t* stage = nullptr;
  ka::GraphDev g{};
  const uint4* rec = nullptr;       // small graphs: packed bonds and class offsets (ka_resident.cuh)
  const int32_t* coff = nullptr;
  int64_t class_max = 0;            // bonds of the largest class
  int sms = 0;
  // side stream of the second chain of planes of large three-dimensional
  // lattices (ka_internal.cuh: stream_chains), made with the context; the
  // context's stream waits for it before a sweep call returns
  cudaStream_t side = nullptr;
  cudaEvent_t turn = nullptr;  // the fork, then the join, of a call
  ka::Topology host;  // class offsets (graphs) and tables for inspection
  bool initialized = false;
  bool waits = false;      // sweeps of this context have run kernels with bounded waits
  bool timed_out = false;  // a bounded wait ran out: the state is not valid until init or set_state
  int64_t sweep = 0, K = -1;
  uint64_t seed = 0;
  ka::RoundKeys rk{};
  std::string err;
  // kernel timing
  bool prof = false;
  std::vector<cudaEvent_t> ev;
  std::vector<int> ev_dir;  // direction of every recorded event pair
  size_t ev_used = 0;
  double prof_ms[4] = {0.0, 0.0, 0.0, 0.0};  // by direction mu (graph classes: 0)
  int64_t prof_launches[4] = {0, 0, 0, 0};
};

namespace ka {
// Creates a context in a caller-provided (or owned) device buffer; defined in ka_api.cu.
ka_status create_context(const ka_params* params, void* buf, size_t bytes, bool owns, ka_ctx** out);
// Whether the sweeps of a context stay on chip (ka_resident.cuh), with `words`
// words in the launch: the CTAs per word, or 0; and word w's unit for the
// sweeps t0 .. t0 + count - 1.  Defined in ka_api.cu.
int resident_cluster(const ka_ctx* c, int64_t words);
resident::Unit resident_unit(const ka_ctx* c, int w, uint32_t t0, uint32_t count);
// KA_OK if the context holds a valid state, else why not (also ka_last_error).
// what: the call; defined in ka_api.cu.
ka_status valid_state(ka_ctx* c, const char* what);
// KA_ETIMEOUT if a bounded wait ran out (reads the device error word;
// synchronises the context's stream); defined in ka_api.cu.
ka_status check_waits(ka_ctx* c);
// Device bytes a context needs; defined in ka_api.cu.
ka_status context_bytes(const ka_params* params, size_t* bytes);
}  // namespace ka

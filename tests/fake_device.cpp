// The library's host code on a device that is not there: work queued on a stream runs when
// something waits for it, in order, and a copy from pageable memory reads its source only then.
// Kernels do nothing but what a scenario asks for.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
#include <set>
#include <string>
#include <vector>

#include "../include/sv.h"
#include "batch.h"
#include "jit.h"
#include "kernels.h"
#include "state.h"

namespace {
std::deque<std::function<void()>> g_queue;
size_t g_done = 0, g_queued = 0;
int g_device = 0;
int g_stale = 0, g_copies = 0;  // copies whose source was not what it was when they were queued

void queue(std::function<void()> f) {
  g_queue.push_back(std::move(f));
  ++g_queued;
}
void drain(size_t until = ~(size_t)0) {
  while (!g_queue.empty() && g_done < until) {
    std::function<void()> f = std::move(g_queue.front());
    g_queue.pop_front();
    ++g_done;
    f();
  }
}
}  // namespace

// ---- runtime ----------------------------------------------------------------------------
extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) {
  if (n > 1ull << 40) { *p = nullptr; return cudaErrorMemoryAllocation; }
  *p = std::calloc(1, n);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void *p) { drain(); std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { drain(); std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { drain(); std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  if (kind != cudaMemcpyHostToDevice) { queue([=] { std::memcpy(d, s, n); }); return cudaSuccess; }
  const char *c = static_cast<const char *>(s);
  std::vector<char> then(c, c + n);
  queue([=] {
    ++g_copies;
    if (std::memcmp(c, then.data(), n) != 0) ++g_stale;
    std::memcpy(d, then.data(), n);
  });
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { queue([=] { std::memset(d, v, n); }); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { drain(); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) { *s = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = nullptr; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { *x = reinterpret_cast<cudaGraphExec_t>(8); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
// an event: the number of operations queued before it was recorded
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = reinterpret_cast<cudaEvent_t>(new size_t(0)); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { *reinterpret_cast<size_t *>(e) = g_queued; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { drain(*reinterpret_cast<size_t *>(e)); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete reinterpret_cast<size_t *>(e); return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_device = d; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) { std::memset(p, 0, sizeof(*p)); return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
}

// ---- kernels ----------------------------------------------------------------------------
namespace svk {
namespace { cudaError_t nothing() { queue([] {}); return cudaSuccess; } }
int device_sm_count() { return 152; }
int tile_pass_max_bits() { return 13; }
bool fused_supported() { return true; }
int reduce_partials_needed() { return 8; }
cudaError_t launch_init(float2 *, int, bool, float, cudaStream_t) { return nothing(); }
cudaError_t launch_tile_pass(float2 *, int, const unsigned char *, uint32_t, int, int, cudaStream_t) { return nothing(); }
cudaError_t launch_fused_pass(float2 *, int, const DevPlanView &, int, const svp::DevPass &, cudaStream_t, bool, int) { return nothing(); }
cudaError_t launch_gate_1q(float2 *, int, int, const Mat2 &, cudaStream_t) { return nothing(); }
cudaError_t launch_gate_diag(float2 *, int, uint64_t, uint64_t, float, float, cudaStream_t) { return nothing(); }
cudaError_t launch_norm(const float2 *, int, double *, double *, cudaStream_t) { return nothing(); }
cudaError_t launch_norm_final(const double *, int, double *, cudaStream_t) { return nothing(); }
cudaError_t launch_gather(const float2 *, const uint64_t *, int64_t, double *, cudaStream_t) { return nothing(); }
cudaError_t launch_gather_prob(const float2 *, const uint64_t *, int64_t, double *, cudaStream_t) { return nothing(); }
cudaError_t launch_branch_gather(const float2 *, int, int, const uint64_t *, uint64_t, float2 *, cudaStream_t) { return nothing(); }
cudaError_t launch_branch_sum(const float2 *, int, const float2 *, int, int, const uint64_t *, const uint64_t *, int, double, double *, cudaStream_t) { return nothing(); }
cudaError_t launch_fork(float2 *, int, int, cudaStream_t) { return nothing(); }
int g_outer = 0;
bool g_outer_tc = false;
cudaError_t launch_outer_sum(const float2 *, const float2 *, const OuterShape &, float2, float2 *, cudaStream_t) { ++g_outer; return nothing(); }
bool outer_sum_tc_supported(const OuterShape &) { return g_outer_tc; }
size_t outer_sum_tc_scratch(const OuterShape &) { return (size_t)1 << 41; }
cudaError_t launch_outer_sum_tc(const float2 *, const float2 *, const OuterShape &, float2, float2 *, void *, int *, cudaStream_t) { return nothing(); }
cudaError_t launch_inner(const float2 *, const float2 *, int, double *, double *, cudaStream_t) { return nothing(); }
cudaError_t launch_basis_state(float2 *, int, uint64_t, cudaStream_t) { return nothing(); }
cudaError_t launch_batch_items(const BatchCP *, uint32_t, BatchItem *, uint32_t, cudaStream_t) { return nothing(); }
int batch_run_log(uint32_t, double) { return 0; }
int batch_grid(uint32_t, int) { return 152; }
cudaError_t launch_batch(float2 *, const unsigned char *, uint32_t, const BatchCP *, const BatchItem *, uint32_t, unsigned *, int, cudaStream_t, unsigned long long, int) { return nothing(); }
int g_picked_on = -1;
cudaError_t launch_pick(const float2 *, const PickArgs &, int, float2 *, cudaStream_t) { g_picked_on = g_device; return nothing(); }
cudaError_t launch_batch_stats(const float2 *, const BatchChunk *, int, double *, const int *, int, double *, cudaStream_t) { return nothing(); }
}  // namespace svk
namespace svc {
sv_status build_stage_mats(svp::Plan *, const std::vector<svp::Gate> &, int, bool) { return SV_OK; }
sv_status build_stage_mats_packed(svp::Plan *, const std::vector<svp::Gate> &, bool) { return SV_OK; }
}  // namespace svc
namespace svj {  // every plan has its module and every pass is of the pipelined kind
struct Module {};
namespace { Module g_module; }
int register_slots() { return 4; }
unsigned max_pass_grid() { return 152; }
bool pass_is_pipelined(const svp::Plan &, int) { return true; }
bool pass_can_fork(const svp::Plan &, int bits) { return bits > 0; }
int basis_state_bits(const svp::Plan &) { return 12; }
std::string pipe_pass_source(const svp::Plan &, int, int, bool) { return ""; }
std::string pass_source(const svp::Plan &, int, int, bool) { return ""; }
bool compile(const std::string &, const char *, std::string *, std::string *) { return false; }
bool compile_plan(const svp::Plan &, int, const char *, std::vector<std::string> *, std::string *, const std::string &) { return false; }
const Module *get_module(const svp::Plan &, int, std::string *, bool) { return &g_module; }
bool get_modules(const std::vector<const svp::Plan *> &p, int, std::vector<const Module *> *out, std::string *, bool) {
  out->assign(p.size(), &g_module);
  return true;
}
cudaError_t prepare_passes(const Module *, const svp::Plan &) { return cudaSuccess; }
// the plan kernels' launches, counted; the one with number g_fail gives up a wait
int g_passes = 0, g_fail = -1;
std::string g_kinds;  // w(hole), b(asis), f(ork), l(isted)
namespace {
cudaError_t pass(char kind, const svk::DevPlanView &view) {
  g_kinds += kind;
  int *const err = g_passes++ == g_fail ? view.err : nullptr;
  queue([err] { if (err) *err = 3; });
  return cudaSuccess;
}
}  // namespace
cudaError_t launch_pass(const Module *, float2 *, int, const svk::DevPlanView &view, int, const svp::DevPass &, cudaStream_t,
                        double *, unsigned *grid, const float2 *) {
  if (grid) *grid = 1;
  return pass('w', view);
}
cudaError_t launch_basis_pass(const Module *, float2 *, const svk::DevPlanView &view, const svp::Plan &, int, uint64_t,
                              cudaStream_t, double *, unsigned *grid, const float2 *) {
  if (grid) *grid = 1;
  return pass('b', view);
}
cudaError_t launch_fork_pass(const Module *, float2 *, const svk::DevPlanView &view, const svp::Plan &, cudaStream_t) { return pass('f', view); }
bool last_pass_tiles(const svp::Plan &, const std::vector<uint64_t> &needed, uint64_t, std::vector<uint64_t> *tiles) {
  *tiles = needed;
  return true;
}
cudaError_t launch_listed_pass(const Module *, float2 *, const svk::DevPlanView &view, const svp::Plan &, const uint64_t *,
                               size_t, cudaStream_t) { return pass('l', view); }
}  // namespace svj

// ---- scenarios ----------------------------------------------------------------------------
namespace {

sv_lattice lattice(int rows, int cols, int depth, uint64_t seed) {
  sv_lattice l;
  std::memset(&l, 0, sizeof(l));
  l.rows = rows;
  l.cols = cols;
  l.depth = depth;
  l.seed = seed;
  return l;
}
std::vector<sv_gate> circuit(const sv_lattice &l) {
  size_t n = 0;
  sv_generate_circuit(&l, nullptr, 0, &n);
  std::vector<sv_gate> g(n);
  sv_generate_circuit(&l, g.data(), n, &n);
  return g;
}
sv_options options(int jit, int precision = SV_PREC_PLAIN) {
  sv_options o;
  std::memset(&o, 0, sizeof(o));
  o.jit = jit;
  o.precision = precision;
  return o;
}
int check(sv_status st) {
  if (st != SV_OK) std::printf("status %d: %s\n", (int)st, sv_last_error());
  return st == SV_OK;
}

// Sources of copies: cut amplitudes (their halves' segments follow one another without a wait),
// the full state from two halves, and circuits one after the other on one handle.
int uploads(int jit, int precision) {
  const sv_options o = options(jit, precision);
  sv_cut cut;
  std::memset(&cut, 0, sizeof(cut));
  const sv_lattice l = lattice(4, 4, 12, 5);
  cut.half_a_mask = 0xff;
  std::vector<uint64_t> bits = {1, 0x1234, 0xffff};
  std::vector<double> out(2 * bits.size());
  if (!check(sv_branch_amplitudes(&l, &cut, bits.data(), bits.size(), &o, out.data()))) return 2;
  sv_state *s = nullptr;
  if (!check(sv_create(16, &o, &s)) || !check(sv_branch_full_state(&l, &cut, &o, s))) return 2;
  for (int k = 0; k < 12; ++k) {
    const std::vector<sv_gate> g = circuit(lattice(4, 4, 4 + k, 100 + k));
    if (!check(sv_apply_circuit(s, g.data(), g.size()))) return 2;
  }
  sv_destroy(s);
  drain();
  std::printf("%d copies, %d stale\n", g_copies, g_stale);
  return g_copies < 12 || g_stale != 0;
}

// A wait that gave up in pass `fail` of a state: what the call says that reads the state.
int gave_up(const std::string &how, int fail) {
  sv_options o = options(1);
  std::vector<double> out(4);
  svj::g_fail = fail;
  sv_status st = SV_OK;
  if (how != "product") {  // the forward state of the inner-product amplitudes
    if (how == "whole") o.pipeline = -1;  // (its backward states on whole passes)
    const sv_lattice l = lattice(4, 4, 10, 5);
    const uint64_t bits[2] = {1, 0x1234};
    st = sv_amplitudes_by_inner_product(&l, 5, bits, 2, &o, out.data());
  } else {
    const std::vector<sv_gate> g = circuit(lattice(3, 4, 8, 5));
    sv_state *s[2] = {nullptr, nullptr};
    for (sv_state *&x : s)
      if (!check(sv_create(12, &o, &x)) || !check(sv_apply_circuit(x, g.data(), g.size()))) return 2;
    st = sv_inner_product(s[0], s[1], out.data());
    for (sv_state *x : s) sv_destroy(x);
  }
  std::printf("status %d after %d passes\n", (int)st, svj::g_passes);
  return st != (fail < 0 ? SV_OK : SV_ERR_TIMEOUT);
}

// One gate list on a handle as a tree's segment (forking its prefix, or storing listed tiles), as a
// whole state, and as a segment again; and the fork of an empty list.
int segments() {
  const sv_options o = options(1);
  sv_state *s = nullptr;
  if (!check(sv_create(12, &o, &s))) return 2;
  s->fresh = false;
  const std::vector<svp::Gate> g = {svp::Gate{svp::K_SX, 3, 0}};
  const std::vector<uint64_t> needed = {5};
  auto apply = [&](int fork, bool listed, const std::vector<svp::Gate> &list) {
    s->fork = fork;
    s->needed = listed ? &needed : nullptr;
    const bool ok = check(svc::apply_gates(s, list));
    s->needed = nullptr;
    return ok && s->fork == 0;
  };
  const bool ok = apply(1, false, g) && apply(0, false, g) && apply(0, true, g) && apply(0, false, g) &&
                  apply(0, false, g) && apply(1, false, g) && apply(0, true, g) && apply(1, false, {});
  sv_destroy(s);
  std::printf("passes %s\n", svj::g_kinds.c_str());
  return !ok || svj::g_kinds != "fwlwwfl";
}

// Amplitudes of a batch, read while the thread's current device is another one.
int other_device() {
  const sv_lattice l = lattice(3, 4, 8, 5);
  const uint64_t bits[2] = {1, 2};
  double out[4];
  g_device = 1;
  if (!check(sv_apply_batch(&l, 1, nullptr, nullptr))) return 2;
  g_device = 0;
  if (!check(sv_batch_amplitudes(0, bits, 2, out))) return 2;
  std::printf("picked on device %d, left on %d\n", svk::g_picked_on, g_device);
  return svk::g_picked_on != 1 || g_device != 0;
}

// The full state from two halves on the tensor cores, whose operand images find no room.
int no_room() {
  const sv_options o = options(0, SV_PREC_TF32X3);
  sv_cut cut;
  std::memset(&cut, 0, sizeof(cut));
  cut.half_a_mask = 0xff;
  const sv_lattice l = lattice(4, 4, 8, 5);
  sv_state *s = nullptr;
  svk::g_outer_tc = true;
  if (!check(sv_create(16, &o, &s))) return 2;
  const bool ok = check(sv_branch_full_state(&l, &cut, &o, s));
  sv_destroy(s);
  return !ok || svk::g_outer != 1;
}

}  // namespace

int main(int argc, char **argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  auto arg = [&](int i) { return argc > i ? std::atoi(argv[i]) : 0; };
  if (what == "uploads") return uploads(arg(2), arg(3));
  if (what == "gave_up") return gave_up(argc > 2 ? argv[2] : "", arg(3));
  if (what == "segments") return segments();
  if (what == "other_device") return other_device();
  if (what == "no_room") return no_room();
  return 3;
}

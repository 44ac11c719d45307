// The host logic of the library (csrc/api.cu) on a CUDA runtime and on kernel
// launchers that only keep a record: each operation with the operations that
// are ordered before it by streams and events.  No GPU, no device memory;
// test_host_order.py builds and drives it.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>

#include "lattice.h"

namespace {

using Order = std::set<int>;

int next_op = 0;
std::map<const void*, Order> streams, events;
std::string record_text;
std::map<std::string, long> knobs;  // set by the test; counted down where a call is to fail

long knob(const char* name) { return knobs[name]; }

cudaError_t fails(const char* name) {  // the n-th call from now
  long& n = knobs[name];
  return n > 0 && --n == 0 ? cudaErrorUnknown : cudaSuccess;
}

void op(const char* name, const void* stream, long a = 0, long b = 0) {
  Order& o = streams[stream];
  char head[96];
  std::snprintf(head, sizeof head, "%d %s %ld %ld", next_op, name, a, b);
  record_text += head;
  for (int k : o) record_text += ' ' + std::to_string(k);
  record_text += '\n';
  o.insert(next_op++);
}

void* handle() {  // never dereferenced
  static uintptr_t h = 0x1000;
  return (void*)(h += 0x1000);
}

}  // namespace

extern "C" {

void fake_reset() {
  next_op = 0;
  streams.clear();
  events.clear();
  record_text.clear();
  knobs.clear();
}
void fake_set(const char* name, long v) { knobs[name] = v; }
const char* fake_record() { return record_text.c_str(); }
void fake_forget() { record_text.clear(); }

// ---- runtime ----
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
  static uintptr_t at = 1ull << 40;
  *p = (void*)at;
  at += (n + 0xffffull) & ~0xffffull;
  return cudaSuccess;
}
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  *p = std::malloc(n);
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  std::memset(a, 0, sizeof *a);
  a->type = cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t s) {
  op("memset", s);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind kind, cudaStream_t s) {
  if (kind == cudaMemcpyDeviceToHost) {
    if (const cudaError_t e = fails("fail_read")) return e;
    op("read", s);
  } else {
    op("copy", s);
  }
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  op("synchronize", s);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)handle();
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  *e = (cudaEvent_t)handle();
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  events[e] = streams[s];
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  streams[s].insert(events[e].begin(), events[e].end());
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  if (const cudaError_t e = fails("fail_capture")) return e;
  op("capture", s);
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  op("captured", s);
  *g = (cudaGraph_t)handle();
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  *x = (cudaGraphExec_t)handle();
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) {
  op("graph", s);
  return cudaSuccess;
}
// api.cu holds no kernels; its registration is empty
void** __cudaRegisterFatBinary(void*) {
  static void* none[1];
  return none;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}

}  // extern "C"

// ---- launchers ----
namespace ianus {

cudaError_t launch_init_i8(Lattice&, int) { return cudaSuccess; }
cudaError_t launch_init_bits(Lattice&, int) { return cudaSuccess; }
cudaError_t launch_sweep_i8(Lattice& l, int c, uint64_t t, int) {
  op("sweep", l.stream, (long)t, c);
  return cudaSuccess;
}
cudaError_t launch_sweep_bits(Lattice& l, int c, uint64_t t, int) {
  if (const cudaError_t e = fails("fail_sweep")) return e;
  op("sweep_bits", l.stream, (long)t, c);
  return cudaSuccess;
}
cudaError_t launch_measure_i8(Lattice& l, int) {
  op("measure", l.stream);
  return cudaSuccess;
}
cudaError_t launch_measure_bits(Lattice& l, int, bool) {
  op("measure", l.stream);
  return cudaSuccess;
}
cudaError_t launch_measure_bits_counts(Lattice& l, bool) {
  op("measure", l.stream);
  return cudaSuccess;
}
bool overlap_apart(const Lattice&, int) { return false; }
cudaError_t launch_overlap_bits(Lattice&) { return cudaSuccess; }
cudaError_t launch_finalize(Lattice& l, int64_t*, int64_t*, int64_t*, uint64_t*, int) {
  op("finalize", l.stream);
  return cudaSuccess;
}
cudaError_t launch_finalize_row(Lattice& l, uint32_t, uint64_t, int) {
  op("finalize", l.stream);
  return cudaSuccess;
}
cudaError_t launch_pt_swap(Lattice& l, uint32_t) {
  op("swap", l.stream);
  return cudaSuccess;
}
cudaError_t launch_build_planes(Lattice& l) {
  op("planes", l.stream);
  return cudaSuccess;
}
cudaError_t launch_set_tick(Lattice&, uint64_t, uint64_t, uint64_t) { return cudaSuccess; }
cudaError_t launch_advance_tick(Lattice&, uint64_t, uint64_t, uint64_t) { return cudaSuccess; }
cudaError_t launch_pack_words(Lattice& l) {
  op("pack_words", l.stream);
  return cudaSuccess;
}
cudaError_t launch_unpack_spins(Lattice& l) {
  op("unpack_spins", l.stream);
  return cudaSuccess;
}
void prepare_sweep_bits(Lattice&, int) {}
int sweep_chains_i8(const Lattice&) { return (int)std::max(1l, knob("chains")); }
int sweep_chains_bits(const Lattice&, int) { return (int)std::max(1l, knob("chains")); }
bool persistent_variant(const Lattice&) { return false; }
bool resident_i8_fits(const Lattice&) { return false; }
bool resident_i8_pays(Lattice&, uint32_t) { return false; }
bool resident_bits_fits(const Lattice&) { return false; }
uint32_t resident_cluster_bits(Lattice&) { return 0; }
bool packed_i8_pays(const Lattice&, uint64_t) { return false; }
size_t packed_mask_bytes(uint32_t, uint64_t) { return 0; }
bool words_pay(const Lattice& l, uint64_t) { return l.words && knob("words"); }
size_t sweep_bits_smem(int R) { return (size_t)R * kPlanes * kMaxClasses * 8; }

}  // namespace ianus

// A stand-in for the runtime's streams and events and for the ledger calls, for host tests of code
// that only enqueues: every enqueued layer call is an operation with a vector clock, so a test can ask
// which operations are ordered before which.  Streams and events are small integers behind pointers.
#include <cuda_runtime.h>
#include <stdint.h>
#include <map>
#include <vector>
#include "../include/routerelay.h"

namespace {
typedef std::map<int, int> Clock;                 // stream -> how many of its operations are done
std::map<int, Clock> g_stream, g_event;
struct Op { int ledger, stream; Clock before; int seq; };
std::vector<Op> g_ops;
int g_next = 1, g_fail_ledger = 0, g_fail_wait = 0;
int id(const void* p) { return (int)(intptr_t)p; }
void join(Clock& into, const Clock& from) {
  for (auto& kv : from) if (into[kv.first] < kv.second) into[kv.first] = kv.second;
}
int enqueue(int ledger, int stream) {
  if (ledger && ledger == g_fail_ledger) return RR_ERR_UNSUPPORTED;
  Clock& c = g_stream[stream];
  Op op{ledger, stream, c, ++c[stream]};
  g_ops.push_back(op);
  return RR_OK;
}
}  // namespace

extern "C" {
// ---- runtime ----
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 1; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)(intptr_t)g_next++; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)(intptr_t)g_next++; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { g_event[id(e)] = g_stream[id(s)]; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  if (g_fail_wait && --g_fail_wait == 0) return cudaErrorInvalidValue;
  join(g_stream[id(s)], g_event[id(e)]);
  return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
// ---- ledger ----
int rr_workspace_bytes(const rr_config*, size_t* a, size_t* b) { *a = *b = 256; return RR_OK; }
int rr_ledger_init(const rr_config* c, void*, size_t, void*, size_t, rr_ledger** out) { *out = (rr_ledger*)(intptr_t)c->k; return RR_OK; }
int rr_ledger_destroy(rr_ledger*) { return RR_OK; }
int rr_ledger_reset(rr_ledger*, void*) { return RR_OK; }
int rr_ledger_status(rr_ledger*, void*, uint32_t* s) { *s = 0; return RR_OK; }
int rr_route_anchor(rr_ledger* L, const void*, const void*, int32_t, void* s) { return enqueue(id(L), id(s)); }
int rr_route_relay(rr_ledger* L, const void*, const void*, int32_t, void* s) { return enqueue(id(L), id(s)); }
// ---- the test's side ----
int fake_op(void* stream) { enqueue(0, id(stream)); return (int)g_ops.size() - 1; }   // work of the caller
void fake_fail(int ledger, int nth_wait) { g_fail_ledger = ledger; g_fail_wait = nth_wait; }
int fake_count(void) { return (int)g_ops.size(); }
int fake_ledger(int op) { return g_ops[op].ledger; }
// is operation a ordered before operation b?
int fake_before(int a, int b) {
  const Op &x = g_ops[a], &y = g_ops[b];
  const auto it = y.before.find(x.stream);
  return it != y.before.end() && it->second >= x.seq;
}
}  // extern "C"

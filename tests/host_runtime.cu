// A CUDA runtime for the host alone, linked under the library's own objects in
// place of the real one, for tests of the host code's memory handling. Device
// memory is host memory, kernels do nothing, and
//   - a copy from memory that was not page-locked is made when its stream is
//     next synchronised (the runtime only promises that it may be made by
//     then): a source whose bytes have changed by then is counted as stale;
//   - the n-th allocation after fake_fail_alloc(n) fails;
//   - every launch that takes PathArgs is checked: the buffers its kernel
//     reads or writes must be live allocations of the size their capacities
//     give, else it is counted as a bad launch;
//   - the next k frames after fake_overflow(k, ...) report that the
//     diffraction lists overflowed.
// Compiled twice: by nvcc the part that knows the library's structures, by the
// host compiler the runtime.
#include <cstddef>

extern "C" bool fake_live(const void* p, size_t n);                      // of a device allocation?
extern "C" void fake_bad_launch(const char* kernel, const char* what);
extern "C" void fake_check_paths(const char* kernel, const void* args);
extern "C" void fake_frame_end(void* counters, bool overflow, const unsigned* n);

#ifdef __CUDACC__

#include <cstring>

#include "../paper_2112_07115_gb300/csrc/paths.cuh"

using namespace dcem;

extern "C" void fake_check_paths(const char* k, const void* args) {
  const PathArgs& a = *static_cast<const PathArgs*>(args);
  auto need = [&](const void* p, size_t n, const char* what) {
    if (n != 0 && !fake_live(p, n)) fake_bad_launch(k, what);
  };
  auto has = [&](const char* s) { return std::strstr(k, s) != nullptr; };
  const size_t nw = (size_t)a.nw;
  if (has("k_hidden_planes")) {  // (a set-up kernel: no frame's buffers)
    need(a.quads, 4 * sizeof(float4) * (size_t)a.bvh.ntris, "wall quads");
    need(a.rplanes, sizeof(RPlane) * (size_t)a.nrp, "planes");
    return;
  }
  need(a.ctr, sizeof(DevCounters), "counters");
  need(a.uniq, sizeof(int) * (size_t)a.ucap, "distinct keys");
  need(a.prec, sizeof(PathRec) * (size_t)a.ucap, "records");
  need(a.bucket_cnt, sizeof(unsigned), "bucket counts");
  need(a.bucket, sizeof(int) * (size_t)a.bucket_cap, "buckets");
  need(a.cand, sizeof(Cand) * (size_t)a.cand_cap, "candidates");
  need(a.hkey, sizeof(unsigned long long) * (size_t)a.hcap, "hash keys");
  need(a.hrep, sizeof(unsigned long long) * (size_t)a.hcap, "hash slots");
  need(a.rx, sizeof(float4) * (size_t)a.nrx, "receivers");
  if (!has("k_diff") && !has("k_refl")) return;
  need(a.wedges, sizeof(Wedge) * nw, "wedges");
  need(a.wf, sizeof(WedgeF) * nw, "FP32 wedges");
  need(a.wtopo, sizeof(WedgeTopo) * nw, "wedge topology");
  need(a.wperm, sizeof(int) * nw, "wedge order");
  need(a.wplace, sizeof(int) * nw, "wedge places");
  need(a.wgbox, 6 * sizeof(float) * ((nw + kWedgeGroup - 1) / kWedgeGroup), "group boxes");
  need(a.dsurv, sizeof(unsigned long long) * (size_t)a.dsurv_cap, "survivors");
  need(a.dexact, sizeof(unsigned long long) * (size_t)a.dsurv_cap, "exact candidates");
  if (a.rplanes) {
    need(a.rplanes, sizeof(RPlane) * (size_t)a.nrp, "planes");
    need(a.rmembers, sizeof(int), "members");
    need(a.rkeys, sizeof(float), "member keys");
  }
  if (a.vis || has("k_refl") || has("visible") || has("k_diff_rel") || has("k_diff_pairs")) {
    need(a.quads, 4 * sizeof(float4) * (size_t)a.bvh.ntris, "wall quads");
    if (a.vis || has("k_refl") || has("visible")) {
      need(a.vis, sizeof(unsigned), "visibility rows");
      need(a.vis_any, sizeof(unsigned) * 2 * (size_t)a.nwc, "visibility words");
      need(a.vis_grp, sizeof(int), "visible groups");
    }
  }
  if (a.drefl2) {
    need(a.rmask, sizeof(unsigned), "masks");
    need(a.wobs_cnt, sizeof(unsigned) * 3 * nw, "side counts");
    need(a.dobs, sizeof(DiffObs) * (size_t)a.dobs_cap, "sides");
  }
  if (has("k_diff_rel") || has("k_diff_pairs") || has("multi") || has("triples")) {
    need(a.drel, (nw * nw + 31) / 32 * sizeof(unsigned), "relation");
    need(a.dseq2, sizeof(int4) * (size_t)a.dseq2_cap, "pairs");
    need(a.dseq3, sizeof(int4) * (size_t)a.dseq3_cap, "triples");
  }
}

extern "C" void fake_frame_end(void* counters, bool overflow, const unsigned* n) {
  DevCounters* c = static_cast<DevCounters*>(counters);
  std::memset(counters, 0, 2 * sizeof(DevCounters));
  if (!overflow) return;
  c->err = ERR_DIFF_OVERFLOW;
  c->n_dsurv = n[0], c->n_dobs = n[1], c->n_dpair = n[2], c->n_dtrip = n[3];
}

#else

#include <cuda_runtime_api.h>
#include <malloc.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
struct Pending {
  void* dst;
  const void* src;
  std::vector<char> bytes;
};
std::map<const char*, size_t>& blocks() {  // device allocations
  static auto* m = new std::map<const char*, size_t>;
  return *m;
}
std::map<const char*, size_t>& pinned() {
  static auto* m = new std::map<const char*, size_t>;
  return *m;
}
std::map<const void*, std::string>& kernels() {
  static auto* m = new std::map<const void*, std::string>;
  return *m;
}
std::vector<Pending>& pending() {
  static auto* v = new std::vector<Pending>;
  return *v;
}
int n_stale, n_bad, n_alloc, fail_at, n_over;
unsigned over[4];
bool capturing;
char bad_text[256];

bool within(const std::map<const char*, size_t>& m, const void* p, size_t n) {
  const char* c = static_cast<const char*>(p);
  auto it = m.upper_bound(c);
  if (it == m.begin()) return false;
  --it;
  return c + n <= it->first + it->second;
}
void drain() {
  for (Pending& p : pending()) {
    if (std::memcmp(p.src, p.bytes.data(), p.bytes.size()) != 0) ++n_stale;
    std::memcpy(p.dst, p.bytes.data(), p.bytes.size());
  }
  pending().clear();
}
cudaError_t take(std::map<const char*, size_t>& m, void** p, size_t n) {
  *p = nullptr;
  ++n_alloc;
  if (fail_at > 0 && --fail_at == 0) return cudaErrorMemoryAllocation;
  *p = std::calloc(n ? n : 1, 1);
  m[static_cast<char*>(*p)] = n;
  return cudaSuccess;
}

}  // namespace

// Freed host memory changes at once.
void operator delete(void* p) noexcept {
  if (p) std::memset(p, 0xdd, malloc_usable_size(p));
  std::free(p);
}
void operator delete(void* p, size_t) noexcept { operator delete(p); }

extern "C" {
bool fake_live(const void* p, size_t n) { return within(blocks(), p, n); }
void fake_bad_launch(const char* kernel, const char* what) {
  if (!n_bad++) std::snprintf(bad_text, sizeof(bad_text), "%s: %s", kernel, what);
}
int fake_stale() { return n_stale; }
int fake_bad() { return n_bad; }
const char* fake_bad_text() { return bad_text; }
int fake_allocs() { return n_alloc; }
void fake_fail_alloc(int n) { fail_at = n; }
void fake_overflow(int frames, unsigned surv, unsigned obs, unsigned pairs, unsigned triples) {
  n_over = frames;
  over[0] = surv, over[1] = obs, over[2] = pairs, over[3] = triples;
}

void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  kernels()[host] = name;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(host));
  return cudaSuccess;
}
static dim3 cfg_grid, cfg_block;
static size_t cfg_smem;
static cudaStream_t cfg_stream;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, cudaStream_t s) {
  cfg_grid = g, cfg_block = b, cfg_smem = m, cfg_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
  *g = cfg_grid, *b = cfg_block, *m = cfg_smem, *static_cast<cudaStream_t*>(s) = cfg_stream;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t) {
  const std::string& name = kernels()[reinterpret_cast<const void*>(k)];
  if (name.find("8PathArgs") != std::string::npos) fake_check_paths(name.c_str(), args[0]);
  if (name.find("k_frame_end") != std::string::npos && !capturing) {
    fake_frame_end(*static_cast<void**>(args[11]), n_over > 0, over);
    if (n_over > 0) --n_over;
  }
  return cudaSuccess;
}

cudaError_t cudaMalloc(void** p, size_t n) { return take(blocks(), p, n); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return take(pinned(), p, n); }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
  *d = h;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  drain();
  blocks().erase(static_cast<char*>(p));
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  pinned().erase(static_cast<char*>(p));
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (within(blocks(), src, n) || within(pinned(), src, n) || !within(blocks(), dst, n)) {
    std::memmove(dst, src, n);
  } else {
    const char* c = static_cast<const char*>(src);
    pending().push_back(Pending{dst, src, std::vector<char>(c, c + n)});
  }
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, cudaMemcpyKind) {
  std::memmove(dst, src, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  if (n != 0 && !within(blocks(), p, n)) fake_bad_launch("memset", "target");
  else std::memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  drain();
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  std::memset(static_cast<void*>(a), 0, sizeof(*a));
  a->type = within(blocks(), p, 1)   ? cudaMemoryTypeDevice
            : within(pinned(), p, 1) ? cudaMemoryTypeHost
                                     : cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static void* m = std::calloc(1 << 20, 1);
  *p = m;
  blocks()[static_cast<char*>(m)] = 1 << 20;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  std::memset(static_cast<void*>(a), 0, sizeof(*a));
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { return *n = 2, cudaSuccess; }
static char handle[1];
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)handle, cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = (cudaEvent_t)handle, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { return *t = 0.0f, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = (cudaStream_t)handle, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return capturing = true, cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  capturing = false;
  return *g = (cudaGraph_t)handle, cudaSuccess;
}
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { return *g = (cudaGraph_t)handle, cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphAddChildGraphNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t, cudaGraph_t) {
  return *n = (cudaGraphNode_t)handle, cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  return *x = (cudaGraphExec_t)handle, cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
}
#endif

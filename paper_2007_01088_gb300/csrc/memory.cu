// Device memory of the library: stream-ordered allocations from a private pool
// of the device, and host-to-device copies of small tables.
//
// A Jacobian, left transformation or density call allocates a few dozen
// temporaries and a few tables per batch of triples, and a serving slot builds
// a context per request.  cudaMalloc and cudaFree cost 10-40 us each, and
// cudaFree waits for the whole device, which made the serving slots take turns
// (a burst of six small requests on four slots: 1630 calls, 59 ms, of which the
// device worked 26 ms).  From the pool both cost 1-2 us and order themselves on
// the calling stream.
//
// The pool keeps at most 1/16 of the device's memory unused while a context or
// a server exists (trimmed at the end of each entry point that freed something)
// and at most KEEP bytes after the last one is gone; cc3_serve_stop gives back
// the rest as well when nothing is left, cc3_memory_release at any time.  Only
// memory whose free the host has seen complete can be trimmed, so the stream of
// the frees is waited for before.  A failed allocation first returns all that is
// unused and tries again.  dev_mem_free counts what the pool holds unused as
// free.
//
// A block that is given back serves the next request at once, so every free is
// ordered after the block's last use: a call's own buffers are freed on its
// stream, and a context's buffers after the event that a call records at its
// end unless it has waited for its work (CallScope), which also orders calls of
// one context on different streams.  Waiting for the whole device instead is
// refused while any stream of it is being captured.  Events are recorded only
// where they are needed: with one per context the pool follows their
// dependencies in every allocation (a burst of six requests 23.7 ms, so 22.2).
#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>
#include <chrono>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>

#include "cc3_internal.h"

namespace cc3 {
namespace {
constexpr size_t KEEP = 1ull << 30;

// Pinned buffers for table uploads: taken when the copy out of them is done.
struct HostBuf {
  char *p;
  cudaEvent_t done;
};
constexpr size_t HOST_BYTES = 256 << 10;
constexpr int HOST_MAX = 64;

// What the library keeps in one device context.  A context that cudaDeviceReset
// destroys takes all of it along: the next one, on the same device, has another
// id and gets a Space of its own.
struct Space {
  unsigned long long id = 0;
  cudaMemPool_t pool = nullptr;  // null where pools are not supported (then cudaMalloc serves)
  cudaStream_t side = nullptr;
  unsigned long long cap = 0;  // unused bytes the pool may keep
  std::atomic<int> live{0};    // contexts and servers
  std::mutex host_mu;
  std::vector<HostBuf> host;  // idle or with a copy in flight (see done)
  int host_made = 0;
};

std::mutex g_mu;
std::vector<Space *> g_spaces;  // few: one per device and reset; they stay
thread_local cudaStream_t t_stream = nullptr;
thread_local int t_depth = 0;           // StreamScopes of this thread
thread_local Space *t_space = nullptr;  // that of the outermost one
thread_local bool t_freed = false;      // something was freed in the outermost one
thread_local bool t_gone = false;       // frees are of memory that went with a reset

int device() {
  int dev = -1;
  cudaGetDevice(&dev);
  return dev;
}

// The id of the device context that the runtime works in (through its driver
// entry points, so that the library does not link the driver library): it
// outlives no reset, while the context's address may return.  0: not known.
unsigned long long context_id() {
  using GetCurrent = CUresult (*)(CUcontext *);
  using GetId = CUresult (*)(CUcontext, unsigned long long *);
  static GetCurrent current = nullptr;
  static GetId id_of = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    auto find = [](const char *name) -> void * {
      void *f = nullptr;
      cudaDriverEntryPointQueryResult q;
      if (cudaGetDriverEntryPointByVersion(name, &f, 12000, cudaEnableDefault, &q) !=
              cudaSuccess ||
          q != cudaDriverEntryPointSuccess) {
        cudaGetLastError();
        return nullptr;
      }
      return f;
    };
    current = reinterpret_cast<GetCurrent>(find("cuCtxGetCurrent"));
    id_of = reinterpret_cast<GetId>(find("cuCtxGetId"));
  });
  if (!current || !id_of) return 0;
  for (int tries = 0; tries < 2; ++tries) {
    CUcontext c = nullptr;
    unsigned long long id = 0;
    if (current(&c) == CUDA_SUCCESS && c && id_of(c, &id) == CUDA_SUCCESS) return id;
    // none is current in this thread yet, or it was reset: the runtime makes one
    if (cudaFree(nullptr) != cudaSuccess) cudaGetLastError();
  }
  return 0;
}

Space *find_space() {
  unsigned long long id = context_id();
  const int dev = device();
  if (id == 0) id = ~0ull - (unsigned long long)dev;  // by device alone
  std::lock_guard<std::mutex> lk(g_mu);
  for (Space *s : g_spaces)
    if (s->id == id) return s;
  Space *s = new Space();
  s->id = id;
  int ok = 0;
  cudaDeviceGetAttribute(&ok, cudaDevAttrMemoryPoolsSupported, dev);
  cudaMemPoolProps p;
  std::memset(&p, 0, sizeof(p));
  p.allocType = cudaMemAllocationTypePinned;
  p.handleTypes = cudaMemHandleTypeNone;
  p.location.type = cudaMemLocationTypeDevice;
  p.location.id = dev;
  cudaMemPool_t pool = nullptr;
  size_t fr = 0, tot = 0;
  if (ok && cudaMemPoolCreate(&pool, &p) == cudaSuccess) {
    cudaMemGetInfo(&fr, &tot);
    // (a release threshold would count the memory in use as well)
    unsigned long long keep = ~0ull;
    s->cap = tot / 16;
    if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess &&
        cudaStreamCreateWithFlags(&s->side, cudaStreamNonBlocking) == cudaSuccess)
      s->pool = pool;
    else
      cudaMemPoolDestroy(pool);
  }
  cudaGetLastError();
  g_spaces.push_back(s);
  return s;
}
Space *space() { return t_depth > 0 && t_space ? t_space : find_space(); }

bool host_take(Space *S, HostBuf *out) {
  std::lock_guard<std::mutex> lk(S->host_mu);
  for (size_t i = 0; i < S->host.size(); ++i)
    if (cudaEventQuery(S->host[i].done) == cudaSuccess) {
      *out = S->host[i];
      S->host[i] = S->host.back();
      S->host.pop_back();
      return true;
    }
  cudaGetLastError();  // cudaErrorNotReady of the queries
  if (S->host_made >= HOST_MAX) return false;
  HostBuf b{nullptr, nullptr};
  if (cudaMallocHost(&b.p, HOST_BYTES) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (cudaEventCreateWithFlags(&b.done, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    cudaFreeHost(b.p);
    return false;
  }
  ++S->host_made;
  *out = b;
  return true;
}
}  // namespace

// Bytes the pool has reserved and those in use; false: not known.
static bool pool_state(cudaMemPool_t pool, unsigned long long *held, unsigned long long *used) {
  if (cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, held) == cudaSuccess &&
      cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, used) == cudaSuccess)
    return true;
  cudaGetLastError();
  return false;
}

StreamScope::StreamScope(cudaStream_t s) : prev(t_stream) {
  t_stream = s;
  if (t_depth == 0) {
    t_space = find_space();
    t_freed = false;
  }
  ++t_depth;
}
StreamScope::~StreamScope() {
  const cudaStream_t s = t_stream;
  t_stream = prev;
  if (--t_depth > 0 || !t_freed) return;
  const Space *S = t_space;
  unsigned long long held = 0, used = 0;
  if (!S->pool || !pool_state(S->pool, &held, &used) || held <= S->cap) return;
  cudaStreamSynchronize(s);  // frees under way count as used
  if (pool_state(S->pool, &held, &used) && held > used + S->cap)
    cudaMemPoolTrimTo(S->pool, used + S->cap);
  cudaGetLastError();
}

bool stream_recording(cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) == cudaSuccess) return cap != cudaStreamCaptureStatusNone;
  cudaGetLastError();  // the legacy stream, while another thread's capture forbids its use
  return true;
}

static bool is_legacy(cudaStream_t s) { return s == nullptr || s == cudaStreamLegacy; }
static bool mark(cc3_ctx *c, cudaStream_t s) {
  if ((c->done || cudaEventCreateWithFlags(&c->done, cudaEventDisableTiming) == cudaSuccess) &&
      cudaEventRecord(c->done, s) == cudaSuccess)
    return true;
  cudaGetLastError();
  return false;
}
// Orders s after the context's last call.
static bool after_last(cc3_ctx *c, cudaStream_t s) {
  if (!c->in_flight || (c->on_legacy && is_legacy(s))) return true;
  if (c->on_legacy && !mark(c, nullptr)) return false;
  if (cudaStreamWaitEvent(s, c->done, 0) == cudaSuccess) return true;
  cudaGetLastError();
  return false;
}

CallScope::CallScope(cc3_ctx *c_, cudaStream_t s_)
    : scope(s_), c(c_), s(s_), recording(stream_recording(s_)) {
  if (recording) return;
  if (!after_last(c, s)) c->unmarked = true;
  c->in_flight = true;
  c->on_legacy = is_legacy(s);
}
void CallScope::complete() {
  if (!recording) c->in_flight = false;
}
CallScope::~CallScope() {
  // the legacy default stream cannot go away: its event can be recorded when needed
  if (recording || (c->in_flight && !c->on_legacy && !mark(c, s))) c->unmarked = true;
}

// Waits for the whole device, which is refused while a stream of it is being
// captured: captures are short, so it tries again for up to ten seconds.
static bool wait_device() {
  for (int i = 0; i < 10000; ++i) {
    const cudaError_t e = cudaDeviceSynchronize();
    cudaGetLastError();
    if (e < cudaErrorStreamCaptureUnsupported || e > cudaErrorStreamCaptureWrongThread)
      return true;  // idle, or lost to an earlier failure
    std::this_thread::sleep_for(std::chrono::milliseconds(1));
  }
  return false;
}

bool ctx_order(cc3_ctx *c, cudaStream_t s) {
  if (c->space != dev_space()) return true;  // its memory and its work went with a reset
  return (!c->unmarked && after_last(c, s)) || wait_device();
}

cudaStream_t ctx_free_stream(cc3_ctx *c) {
  return c->on_legacy && !stream_recording(nullptr) ? nullptr : dev_side_stream();
}

DeviceScope::DeviceScope(int dev) : prev(device()) { cudaSetDevice(dev); }
DeviceScope::~DeviceScope() {
  if (prev >= 0) cudaSetDevice(prev);
}

unsigned long long dev_space() { return space()->id; }
cudaStream_t dev_side_stream() { return space()->side; }

cudaError_t dev_malloc_bytes(void **p, size_t n) {
  *p = nullptr;
  cudaMemPool_t pool = space()->pool;
  if (!pool) return cudaMalloc(p, n);
  // no allocation becomes part of a caller's graph
  if (stream_recording(t_stream)) return cudaErrorStreamCaptureUnsupported;
  cudaError_t e = cudaMallocFromPoolAsync(p, n, pool, t_stream);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    cudaDeviceSynchronize();
    cudaMemPoolTrimTo(pool, 0);
    e = cudaMallocFromPoolAsync(p, n, pool, t_stream);
  }
  if (e != cudaSuccess) *p = nullptr;
  return e;
}

void dev_free(void *p) {
  if (!p || t_gone) return;
  t_freed = true;
  if (!space()->pool) {
    cudaFree(p);
  } else if (cudaFreeAsync(p, t_stream) != cudaSuccess) {
    cudaGetLastError();
    // (a capture on another thread that forbids the legacy stream) cudaFree does
    // not wait for work on a pool's memory; not waited for, it stays allocated
    if (wait_device()) cudaFree(p);
  }
}

size_t dev_mem_free() {
  size_t fr = 0, tot = 0;
  if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (cudaMemPool_t pool = space()->pool) {
    unsigned long long held = 0, used = 0;
    if (pool_state(pool, &held, &used) && held > used) fr += (size_t)(held - used);
  }
  return fr;
}

unsigned long long dev_ctx_born() {
  Space *S = space();
  ++S->live;
  return S->id;
}
void dev_ctx_gone(unsigned long long id, cudaStream_t s) {
  Space *S = space();
  if (id != S->id || --S->live > 0) return;
  cudaStreamSynchronize(s);
  if (S->pool) cudaMemPoolTrimTo(S->pool, KEEP);
  cudaGetLastError();
}
void dev_give_back() {
  Space *S = space();
  if (S->live > 0 || !S->pool) return;
  cudaMemPoolTrimTo(S->pool, 0);
  cudaGetLastError();
}

GoneScope::GoneScope(bool gone) : prev(t_gone) { t_gone = gone; }
GoneScope::~GoneScope() { t_gone = prev; }
bool dev_gone() { return t_gone; }

int dev_upload(void *dst, const void *src, size_t n, cudaStream_t s) {
  if (n == 0) return CC3_OK;
  HostBuf b;
  Space *S = space();
  if (n <= HOST_BYTES && host_take(S, &b)) {
    std::memcpy(b.p, src, n);
    cudaError_t e = cudaMemcpyAsync(dst, b.p, n, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaEventRecord(b.done, s);
    if (e != cudaSuccess) cudaStreamSynchronize(s);  // no copy out of the buffer is left
    {
      std::lock_guard<std::mutex> lk(S->host_mu);
      S->host.push_back(b);
    }
    return e == cudaSuccess ? CC3_OK : CC3_FAIL(CC3_ERR_CUDA, cudaGetErrorString(e));
  }
  // large tables: the copy is complete on return
  cudaError_t e = cudaMemcpyAsync(dst, src, n, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e == cudaSuccess ? CC3_OK : CC3_FAIL(CC3_ERR_CUDA, cudaGetErrorString(e));
}

}  // namespace cc3

extern "C" int cc3_memory_release(void) {
  using namespace cc3;
  Space *S = space();
  if (cudaDeviceSynchronize() != cudaSuccess)  // what is being freed can be given back too
    return CC3_FAIL(CC3_ERR_CUDA, cudaGetErrorString(cudaGetLastError()));
  if (S->pool && cudaMemPoolTrimTo(S->pool, 0) != cudaSuccess)
    return CC3_FAIL(CC3_ERR_CUDA, cudaGetErrorString(cudaGetLastError()));
  std::lock_guard<std::mutex> lk(S->host_mu);
  for (HostBuf &b : S->host) {  // (no copy out of them is left)
    cudaEventDestroy(b.done);
    cudaFreeHost(b.p);
  }
  S->host_made -= (int)S->host.size();
  S->host.clear();
  return CC3_OK;
}

extern "C" int cc3_debug_memory(size_t *held, size_t *used, size_t *peak) {
  using namespace cc3;
  if (!held || !used || !peak) return CC3_ERR_ARG;
  cudaMemPool_t pool = space()->pool;
  if (!pool) return CC3_ERR_UNSUPPORTED;
  unsigned long long h = 0, u = 0, p = 0, zero = 0;
  if (cudaDeviceSynchronize() != cudaSuccess || !pool_state(pool, &h, &u) ||
      cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemHigh, &p) != cudaSuccess ||
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrUsedMemHigh, &zero) != cudaSuccess)
    return CC3_FAIL(CC3_ERR_CUDA, cudaGetErrorString(cudaGetLastError()));
  *held = h;
  *used = u;
  *peak = p;
  return CC3_OK;
}

// Device memory of the library's objects: an account with an optional limit,
// and freed blocks kept for the next allocation.  The account counts blocks as
// they were allocated (block_size), not what their buffers asked for; under a
// limit a buffer gets exactly what it asks for, from a block of that size or a
// new one, and idle blocks count as long as they are there.
//
// Why blocks are kept: a P build makes about 30 allocations, most of them
// temporaries.  On GB300 cudaMalloc takes 35 us and cudaFree 31 us (a wait for
// the whole device) to 160 us (256 MB); taking a kept block and giving it back
// takes 2 us.  (CUDA's own pools were slower: with every layout on a stream of
// its own, cudaMallocFromPoolAsync grew by 3 us a call with every stream that
// had freed memory, to 2 ms a build after 20 layouts.)
//
// Rules.  An allocation belongs to the stream of the object that makes it
// (alloc_stream(): set by every entry point for its call); its uses are
// ordered on that stream.  Giving it back records an event there, and whoever
// takes the block next makes its own stream wait for that event, so a block
// never changes hands before the work that used it is done, whatever the
// streams and threads (cudaStreamPerThread names another stream in every
// thread, so its buffers are not kept).  At most kIdleBytes are kept per device
// between calls: what an entry point's temporaries leave above that goes back
// when the entry point returns (the end of its AllocScope, which stands before
// them), what is freed outside of one at once.  All idle blocks go back to the
// device when an allocation fails and when the library's memory limit is set.
// Blocks belong to one CUDA context (recognised by its id): what a context
// destroyed by cudaDeviceReset held is not touched again.  A buffer carries its block's size,
// device and context itself, so it goes back where it came from whatever the
// freeing thread has selected, and nothing about it is kept here meanwhile.
#include <atomic>
#include <list>
#include <mutex>
#include <vector>

#include "tsgne_internal.cuh"

namespace tsgne {

namespace {

std::atomic<int64_t> g_used{0};   // bytes of the blocks in use, as they were allocated
std::atomic<int64_t> g_limit{0};  // on those and the idle ones together; 0: none

constexpr size_t kIdleBytes = (size_t)256 << 20;  // freed bytes kept (0.1 % of a GB300)
thread_local bool t_over = false;                 // this thread's call left a device with more than that

struct Block {
  void* p;
  size_t bytes;
  cudaEvent_t done;  // recorded on the last owner's stream when the block came back
};
struct Blocks {
  unsigned long long context = 0;
  int device = 0;
  std::list<Block> idle;  // longest idle first
  size_t idle_bytes = 0;
  std::vector<cudaEvent_t> spare;
};
std::mutex g_mu;

// Never destroyed: objects may be freed after main.
std::list<Blocks>& all_blocks() {
  static std::list<Blocks>* v = new std::list<Blocks>();
  return *v;
}

// Id of the current context, unique for the life of the process.
bool context_id(unsigned long long* id) {
  typedef int (*Fn)(void*, unsigned long long*);
  static const Fn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<Fn>(p);
  }();
  return fn != nullptr && fn(nullptr, id) == 0;
}

// Selects a device with its context current, and the caller's device again at the end.
struct OnDevice {
  int prev = -1;
  unsigned long long context = 0;  // the current context; ok: there is one
  bool ok;
  explicit OnDevice(int device) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    ok = prev == device && context_id(&context);  // a new thread has no context until it selects its device
    if (!ok) ok = cudaSetDevice(device) == cudaSuccess && context_id(&context);
    if (prev == device) prev = -1;
  }
  ~OnDevice() {
    if (prev >= 0) cudaSetDevice(prev);
  }
  OnDevice(const OnDevice&) = delete;
  OnDevice& operator=(const OnDevice&) = delete;
};

// The current context's blocks.
Blocks& blocks_of(unsigned long long id) {
  for (Blocks& b : all_blocks())
    if (b.context == id) return b;
  int device = 0;
  cudaGetDevice(&device);
  all_blocks().emplace_back();
  all_blocks().back().context = id;
  all_blocks().back().device = device;
  return all_blocks().back();
}

// Sizes of blocks, so that similar requests share them: quarter octaves from
// 4 KiB, multiples of 2 MiB from there (the pages that cudaMalloc maps).
constexpr size_t kPage = (size_t)2 << 20;
size_t block_size(size_t bytes) {
  size_t step = 1024;
  while (8 * step < bytes && step < kPage) step *= 2;
  return (bytes + step - 1) / step * step;
}
// Whether an idle block serves a request of want bytes: up to a quarter more.
// (A sixteenth above 2 MiB makes a call need so many blocks of its own
// that they pass the bound and are allocated anew each time: P by walks on
// 100,000 nodes takes 3.80 ms instead of 3.58, twice the size 3.46.)
bool serves(size_t block, size_t want) { return block >= want && block - want <= want / 4; }

void keep_event(Blocks& b, cudaEvent_t ev) {
  try {
    b.spare.push_back(ev);
  } catch (const std::bad_alloc&) {
    cudaEventDestroy(ev);
  }
}

// Returns idle blocks to the device until at most keep bytes are left: the
// longest idle one that is enough by itself, else the longest idle one and so
// on, so that few of the blocks that a repeated call wants have to be allocated
// again.
void shrink(Blocks& b, size_t keep) {
  while (b.idle_bytes > keep) {
    auto it = b.idle.begin();
    while (it != b.idle.end() && it->bytes < b.idle_bytes - keep) ++it;
    if (it == b.idle.end()) it = b.idle.begin();
    const Block k = *it;
    b.idle.erase(it);
    b.idle_bytes -= k.bytes;
    cudaEventSynchronize(k.done);
    cudaFree(k.p);
    keep_event(b, k.done);
  }
}

// Every context's idle blocks down to keep bytes; those of a context that can
// no longer be selected stay where they are.
void shrink_all(size_t keep) {
  unsigned long long id = 0;
  context_id(&id);
  for (Blocks& b : all_blocks()) {
    if (b.idle_bytes <= keep) continue;
    if (b.context == id) {
      shrink(b, keep);
      continue;
    }
    OnDevice on(b.device);
    if (on.ok && on.context == b.context) shrink(b, keep);
  }
}

// Whether the limit leaves room for a block of bytes in use beside the others;
// fresh: one that is not among the idle ones yet, which then make way for it.
bool within_limit(size_t bytes, bool fresh) {
  const int64_t lim = g_limit.load();
  if (lim <= 0) return true;
  if (g_used.load() + (int64_t)bytes > lim) return false;
  if (!fresh) return true;
  int64_t idle = 0;
  for (const Blocks& b : all_blocks()) idle += (int64_t)b.idle_bytes;
  if (idle > 0 && g_used.load() + idle + (int64_t)bytes > lim) shrink_all(0);
  return true;
}

cudaError_t fresh_block(DevMem* m, Blocks* b, size_t bytes) {
  cudaError_t e = cudaMalloc(&m->p, bytes);
  if (e == cudaErrorMemoryAllocation && b != nullptr && b->idle_bytes > 0) {
    cudaGetLastError();
    shrink(*b, 0);
    e = cudaMalloc(&m->p, bytes);
  }
  m->bytes = bytes;
  return e;
}

// A block for bytes (cudaErrorMemoryAllocation with m->bytes = 0: the limit forbids it).
cudaError_t take(DevMem* m, size_t bytes) {
  std::lock_guard<std::mutex> lk(g_mu);
  Blocks* const b = m->stream ? &blocks_of(m->context) : nullptr;
  // Exactly what is asked for while a limit is set, so that rounding refuses
  // nothing, and where the block can never be kept.
  const bool exact = b == nullptr || g_limit.load() > 0 || bytes > kIdleBytes;
  const size_t want = exact ? bytes : block_size(bytes);
  if (b != nullptr) {
    auto best = b->idle.end();
    for (auto it = b->idle.begin(); it != b->idle.end(); ++it)
      if ((exact ? it->bytes == want : serves(it->bytes, want)) && (best == b->idle.end() || it->bytes < best->bytes))
        best = it;
    if (best != b->idle.end()) {
      const Block k = *best;
      if (!within_limit(k.bytes, false)) return cudaErrorMemoryAllocation;
      if (cudaStreamWaitEvent(m->stream, k.done, 0) == cudaSuccess) {
        b->idle.erase(best);
        b->idle_bytes -= k.bytes;
        keep_event(*b, k.done);
        m->p = k.p;
        m->bytes = k.bytes;
        g_used += (int64_t)k.bytes;
        return cudaSuccess;
      }
      cudaGetLastError();
    }
  }
  if (!within_limit(want, true)) return cudaErrorMemoryAllocation;
  cudaError_t e = fresh_block(m, b, want);
  if (e == cudaErrorMemoryAllocation && want > bytes) {
    cudaGetLastError();
    e = fresh_block(m, b, bytes);
  }
  if (e == cudaSuccess) g_used += (int64_t)m->bytes;
  return e;
}

// False if the block has to be freed by the caller.
bool give_back(const DevMem& m) {
  if (m.bytes > kIdleBytes) return false;
  std::lock_guard<std::mutex> lk(g_mu);
  Blocks& b = blocks_of(m.context);
  cudaEvent_t ev = nullptr;
  if (!b.spare.empty()) {
    ev = b.spare.back();
    b.spare.pop_back();
  } else if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (cudaEventRecord(ev, m.stream) != cudaSuccess) {
    cudaGetLastError();
    keep_event(b, ev);
    return false;
  }
  try {
    b.idle.push_back(Block{m.p, m.bytes, ev});
  } catch (const std::bad_alloc&) {
    keep_event(b, ev);
    return false;
  }
  b.idle_bytes += m.bytes;
  g_used -= (int64_t)m.bytes;
  if (b.idle_bytes > kIdleBytes) {
    if (alloc_stream()) t_over = true;  // the end of the scope sees to it
    else shrink(b, kIdleBytes);
  }
  return true;
}

}  // namespace

cudaStream_t& alloc_stream() {
  thread_local cudaStream_t s = nullptr;
  return s;
}

tsgne_status device_alloc(DevMem* m, size_t bytes) {
  *m = DevMem{};
  m->stream = alloc_stream();
  if (m->stream == cudaStreamPerThread) m->stream = nullptr;  // orders nothing beyond this thread
  if (m->stream && !context_id(&m->context)) m->stream = nullptr;
  cudaError_t e;
  try {
    e = take(m, bytes);
  } catch (const std::bad_alloc&) {  // no host memory for the list: a block without it
    m->stream = nullptr;
    e = take(m, bytes);
  }
  if (e == cudaSuccess) return TSGNE_OK;
  const bool limit = m->bytes == 0;
  *m = DevMem{};
  if (!limit) return cuda_fail(e, "cudaMalloc", __FILE__, __LINE__);
  last_msg() = "device memory limit reached (tsgne_set_device_memory_limit)";
  return TSGNE_ERR_OOM;
}

void device_free(const DevMem& m) {
  if (m.stream) {
    unsigned long long id = 0;
    if (context_id(&id) && id == m.context) {
      if (give_back(m)) return;
    } else {  // another device is selected, or the thread has no context
      int device = -1;
      {
        std::lock_guard<std::mutex> lk(g_mu);
        for (const Blocks& b : all_blocks())
          if (b.context == m.context) device = b.device;
      }
      if (device >= 0) {
        OnDevice on(device);
        if (on.ok && on.context == m.context && give_back(m)) return;
      }
    }
  }
  cudaFree(m.p);
  g_used -= (int64_t)m.bytes;
}

int64_t idle_device_bytes() {
  unsigned long long id = 0;
  if (!context_id(&id)) return 0;
  std::lock_guard<std::mutex> lk(g_mu);
  for (const Blocks& b : all_blocks())
    if (b.context == id) return (int64_t)b.idle_bytes;
  return 0;
}

void trim_idle_blocks() {
  if (!t_over) return;
  t_over = false;
  std::lock_guard<std::mutex> lk(g_mu);
  shrink_all(kIdleBytes);
}

}  // namespace tsgne

extern "C" void tsgne_set_device_memory_limit(int64_t bytes) {
  std::lock_guard<std::mutex> lk(tsgne::g_mu);
  tsgne::g_limit.store(bytes > 0 ? bytes : 0);
  tsgne::shrink_all(0);
}

extern "C" int64_t tsgne_device_memory_in_use(void) { return tsgne::g_used.load(); }

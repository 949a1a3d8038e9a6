// Device memory of the library's objects: an account with an optional limit,
// and freed blocks kept for the next allocation.
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
// streams and threads.  At most kIdleBytes are kept per device, the longest
// idle block goes first: what an entry point's temporaries leave above that
// goes back when the entry point returns (the end of its AllocScope, which
// stands before them), what is freed outside of one at once.  All idle blocks
// go back to the device when
// an allocation fails and when the library's memory limit is set.  Blocks
// belong to one CUDA context (recognised by its id): what a context destroyed
// by cudaDeviceReset held is forgotten.  A buffer carries its block's size,
// device and context itself, so it goes back where it came from whatever the
// freeing thread has selected, and nothing about it is kept here meanwhile.
#include <atomic>
#include <list>
#include <mutex>
#include <vector>

#include "tsgne_internal.cuh"

namespace tsgne {

namespace {

std::atomic<int64_t> g_dev_bytes{0};
std::atomic<int64_t> g_dev_limit{0};  // 0: no limit

constexpr size_t kIdleBytes = (size_t)256 << 20;  // freed bytes kept (0.1 % of a GB300)
std::atomic<bool> g_over{false};                  // a device may hold more than that

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

Blocks& blocks_of(unsigned long long id, int device) {
  for (Blocks& b : all_blocks())
    if (b.context == id) return b;
  all_blocks().emplace_back();
  all_blocks().back().context = id;
  all_blocks().back().device = device;
  return all_blocks().back();
}

// Sizes of blocks: quarter octaves from 4 KiB, so that similar requests share blocks.
size_t block_size(size_t bytes) {
  size_t step = 1024;
  while (8 * step < bytes) step *= 2;
  return (bytes + step - 1) / step * step;
}

// Returns idle blocks to the device, longest idle first, until at most keep bytes are left.
void shrink(Blocks& b, size_t keep) {
  while (b.idle_bytes > keep) {
    const Block k = b.idle.front();
    b.idle.pop_front();
    b.idle_bytes -= k.bytes;
    cudaEventSynchronize(k.done);
    cudaFree(k.p);
    b.spare.push_back(k.done);
  }
}

cudaError_t take(DevMem* m, size_t bytes) {
  std::lock_guard<std::mutex> lk(g_mu);
  Blocks& b = blocks_of(m->context, m->device);
  const size_t want = block_size(bytes);
  auto best = b.idle.end();
  for (auto it = b.idle.begin(); it != b.idle.end(); ++it)  // at most twice the size asked for
    if (it->bytes >= want && it->bytes <= 2 * want && (best == b.idle.end() || it->bytes < best->bytes)) best = it;
  if (best != b.idle.end()) {
    const Block k = *best;
    b.spare.reserve(b.spare.size() + 1);  // before anything changes
    if (cudaStreamWaitEvent(m->stream, k.done, 0) == cudaSuccess) {
      b.idle.erase(best);
      b.idle_bytes -= k.bytes;
      b.spare.push_back(k.done);
      m->p = k.p;
      m->bytes = k.bytes;
      return cudaSuccess;
    }
    cudaGetLastError();
  }
  cudaError_t e = cudaMalloc(&m->p, want);
  if (e == cudaErrorMemoryAllocation && b.idle_bytes > 0) {
    cudaGetLastError();
    shrink(b, 0);
    e = cudaMalloc(&m->p, want);
  }
  m->bytes = want;
  return e;
}

// False if the block has to be freed by the caller.
bool give_back(const DevMem& m) {
  if (m.bytes > kIdleBytes) return false;
  std::lock_guard<std::mutex> lk(g_mu);
  Blocks& b = blocks_of(m.context, m.device);
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
    b.spare.push_back(ev);
    return false;
  }
  b.idle.push_back(Block{m.p, m.bytes, ev});
  b.idle_bytes += m.bytes;
  if (b.idle_bytes > kIdleBytes) {
    if (alloc_stream()) g_over = true;  // the end of the scope sees to it
    else shrink(b, kIdleBytes);
  }
  return true;
}

// Every context's idle blocks; a context that is no longer its device's is forgotten.
void trim_to(size_t keep) {
  std::lock_guard<std::mutex> lk(g_mu);
  for (auto b = all_blocks().begin(); b != all_blocks().end();) {
    if (b->idle_bytes > keep) {
      OnDevice on(b->device);
      if (!on.ok || on.context != b->context) {
        b = all_blocks().erase(b);
        continue;
      }
      shrink(*b, keep);
    }
    ++b;
  }
}

}  // namespace

cudaStream_t& alloc_stream() {
  thread_local cudaStream_t s = nullptr;
  return s;
}

bool device_bytes_reserve(size_t bytes) {
  const int64_t b = (int64_t)bytes;
  const int64_t lim = g_dev_limit.load();
  int64_t cur = g_dev_bytes.load();
  do {
    if (lim > 0 && cur + b > lim) return false;
  } while (!g_dev_bytes.compare_exchange_weak(cur, cur + b));
  return true;
}

void device_bytes_release(size_t bytes) { g_dev_bytes.fetch_sub((int64_t)bytes); }

cudaError_t device_alloc(DevMem* m, size_t bytes) {
  *m = DevMem{};
  const cudaStream_t s = alloc_stream();
  if (!s || cudaGetDevice(&m->device) != cudaSuccess || !context_id(&m->context)) return cudaMalloc(&m->p, bytes);
  m->stream = s;
  try {
    return take(m, bytes);
  } catch (const std::bad_alloc&) {  // no host memory for the list: CUDA's own answer decides
    m->stream = nullptr;
    return cudaMalloc(&m->p, bytes);
  }
}

void device_free(const DevMem& m) {
  if (m.stream) {
    try {
      OnDevice on(m.device);
      if (on.ok && on.context == m.context && give_back(m)) return;
    } catch (const std::bad_alloc&) {
    }
  }
  cudaFree(m.p);
}

void trim_idle_blocks() {
  if (g_over.exchange(false)) trim_to(kIdleBytes);
}
void release_idle_blocks() { trim_to(0); }

}  // namespace tsgne

extern "C" void tsgne_set_device_memory_limit(int64_t bytes) {
  tsgne::g_dev_limit.store(bytes > 0 ? bytes : 0);
  tsgne::release_idle_blocks();
}

extern "C" int64_t tsgne_device_memory_in_use(void) { return tsgne::g_dev_bytes.load(); }

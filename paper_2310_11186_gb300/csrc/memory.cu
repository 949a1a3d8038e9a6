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
// idle block goes first; trim_pool() sees to that at the end of every build
// and with every object destroyed.  All idle blocks go back to the device when
// an allocation fails and when the library's memory limit is set.  Blocks
// belong to one CUDA context (recognised by its id): what a context destroyed
// by cudaDeviceReset held is forgotten.
#include <atomic>
#include <list>
#include <mutex>
#include <unordered_map>
#include <vector>

#include "tsgne_internal.cuh"

namespace tsgne {

namespace {

std::atomic<int64_t> g_dev_bytes{0};
std::atomic<int64_t> g_dev_limit{0};  // 0: no limit

constexpr size_t kIdleBytes = (size_t)256 << 20;  // freed bytes kept (0.1 % of a GB300)

struct Block {
  void* p;
  size_t bytes;
  cudaEvent_t done;  // recorded on the last owner's stream when the block came back
};
struct Blocks {
  unsigned long long context = 0;
  std::list<Block> idle;  // longest idle first
  size_t idle_bytes = 0;
  std::unordered_map<void*, size_t> lent;  // sizes of the blocks in use
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

Blocks& blocks_of(unsigned long long id) {
  for (Blocks& b : all_blocks())
    if (b.context == id) return b;
  all_blocks().emplace_back();
  all_blocks().back().context = id;
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

cudaError_t take(void** p, size_t bytes, cudaStream_t s, unsigned long long id) {
  std::lock_guard<std::mutex> lk(g_mu);
  Blocks& b = blocks_of(id);
  const size_t want = block_size(bytes);
  auto best = b.idle.end();
  for (auto it = b.idle.begin(); it != b.idle.end(); ++it)  // at most twice the size asked for
    if (it->bytes >= want && it->bytes <= 2 * want && (best == b.idle.end() || it->bytes < best->bytes)) best = it;
  if (best != b.idle.end()) {
    const Block k = *best;
    if (cudaStreamWaitEvent(s, k.done, 0) == cudaSuccess) {
      b.lent.emplace(k.p, k.bytes);
      b.idle.erase(best);
      b.idle_bytes -= k.bytes;
      b.spare.push_back(k.done);
      *p = k.p;
      return cudaSuccess;
    }
    cudaGetLastError();
  }
  cudaError_t e = cudaMalloc(p, want);
  if (e == cudaErrorMemoryAllocation && b.idle_bytes > 0) {
    cudaGetLastError();
    shrink(b, 0);
    e = cudaMalloc(p, want);
  }
  if (e == cudaSuccess) {
    try {
      b.lent.emplace(*p, want);
    } catch (...) {
      cudaFree(*p);
      throw;
    }
  }
  return e;
}

// False if the block has to be freed by the caller.
bool give_back(void* p, cudaStream_t s, unsigned long long id) {
  std::lock_guard<std::mutex> lk(g_mu);
  Blocks& b = blocks_of(id);
  const auto it = b.lent.find(p);
  if (it == b.lent.end()) return false;
  const size_t bytes = it->second;
  b.lent.erase(it);
  if (bytes > kIdleBytes) return false;
  cudaEvent_t ev = nullptr;
  if (!b.spare.empty()) {
    ev = b.spare.back();
    b.spare.pop_back();
  } else if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (cudaEventRecord(ev, s) != cudaSuccess) {
    cudaGetLastError();
    b.spare.push_back(ev);
    return false;
  }
  b.idle.push_back(Block{p, bytes, ev});
  b.idle_bytes += bytes;
  return true;
}

void trim_to(size_t keep) {
  unsigned long long id = 0;
  if (!context_id(&id)) return;
  std::lock_guard<std::mutex> lk(g_mu);
  for (Blocks& b : all_blocks())
    if (b.context == id) shrink(b, keep);
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

cudaError_t device_alloc(void** p, size_t bytes, cudaStream_t* owner) {
  const cudaStream_t s = alloc_stream();
  unsigned long long id = 0;
  *owner = nullptr;
  if (!s || !context_id(&id)) return cudaMalloc(p, bytes);
  try {
    const cudaError_t e = take(p, bytes, s, id);
    if (e == cudaSuccess) *owner = s;
    return e;
  } catch (const std::bad_alloc&) {  // no host memory for the list: CUDA's own answer decides
    return cudaMalloc(p, bytes);
  }
}

void device_free(void* p, cudaStream_t owner) {
  unsigned long long id = 0;
  if (owner && context_id(&id)) {
    try {
      if (give_back(p, owner, id)) return;
    } catch (const std::bad_alloc&) {
    }
  }
  cudaFree(p);
}

void trim_pool() { trim_to(kIdleBytes); }
void release_idle_blocks() { trim_to(0); }

}  // namespace tsgne

extern "C" void tsgne_set_device_memory_limit(int64_t bytes) {
  tsgne::g_dev_limit.store(bytes > 0 ? bytes : 0);
  tsgne::release_idle_blocks();
}

extern "C" int64_t tsgne_device_memory_in_use(void) { return tsgne::g_dev_bytes.load(); }

// The calls of the CUDA runtime that memory.cu makes, over two pretended
// devices with one context each, and scenarios over the library's buffers.
// Addresses are handed out lowest first, so that a freed address comes back;
// a thread has no context until it selects a device.  Every buffer's bytes
// are checked against what its address was allocated with.
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "tsgne_internal.cuh"

namespace fake {
std::mutex mu;
struct Allocation {
  size_t bytes;
  int device;
};
std::map<uintptr_t, Allocation> live;
struct Event {
  int device;
  cudaStream_t on;
};
thread_local int device = 0;
thread_local bool bound = false;  // whether the thread has a context
int bad = 0;
long mallocs = 0, frees = 0;
size_t capacity = (size_t)1 << 40;

size_t held(int dev = -1) {
  std::lock_guard<std::mutex> lk(mu);
  size_t s = 0;
  for (auto& a : live)
    if (dev < 0 || a.second.device == dev) s += a.second.bytes;
  return s;
}
int context_id(void*, unsigned long long* id) {
  if (!bound) return 201;  // invalid context
  *id = 1000 + device;
  return 0;
}
}  // namespace fake

#define EXPECT(c)                                                          \
  do {                                                                     \
    if (!(c)) {                                                            \
      std::fprintf(stderr, "line %d: not true: %s\n", __LINE__, #c);       \
      std::exit(1);                                                        \
    }                                                                      \
  } while (0)

extern "C" {
cudaError_t CUDARTAPI cudaGetDevice(int* d) {
  *d = fake::device;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaSetDevice(int d) {
  if (d < 0 || d > 1) return cudaErrorInvalidDevice;
  fake::device = d;
  fake::bound = true;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMalloc(void** p, size_t bytes) {
  fake::bound = true;
  size_t all = fake::held(fake::device);
  std::lock_guard<std::mutex> lk(fake::mu);
  if (all + bytes > fake::capacity) return cudaErrorMemoryAllocation;
  uintptr_t at = (uintptr_t)(fake::device + 1) << 44;
  for (auto& a : fake::live) {
    if (a.second.device != fake::device) continue;
    if (at + bytes <= a.first) break;
    at = (a.first + a.second.bytes + 511) / 512 * 512;
  }
  fake::live[at] = {bytes, fake::device};
  ++fake::mallocs;
  *p = reinterpret_cast<void*>(at);
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaFree(void* p) {
  std::lock_guard<std::mutex> lk(fake::mu);
  if (fake::live.erase(reinterpret_cast<uintptr_t>(p)) == 0) ++fake::bad;
  ++fake::frees;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaEventCreateWithFlags(cudaEvent_t* e, unsigned int) {
  fake::bound = true;
  *e = reinterpret_cast<cudaEvent_t>(new fake::Event{fake::device, nullptr});
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaEventDestroy(cudaEvent_t e) {
  delete reinterpret_cast<fake::Event*>(e);
  return cudaSuccess;
}
// streams 100..199 belong to device 0, 200..299 to device 1
static int device_of(cudaStream_t s) { return (int)(reinterpret_cast<uintptr_t>(s) / 100) - 1; }
cudaError_t CUDARTAPI cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  auto* v = reinterpret_cast<fake::Event*>(e);
  if (reinterpret_cast<uintptr_t>(s) >= 100 && device_of(s) != v->device) return cudaErrorInvalidResourceHandle;
  v->on = s;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned int) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaGetLastError(void) { return cudaSuccess; }
const char* CUDARTAPI cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t CUDARTAPI cudaMemGetInfo(size_t* free, size_t* total) {
  *total = fake::capacity;
  *free = fake::capacity - fake::held(fake::device);
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaStreamCreateWithFlags(cudaStream_t* s, unsigned int) {
  *s = reinterpret_cast<cudaStream_t>((uintptr_t)150);
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaGetDriverEntryPointByVersion(const char* symbol, void** fn, unsigned int, unsigned long long,
                                                       cudaDriverEntryPointQueryResult* q) {
  EXPECT(std::strcmp(symbol, "cuCtxGetId") == 0);
  *fn = reinterpret_cast<void*>(&fake::context_id);
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}  // extern "C"

namespace tsgne {
std::string& last_msg() {
  static thread_local std::string m;
  return m;
}
tsgne_status cuda_fail(cudaError_t e, const char*, const char*, int) {
  return e == cudaErrorMemoryAllocation ? TSGNE_ERR_OOM : TSGNE_ERR_CUDA;
}
}  // namespace tsgne

using tsgne::AllocScope;
using Buf = tsgne::DevBuf<unsigned char>;

// A batch whose members hold what the server estimates for them.
struct tsgne_member {
  Buf mem;
};
struct tsgne_batch {
  std::vector<std::unique_ptr<tsgne_member>> members;
};
extern "C" {
tsgne_status tsgne_batch_create(tsgne_batch** out, const tsgne_config*, int32_t, void*) {
  *out = new tsgne_batch();
  return TSGNE_OK;
}
void tsgne_batch_destroy(tsgne_batch* b) { delete b; }
const char* tsgne_batch_last_error(const tsgne_batch*) { return ""; }
const char* tsgne_last_error(const tsgne_ctx*) { return ""; }
const char* tsgne_status_string(tsgne_status) { return ""; }
tsgne_status tsgne_batch_prepare(tsgne_batch*, int32_t n, const int64_t* rp, const int32_t*, const float*, int32_t,
                                 const float*, int32_t, int32_t, void* s, tsgne_member** out) {
  AllocScope as(static_cast<cudaStream_t>(s));
  *out = new tsgne_member();
  return (*out)->mem.alloc((size_t)tsgne_server_estimate_bytes(n, 2 * rp[n], 1));
}
tsgne_status tsgne_batch_attach(tsgne_batch* b, tsgne_member* m, int32_t* id) {
  *id = (int32_t)b->members.size();
  b->members.emplace_back(m);
  return TSGNE_OK;
}
void tsgne_batch_discard(tsgne_member* m) { delete m; }
tsgne_status tsgne_batch_remove(tsgne_batch* b, int32_t id) {
  b->members[id].reset();
  return TSGNE_OK;
}
tsgne_status tsgne_batch_set_active(tsgne_batch*, int32_t, int32_t) { return TSGNE_OK; }
tsgne_status tsgne_batch_run(tsgne_batch*, int32_t) { return TSGNE_OK; }
tsgne_status tsgne_batch_get_Y(tsgne_batch*, int32_t, float*, int32_t* iter, int32_t) {
  *iter = 20;
  return TSGNE_OK;
}
}  // extern "C"

static cudaStream_t stream(int k) { return reinterpret_cast<cudaStream_t>((uintptr_t)k); }
static void holds(const Buf& b) {  // the buffer lies within one allocation
  std::lock_guard<std::mutex> lk(fake::mu);
  auto it = fake::live.find(reinterpret_cast<uintptr_t>(b.get()));
  EXPECT(it != fake::live.end());
  EXPECT(b.n <= it->second.bytes);
}
static tsgne_status take(Buf& b, size_t bytes, int s) {
  AllocScope as(stream(s));
  return b.alloc(bytes);
}

constexpr size_t KiB = 1 << 10, MiB = 1 << 20;

// A buffer freed where its device is not the current one, or where the thread
// has no context, leaves nothing behind that a later buffer could be given.
static void freed_elsewhere(bool fresh_thread) {
  EXPECT(cudaSetDevice(0) == cudaSuccess);
  auto a = std::make_unique<Buf>();
  EXPECT(take(*a, MiB, 100) == TSGNE_OK);
  if (fresh_thread) {
    std::thread([&] { a.reset(); }).join();
  } else {
    EXPECT(cudaSetDevice(1) == cudaSuccess);
    a.reset();
    EXPECT(fake::device == 1);  // the caller's device stays selected
    EXPECT(cudaSetDevice(0) == cudaSuccess);
  }
  Buf keep;  // nothing idle is left to hide the driver's reuse of the address
  tsgne_set_device_memory_limit(0);
  for (size_t bytes : {64 * KiB, 48 * KiB, 4 * KiB}) {
    Buf b;
    EXPECT(take(b, bytes, 100) == TSGNE_OK);
    holds(b);
  }
  std::vector<Buf> all(8);
  for (Buf& b : all) {
    EXPECT(take(b, MiB, 100) == TSGNE_OK);
    holds(b);
  }
  EXPECT(fake::bad == 0);
}

// Buffers of both devices, freed under either, come back to their own device.
static void two_devices() {
  for (int round = 0; round < 4; ++round) {
    std::vector<Buf> v(16);
    for (int k = 0; k < 16; ++k) {
      EXPECT(cudaSetDevice(k & 1) == cudaSuccess);
      EXPECT(take(v[k], (size_t)(k + 1) * 96 * KiB, k & 1 ? 200 : 100) == TSGNE_OK);
      holds(v[k]);
      EXPECT(fake::live.at(reinterpret_cast<uintptr_t>(v[k].get())).device == (k & 1));
    }
    EXPECT(cudaSetDevice(round & 1) == cudaSuccess);
  }
  tsgne_set_device_memory_limit(0);
  EXPECT(fake::held() == 0 && fake::bad == 0);
}

// At most 256 MiB stay idle once a call has returned (its scope has ended),
// also when it failed, and at once where no call is running.
static void idle_bound() {
  EXPECT(cudaSetDevice(0) == cudaSuccess);
  const size_t bound = 256 * MiB;
  for (int k = 0; k < 3; ++k) {
    AllocScope as(stream(100));
    std::vector<Buf> v(6);
    for (Buf& b : v) EXPECT(b.alloc(100 * MiB) == TSGNE_OK);
  }
  EXPECT(fake::held() <= bound);
  std::vector<Buf> v(6);
  {
    AllocScope outer(stream(100));
    for (Buf& b : v) EXPECT(take(b, 90 * MiB, 101) == TSGNE_OK);
    Buf t;  // the inner scopes' ends leave the call's own temporaries alone
    EXPECT(t.alloc(30 * MiB) == TSGNE_OK);
  }
  const long frees = fake::frees;  // a call that frees nothing leaves it to the one that does
  std::thread([&] {
    EXPECT(cudaSetDevice(0) == cudaSuccess);
    AllocScope as(stream(102));
    std::vector<Buf> w(4);
    for (Buf& b : w) b.alloc(80 * MiB);
    for (Buf& b : w) b.reset();
    std::thread([] {
      EXPECT(cudaSetDevice(0) == cudaSuccess);
      AllocScope other(stream(103));
    }).join();
    EXPECT(fake::frees == frees);
  }).join();
  EXPECT(fake::frees > frees);
  const size_t before = fake::held();
  size_t out = 0;
  for (Buf& b : v) {
    out += b.n;
    b.reset();
    EXPECT(fake::held() <= before - out + bound);
  }
  EXPECT(fake::held() <= bound && fake::held() > 0);
  tsgne_set_device_memory_limit(0);
  EXPECT(fake::held() == 0 && fake::bad == 0);
}

// The account is what the device has given, and rounding refuses nothing that
// the device itself would give.
static void account() {
  EXPECT(cudaSetDevice(0) == cudaSuccess);
  std::vector<Buf> v(40);
  for (int k = 0; k < 40; ++k) EXPECT(take(v[k], (size_t)(k * k * k) * 9001 + 1, 100) == TSGNE_OK);
  EXPECT(fake::held() == (size_t)tsgne_device_memory_in_use());
  size_t asked = 0;
  for (int round = 0; round < 3; ++round)
    for (int k = 0; k < 40; ++k) {
      v[k].reset();
      EXPECT(take(v[k], (size_t)((k + round) * k * k) * 8513 + 1, 100) == TSGNE_OK);
      holds(v[k]);
    }
  for (const Buf& b : v) asked += b.n;
  EXPECT((size_t)tsgne_device_memory_in_use() <= asked + asked / 4 + 40 * (2 * MiB + MiB / 2));
  for (Buf& b : v) b.reset();
  tsgne_set_device_memory_limit(0);
  EXPECT(fake::held() == 0 && tsgne_device_memory_in_use() == 0);
  fake::capacity = 99 * MiB + 512 * KiB;
  Buf b;
  EXPECT(take(b, 99 * MiB + 1, 100) == TSGNE_OK);
  EXPECT(fake::held() == 99 * MiB + 1 && tsgne_device_memory_in_use() == (int64_t)(99 * MiB + 1));
  b.reset();
  EXPECT(take(b, 99 * MiB, 100) == TSGNE_OK);  // makes the idle block go, if it is not used
}

// Under a limit the device never gives more than it, in use and idle
// together, and exactly what fits is accepted.
static void limit() {
  EXPECT(cudaSetDevice(0) == cudaSuccess);
  const size_t lim = 50 * MiB;
  tsgne_set_device_memory_limit((int64_t)lim);
  unsigned long long x = 1;
  auto rnd = [&](size_t below) { return (size_t)((x = x * 6364136223846793005ull + 1442695040888963407ull) >> 33) % below; };
  for (int round = 0; round < 200; ++round) {
    std::vector<Buf> v(12);
    size_t asked = 0;
    for (Buf& b : v) {
      const size_t bytes = rnd(3) ? 1 + rnd(9 * MiB) : 4 * MiB;
      const tsgne_status st = take(b, bytes, 100 + (int)rnd(3));
      EXPECT((st == TSGNE_OK) == (asked + bytes <= lim));
      EXPECT(st == TSGNE_OK || st == TSGNE_ERR_OOM);
      if (st == TSGNE_OK) asked += bytes, holds(b);
      EXPECT(tsgne_device_memory_in_use() == (int64_t)asked);
      EXPECT(fake::held() <= lim);
    }
  }
  EXPECT(tsgne_device_memory_in_use() == 0);
  const long mallocs = fake::mallocs;  // the same sizes again: kept blocks serve them
  for (int k = 0; k < 10; ++k) {
    Buf a, b;
    EXPECT(take(a, 3 * MiB + 7, 100) == TSGNE_OK && take(b, 5 * MiB, 100) == TSGNE_OK);
  }
  EXPECT(fake::mallocs <= mallocs + 2);
  Buf plain;  // outside a scope: counted alike
  EXPECT(plain.alloc(lim) == TSGNE_OK && tsgne_device_memory_in_use() == (int64_t)lim);
  Buf more;
  EXPECT(more.alloc(1) == TSGNE_ERR_OOM && fake::held() == lim);
  plain.reset();
  tsgne_set_device_memory_limit(0);
  EXPECT(fake::held() == 0 && fake::bad == 0);
}

// cudaStreamPerThread is another stream in every thread: an event recorded by
// the thread that frees says nothing about the work of the one that used the
// buffer.  Such a buffer is not kept; its cudaFree waits for the device.
static void per_thread_stream() {
  EXPECT(cudaSetDevice(0) == cudaSuccess);
  Buf a;
  {
    AllocScope as(cudaStreamPerThread);
    EXPECT(a.alloc(MiB) == TSGNE_OK);
  }
  std::thread([&] { a.reset(); }).join();
  EXPECT(fake::held() == 0 && fake::frees == 1 && tsgne_device_memory_in_use() == 0);
}

// A request waits for memory that is in use, not for memory that the library
// only keeps for its next allocations.
static void server_admission() {
  EXPECT(cudaSetDevice(0) == cudaSuccess);
  tsgne_server_config c{};
  c.budget_bytes = (int64_t)1 << 40;
  c.iters = 100000;
  c.tick_iters = 10;
  c.max_members = 8;
  c.tile_warps = 1;
  c.fill_pairs = 1e18;
  tsgne_server* s = nullptr;
  EXPECT(tsgne_server_create(&s, &c, nullptr, nullptr) == TSGNE_OK);
  const int32_t n = 300000;
  const int64_t need = tsgne_server_estimate_bytes(n, 0, 1);
  std::vector<int64_t> rp(n + 1, 0);
  std::vector<float> X(n, 0.f);
  Buf kept;  // 200 MiB idle, and room for less than one more request beside the first
  EXPECT(take(kept, 200 * MiB, 100) == TSGNE_OK);
  kept.reset();
  fake::capacity = 200 * MiB + (size_t)need + (size_t)need / 2;
  int32_t resident = 0, queued = 0;
  for (int want = 1; want <= 2; ++want) {
    int64_t id;
    EXPECT(tsgne_server_submit(s, n, rp.data(), nullptr, X.data(), 1, nullptr, &id) == TSGNE_OK);
    for (int t = 0; t < 2000 && resident < want; ++t) {
      EXPECT(tsgne_server_tick(s, &resident, &queued, nullptr) == TSGNE_OK);
      std::this_thread::sleep_for(std::chrono::milliseconds(1));
    }
  }
  EXPECT(resident == 2 && queued == 0);
  EXPECT(fake::held() <= fake::capacity);
  tsgne_server_destroy(s);
  tsgne_set_device_memory_limit(0);
  EXPECT(fake::held() == 0 && fake::bad == 0);
}

int main(int argc, char** argv) {
  const std::string s = argc > 1 ? argv[1] : "";
  if (s == "other_device") freed_elsewhere(false);
  else if (s == "fresh_thread") freed_elsewhere(true);
  else if (s == "two_devices") two_devices();
  else if (s == "idle_bound") idle_bound();
  else if (s == "account") account();
  else if (s == "limit") limit();
  else if (s == "per_thread_stream") per_thread_stream();
  else if (s == "server_admission") server_admission();
  else return 2;
  return 0;
}

// Host-side handling of device resources against a fake CUDA runtime (no GPU): the
// functions below take the place of the runtime's in the library.  The case is
// the first argument.  Exits 0 when it holds.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>

#include "engine.hpp"
#include "mpslcc.h"

namespace {
// live objects by kind; the creation that fails (counted from 0), or none
std::map<std::string, int> live;
int created = 0, fail_at = -1;
bool make(const char* kind) {
  if (created++ == fail_at) return false;
  ++live[kind];
  return true;
}
char token[1 << 12];   // addresses of made-up objects
int tokens = 0;
template <class T> T next_token() { return (T)(void*)(token + ++tokens % sizeof(token)); }

// memory: a pool reserves what it has ever had in use until it is trimmed
const size_t CAPACITY = 4ull << 30;
struct Pool { size_t used = 0, reserved = 0; };
std::map<cudaMemPool_t, Pool> pools;
std::map<void*, std::pair<cudaMemPool_t, size_t>> blocks;
uintptr_t next_address = 1ull << 40;
size_t reserved() {
  size_t n = 0;
  for (auto& p : pools) n += p.second.reserved;
  return n;
}
}  // namespace

extern "C" {
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned int) {
  if (!make("stream")) return cudaErrorMemoryAllocation;
  *s = next_token<cudaStream_t>();
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { --live["stream"]; return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned int) {
  if (!make("host page")) return cudaErrorMemoryAllocation;
  *p = std::malloc(n);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { std::free(p); --live["host page"]; return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned int) {
  if (created++ == fail_at) return cudaErrorInvalidValue;
  *d = h;
  return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
  if (!make("pool")) return cudaErrorMemoryAllocation;
  *p = next_token<cudaMemPool_t>();
  pools[*p] = Pool();
  return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) { pools.erase(p); --live["pool"]; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) {
  return created++ == fail_at ? cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t keep) {
  auto it = pools.find(p);
  if (it == pools.end()) return cudaErrorInvalidValue;
  it->second.reserved = std::max(it->second.used, std::min(keep, it->second.reserved));
  return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** q, size_t n, cudaMemPool_t p, cudaStream_t) {
  Pool& l = pools.at(p);
  const size_t grow = l.used + n > l.reserved ? l.used + n - l.reserved : 0;
  if (reserved() + grow > CAPACITY) return cudaErrorMemoryAllocation;
  l.used += n;
  l.reserved += grow;
  *q = (void*)next_address;
  next_address += n + 512;
  blocks[*q] = {p, n};
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* q, cudaStream_t) {
  auto b = blocks.at(q);
  pools.at(b.first).used -= b.second;
  blocks.erase(q);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  if (!make("event")) return cudaErrorMemoryAllocation;
  *e = next_token<cudaEvent_t>();
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { --live["event"]; return cudaSuccess; }
cusolverStatus_t cusolverDnCreate(cusolverDnHandle_t* h) {
  if (!make("solver")) return CUSOLVER_STATUS_ALLOC_FAILED;
  *h = next_token<cusolverDnHandle_t>();
  return CUSOLVER_STATUS_SUCCESS;
}
cusolverStatus_t cusolverDnDestroy(cusolverDnHandle_t) { --live["solver"]; return CUSOLVER_STATUS_SUCCESS; }
cusolverStatus_t cusolverDnSetStream(cusolverDnHandle_t, cudaStream_t) { return CUSOLVER_STATUS_SUCCESS; }
}

using namespace mpslcc;

static bool nothing_left(const char* when) {
  bool ok = true;
  for (auto& k : live)
    if (k.second) {
      printf("%s: %d %s left\n", when, k.second, k.first.c_str());
      ok = false;
    }
  return ok;
}

// memory that one context keeps for its next calls is there for another's
static bool idle_memory() {
  mpslcc_ctx *a = nullptr, *b = nullptr;
  if (mpslcc_create(&a, nullptr) != MPSLCC_OK || mpslcc_create(&b, nullptr) != MPSLCC_OK) return printf("create\n"), false;
  bool ok = true;
  {
    DBuf x, y, z;
    x.alloc((Ctx*)a, 3ull << 30);
    x.release();
    try {
      y.alloc((Ctx*)b, 3ull << 30);
    } catch (const Error& e) {
      printf("%s, with %zu bytes idle\n", e.what(), reserved());
      ok = false;
    }
    try {   // memory in use stays where it is
      z.alloc((Ctx*)a, 3ull << 30);
      printf("more memory than there is\n");
      ok = false;
    } catch (const Error& e) {
      ok = ok && e.status == ST_NOMEM;
    }
  }
  mpslcc_destroy(a);
  mpslcc_destroy(b);
  return nothing_left("idle memory") && ok;
}

// a context whose creation fails half way leaves nothing behind
static bool failed_create() {
  for (int n = 0;; ++n) {
    created = 0;
    fail_at = n;
    mpslcc_ctx* c = nullptr;
    const mpslcc_status st = mpslcc_create(&c, nullptr);
    fail_at = -1;
    if (st == MPSLCC_OK) {
      mpslcc_destroy(c);
      return n > 5 && nothing_left("destroyed");
    }
    if (c || !nothing_left(("creation step " + std::to_string(n)).c_str())) return false;
  }
}

// a buffer whose allocation was refused is empty, so that the next call asks again
static bool refused_buffer() {
  static bool refuse;
  mpslcc_opts o;
  mpslcc_default_opts(&o);
  o.alloc = [](size_t n, void*) -> void* { return refuse ? nullptr : std::malloc(n); };
  o.free = [](void* p, size_t, void*) { std::free(p); };
  mpslcc_ctx* c = nullptr;
  if (mpslcc_create(&c, &o) != MPSLCC_OK) return printf("create\n"), false;
  bool ok = true;
  {
    DBuf x;
    refuse = true;
    for (int i = 0; i < 2; ++i) {
      try {
        x.ensure((Ctx*)c, 100);
        printf("a refused allocation went unnoticed\n");
        ok = false;
      } catch (const Error& e) {
        ok = ok && e.status == ST_NOMEM && !x.p;
      }
    }
    refuse = false;
    x.ensure((Ctx*)c, 100);
    ok = ok && x.p;
  }
  mpslcc_destroy(c);
  return ok && nothing_left("refused buffer");
}

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  if (what == "idle_memory") return idle_memory() ? 0 : 1;
  if (what == "failed_create") return failed_create() ? 0 : 1;
  if (what == "refused_buffer") return refused_buffer() ? 0 : 1;
  printf("no such case\n");
  return 2;
}

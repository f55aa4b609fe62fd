// Error reporting, device memory, handle release and version of the C ABI.
#include <cstdint>
#include <atomic>
#include <cstdarg>
#include <cstdio>
#include <mutex>
#include <string>

#include "lbm_internal.cuh"

namespace lbm {

namespace {
thread_local std::string g_last_error;
// The caller's allocator (both null: the library's own) and the number of
// blocks handed out and not yet released.
lbm_alloc_fn g_alloc = nullptr;
lbm_free_fn g_release = nullptr;
void* g_alloc_ctx = nullptr;
std::atomic<int64_t> g_live{0};

// Ordered blocks of the library's own come from one pool per device, which
// keeps up to 1/64 of the device's memory (4.4 GB on GB300) mapped when it is
// free: mapping fresh pages and giving them back took three quarters of the
// time of assembling a large lattice (1024x256x256 bed with its outputs 11.9
// ms, 2.8 ms with the pool).  Memory beyond that goes back to the device when the
// stream is next synchronised; all of it when an allocation of the library
// fails or lbm_set_allocator is called, and the driver takes it for a cudaMalloc
// of the process that needs it (with 4.0 GB idle, one of the free memory and
// 2.0 GB more succeeded).  1/64, 1.6% of the memory, is what an idle program is
// let keep; a lattice and its public links take 114 bytes a cell and 4 for each
// cell of the box, so on GB300 one of more than some 36 million cells maps
// its excess again in each assembly.  The driver orders the reuse of a block across streams,
// and the calls are safe from several threads.
constexpr int kMaxDevices = 64;
std::mutex g_pool_mutex;
cudaMemPool_t g_pool[kMaxDevices] = {};

// The current device's pool, or null (then the device's default pool serves).
cudaMemPool_t device_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  if (!g_pool[dev]) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    size_t free_bytes = 0, total = 0;
    if (cudaMemGetInfo(&free_bytes, &total) == cudaSuccess &&
        cudaMemPoolCreate(&pool, &props) == cudaSuccess) {
      uint64_t keep = total / 64;
      if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess)
        g_pool[dev] = pool;
      else cudaMemPoolDestroy(pool);
    }
    if (!g_pool[dev]) cudaGetLastError();
  }
  return g_pool[dev];
}

void give_back_pools() {
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  for (cudaMemPool_t pool : g_pool)
    if (pool) cudaMemPoolTrimTo(pool, 0);
}

cudaError_t own_alloc(void** p, size_t bytes, cudaStream_t stream, bool ordered) {
  cudaMemPool_t pool = ordered ? device_pool() : nullptr;
  const auto get = [&]() {
    return pool      ? cudaMallocFromPoolAsync(p, bytes, pool, stream)
           : ordered ? cudaMallocAsync(p, bytes, stream)
                     : cudaMalloc(p, bytes);
  };
  const cudaError_t e = get();
  if (e != cudaErrorMemoryAllocation) return e;
  cudaGetLastError();
  give_back_pools();
  return get();
}
}

cudaError_t dev_alloc(void** p, size_t bytes, cudaStream_t stream, bool ordered) {
  *p = nullptr;
  if (g_alloc) {
    void* q = g_alloc(bytes, (void*)stream, g_alloc_ctx);
    if (!q) return cudaErrorMemoryAllocation;
    if (reinterpret_cast<uintptr_t>(q) % 16 != 0) {   // the kernels use vector accesses
      if (g_release) g_release(q, (void*)stream, g_alloc_ctx);
      return cudaErrorMemoryAllocation;
    }
    *p = q;
  } else {
    const cudaError_t e = own_alloc(p, bytes, stream, ordered);
    if (e != cudaSuccess) {
      *p = nullptr;
      return e;
    }
  }
  ++g_live;
  return cudaSuccess;
}

void dev_free(void* p, cudaStream_t stream, bool ordered) {
  if (!p) return;
  --g_live;
  if (g_release) g_release(p, (void*)stream, g_alloc_ctx);
  else if (ordered) cudaFreeAsync(p, stream);
  else cudaFree(p);
}

int fail(int status, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_last_error = buf;
  return status;
}

int cuda_fail(cudaError_t e, const char* what) {
  return fail(e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA, "%s: %s (%s)", what,
              cudaGetErrorString(e), cudaGetErrorName(e));
}

void clear_error() { g_last_error.clear(); }

void free_sparse(lbm_sparse* sp) {
  if (!sp) return;
  const cudaStream_t s = sp->stream;
  for (void* p : {(void*)sp->cells, (void*)sp->inv, (void*)sp->adj, (void*)sp->adj_ld,
                  (void*)sp->code, (void*)sp->pages})
    dev_free(p, s, true);
  cudaStreamSynchronize(s);
  sp->magic = 0;
  delete sp;
}

}  // namespace lbm

extern "C" void lbm_free(void* handle) {
  if (!handle) return;
  const uint32_t magic = *static_cast<const uint32_t*>(handle);
  if (magic == lbm::kMagicSparse) lbm::free_sparse(static_cast<lbm_sparse*>(handle));
  else if (magic == lbm::kMagicState) lbm::free_state(static_cast<lbm_state*>(handle));
  else if (magic == lbm::kMagicAdjoint) lbm::free_adjoint(static_cast<lbm_adjoint*>(handle));
}

extern "C" const char* lbm_last_error(void) { return lbm::g_last_error.c_str(); }

extern "C" int lbm_set_allocator(lbm_alloc_fn alloc, lbm_free_fn release, void* ctx) {
  lbm::clear_error();
  if ((alloc == nullptr) != (release == nullptr))
    return lbm::fail(LBM_EINVAL, "give both allocator functions or neither");
  const int64_t live = lbm::g_live.load();
  if (live != 0)
    return lbm::fail(LBM_EINVAL, "%lld device blocks of existing handles are still live",
                     (long long)live);
  lbm::give_back_pools();
  lbm::g_alloc = alloc;
  lbm::g_release = release;
  lbm::g_alloc_ctx = ctx;
  return LBM_OK;
}

extern "C" int32_t lbm_abi_version(void) { return 2; }

// Device memory of scratch buffers and handles: stream-ordered allocations from a pool of the
// library's own (one per device), which keeps up to POOL_KEEP bytes of freed memory mapped. The
// device's default pool gives everything back at every synchronisation, and mapping it again
// costs 0.1 to 1 ms per call. The pool gives all it holds back when an allocation fails (which is
// then tried again), and the rest above POOL_KEEP at every synchronisation.
#pragma once
#include <cuda_runtime_api.h>
#include <stddef.h>
#include <stdint.h>
#include <initializer_list>

namespace lsq {

constexpr uint64_t POOL_KEEP = 1ull << 30;   // 0.35 % of the device's memory
// `bytes` on the current device, ordered on `st`.
cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t st);
template <typename T>
inline cudaError_t pool_alloc(T** p, size_t bytes, cudaStream_t st) { return pool_alloc((void**)p, bytes, st); }
// Frees a handle's arrays (NULL entries are skipped) once all work on `device`, which owns them, has
// ended: the handle may have been used on any of its streams, and the caller (a garbage
// collector, say) may have another device current.
void pool_free(int device, std::initializer_list<void*> ptrs);

}  // namespace lsq

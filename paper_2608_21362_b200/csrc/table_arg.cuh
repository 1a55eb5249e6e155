// A call's packed tables as a kernel argument.  Up to kDescBlobBytes they travel by value (two argument sizes, so that a
// small call does not pay for a large one): the kernel finds them in its parameter space, and no launch in front of it has
// to bring them into device memory.  Larger tables are in the context's arena, and the argument is their address.
#pragma once

#include <string.h>

#include "kvb_internal.h"

namespace kvb {

struct TableAddress {
  const uint8_t* p;
#ifdef __CUDACC__
  __device__ __forceinline__ const uint8_t* base() const { return p; }
#endif
};
template <size_t BYTES>
struct alignas(64) TableBytes {
  uint8_t b[BYTES];
#ifdef __CUDACC__
  __device__ __forceinline__ const uint8_t* base() const { return b; }
#endif
};

// Calls launch(argument) with the form the table has.
template <typename Launch>
inline cudaError_t with_table(const Table& t, Launch&& launch) {
  if (t.dev) return launch(TableAddress{t.dev});
  if (t.bytes <= kDescBlobSmall) {
    TableBytes<kDescBlobSmall> a;
    memcpy(a.b, t.host, t.bytes);
    return launch(a);
  }
  if (t.bytes > kDescBlobBytes) return cudaErrorInvalidValue;
  TableBytes<kDescBlobBytes> a;
  memcpy(a.b, t.host, t.bytes);
  return launch(a);
}

}  // namespace kvb

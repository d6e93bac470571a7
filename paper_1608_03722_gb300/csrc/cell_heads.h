// cell_heads.h -- heads of the resident kernel's cell lists.
#pragma once

#ifdef __CUDACC__
#define DSDNA_HD __host__ __device__ __forceinline__
#else
#define DSDNA_HD inline
#endif

namespace dsdna {

// A head holds the number of the rebuild that wrote it above the first item of
// its list, so that no rebuild has to clear the table: heads of other rebuilds,
// and zeroed ones, are empty lists.  Rebuilds count from 1 and get 44 bits (a
// system that rebuilds every 40 us repeats a number after 20 years; 32 bits
// repeated after two days, and zeroed heads matched then).  20 bits of item
// number hold a segment or bead of any system the kernel takes.
constexpr unsigned RES_NONE = 0xffffffffu;
constexpr int RES_ID_BITS = 20;
DSDNA_HD unsigned long long res_head(unsigned long long epoch, unsigned id) { return epoch << RES_ID_BITS | id; }
DSDNA_HD unsigned res_first(unsigned long long head, unsigned long long epoch) {
  return head >> RES_ID_BITS == epoch ? (unsigned)head & ((1u << RES_ID_BITS) - 1u) : RES_NONE;
}

}  // namespace dsdna

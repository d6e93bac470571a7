// kern_launch.cuh -- host-side launch of the persistent engine kernel for one
// precision; included once per precision by kern_mixed.cu / kern_fp64.cu.
#pragma once
#include <algorithm>

#include "engine_kernels.cuh"
#include "rebuild.cuh"
#include "chainlist.cuh"
#include "once_calls.h"
#include "resident.cuh"

namespace dsdna {

constexpr int CAPMAX = 64;

// mode | MODE_EXT selects the instance with circular molecules and the bubble
// rule, MODE_STEP | MODE_FUSED the one that rebuilds the list in the kernel.
template <class Real, bool EXT>
static const void* engine_fn_ext(int mode) {
  switch (mode & 3) {
    case MODE_STEP:
      return (mode & MODE_FUSED) ? (const void*)engine_kernel<Real, MODE_STEP, CAPMAX, EXT, true>
                                 : (const void*)engine_kernel<Real, MODE_STEP, CAPMAX, EXT, false>;
    case MODE_FORCES: return (const void*)engine_kernel<Real, MODE_FORCES, CAPMAX, EXT>;
    default: return (const void*)engine_kernel<Real, MODE_ENERGY, CAPMAX, EXT>;
  }
}
template <class Real>
static const void* engine_fn(int mode) {
  return (mode & MODE_EXT) ? engine_fn_ext<Real, true>(mode) : engine_fn_ext<Real, false>(mode);
}

// Largest co-resident grid for the cooperative launch of `mode` with T threads
// (T above engine_max_threads<Real>() has no resident CTA: 0).
template <class Real>
cudaError_t engine_occupancy(int mode, int T, int* blocks_per_sm, size_t* smem) {
  if (T > engine_max_threads<Real>()) {
    *blocks_per_sm = 0;
    return cudaSuccess;
  }
  *smem = seg_smem_bytes<Real>(T);
  const void* fn = engine_fn<Real>(mode);
  // the attribute is per kernel, shared by every context: allow the largest CTA any context may use
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)seg_smem_bytes<Real>(engine_max_threads<Real>()));
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, T, *smem);
}

template <class Real>
cudaError_t engine_launch(int mode, const KArgs<Real>& a, int grid, int T, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)T);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // the instance chosen by mode, launched with its parameter block
  void* args[] = {const_cast<KArgs<Real>*>(&a)};
  return cudaLaunchKernelExC(&cfg, engine_fn<Real>(mode), args);
}

// Launch shape of the resident kernel: blocks, threads and shared memory for n
// slots (0 blocks: a stretch would be longer than a CTA holds).  One stretch of
// whole segments per SM; warps for all owners and pairs of the stretch at once
// (about two warps per 32 slots), at least one thread per slot.  In FP64, where
// a second chunk in the same warp is another chain of FP64 latencies, four warps
// per tile (20 steps of 1216 bp 563 -> 539 us, of four rings of 300 bp 833 -> 781;
// the most a CTA holds from two tiles on).  Rings evaluate the owners next to
// their junctions besides: three warps per tile up to three tiles (100 steps of
// one ring of 500 bp 744 -> 661 us, 20 rings of 300 bp 930 -> 871), but at five
// tiles the wider barriers cost more (12 rings of 1000 bp 840 -> 880); linear
// molecules in mixed precision gain nothing (1216 bp 574 -> 583).
template <class Real>
cudaError_t resident_shape(int64_t n, int rings, bool ext, int nsm, int* grid, int* T, size_t* smem) {
  const int64_t nu = (n + SEG_W - 1) / SEG_W;
  *grid = (int)std::max<int64_t>(1, std::min<int64_t>(nsm, nu));
  const int64_t len = SEG_W * ((nu + *grid - 1) / *grid);
  static_assert((int64_t)res_max_len<Real>() * 1023 * 17 / 16 < (1 << RES_ID_BITS), "item numbers fit the list heads");
  if (nsm < 1 || nsm > 1023 || len > res_max_len<Real>()) {
    *grid = 0;
    return cudaSuccess;
  }
  const int tiles = (int)(len + 31) / 32;
  const int warps = sizeof(Real) == 8 ? 4 * tiles + 4 : rings && tiles <= 3 ? 3 * tiles + 3 : 2 * tiles + 2;
  *T = 32 * std::min(res_max_threads<Real>() / 32, warps);
  *smem = res_layout<Real>((int)len, rings, *T).bytes;
  const void* fn = ext ? (const void*)resident_kernel<Real, true> : (const void*)resident_kernel<Real, false>;
  // the attribute is per kernel, shared by every context: the largest any may use
  const size_t most = res_layout<Real>(res_max_len<Real>(), 1, res_max_threads<Real>()).bytes;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  int bps = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, fn, *T, *smem);
  if (e == cudaSuccess && bps < 1) *grid = 0;
  return e;
}

// Steps of a small system (mode as engine_launch's, MODE_STEP).
template <class Real>
cudaError_t resident_launch(int mode, const KArgs<Real>& a, int grid, int T, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)T);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  ResLayout lay = res_layout<Real>((int)(SEG_W * ((a.nseg16 + grid - 1) / grid)), a.n_junc > 0, T);
  ResOnce<false> once;
  void* args[] = {const_cast<KArgs<Real>*>(&a), &lay, &once};
  const void* fn = (mode & MODE_EXT) ? (const void*)resident_kernel<Real, true> : (const void*)resident_kernel<Real, false>;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

// One force evaluation (ONCE) of the configuration X, u in device memory.
// Prepared per device by resident_once_prepare.
#ifdef DSDNA_KERN_MIXED
cudaError_t resident_once_prepare() {
  const size_t most = res_layout<float>(res_max_len<float>(), 0, res_max_threads<float>()).bytes;
  cudaError_t e = cudaFuncSetAttribute(resident_kernel<float, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(resident_kernel<float, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}
static_assert(ONCE_CALLS < RES_SEQ, "tags of calls between two clears differ");
cudaError_t resident_once(const KArgs<float>& a, int nsm, const int* off, int steric_phase, unsigned call, const double* X,
                          const double* u, double* Fb, double* Fp, unsigned* err, cudaStream_t st) {
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(std::min(nsm, 1023), a.nseg16));
  const int len = SEG_W * (int)((a.nseg16 + grid - 1) / grid);
  if (len > res_max_len<float>()) return cudaErrorInvalidConfiguration;
  const int T = 32 * std::min(res_max_threads<float>() / 32, 2 * ((len + 31) / 32) + 2);
  ResLayout lay = res_layout<float>(len, 0, T);
  ResOnce<true> once{X, u, Fb, Fp, err, steric_phase, call, {}};
  std::copy(off, off + a.n_mol + 1, once.off);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)T);
  cfg.dynamicSmemBytes = lay.bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void* args[] = {const_cast<KArgs<float>*>(&a), &lay, &once};
  return cudaLaunchKernelExC(&cfg, a.bubble ? (const void*)resident_kernel<float, true, true>
                                            : (const void*)resident_kernel<float, false, true>, args);
}
#endif

// Kernel attributes of the rebuild kernels for the current device, set when a
// context is created: the chain-window list build asks for the largest
// shared-memory carveout, so that four of its CTAs (47 KB of shared memory
// each) are resident per SM.
template <class Real>
cudaError_t rebuild_prepare() {
  return cudaFuncSetAttribute(k_rebuild_list_chain<Real>, cudaFuncAttributePreferredSharedMemoryCarveout,
                              (int)cudaSharedmemCarveoutMaxShared);
}

// The rebuild kernels on stream st (grid-stride; the scan pair shares one grid):
// five for the chain-window build, five or six (pair halving) for the cell walks.
template <class Real>
cudaError_t rebuild_launch(const KArgs<Real>& a, int scan_grid, cudaStream_t st) {
  const int T = 256;
  int nsm = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int64_t want = (a.n + T - 1) / T;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)nsm * 16));
  if (a.segc) {
    // chain-window build (periodic box): segment grid (bin, scan, scatter),
    // then one warp per 32-slot tile builds its lists and their pair halving
    KArgs<Real> as = a;
    as.H = a.sg_H;
    const int sgrid = std::max(1, std::min(scan_grid, (int)((a.sg_H + 2047u) / 2048u)));
    k_rebuild_segbin<Real><<<grid, T, 0, st>>>(a);
    k_rebuild_scan_a<Real><<<sgrid, T, 0, st>>>(as);
    k_rebuild_scan_b<Real><<<sgrid, T, 0, st>>>(as);
    const int64_t swant = (a.nseg16 + T - 1) / T;
    k_rebuild_segscatter<Real><<<(int)std::max<int64_t>(1, std::min<int64_t>(swant, (int64_t)nsm * 16)), T, 0, st>>>(a);
    int cbps = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&cbps, k_rebuild_list_chain<Real>, CL_WARPS * 32, 0);
    const int cgrid = (int)std::max<int64_t>(
        1, std::min<int64_t>((a.nseg + CL_WARPS - 1) / CL_WARPS, (int64_t)nsm * std::max(1, cbps)));
    k_rebuild_list_chain<Real><<<cgrid, CL_WARPS * 32, 0, st>>>(a);
    return cudaGetLastError();
  }
  k_rebuild_bin<Real><<<grid, T, 0, st>>>(a);
  k_rebuild_scan_a<Real><<<scan_grid, T, 0, st>>>(a);
  k_rebuild_scan_b<Real><<<scan_grid, T, 0, st>>>(a);
  k_rebuild_scatter<Real><<<grid, T, 0, st>>>(a);
  const int LT = LIST_WARPS * 32;
  int lbps = 1;
  if (a.table == TABLE_LINEAR) {
    // one lane per bead
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&lbps, k_rebuild_list_lanes<Real>, LT, 0);
    const int lgrid = (int)std::max<int64_t>(1, std::min<int64_t>((a.n + LT - 1) / LT, (int64_t)nsm * std::max(1, lbps)));
    k_rebuild_list_lanes<Real><<<lgrid, LT, 0, st>>>(a);
  } else if (a.table == TABLE_HASH) {
    // open box: one lane per bead over the row ranges of the hashed blocks
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&lbps, k_rebuild_list_lanes_hash<Real>, LT, 0);
    const int lgrid = (int)std::max<int64_t>(1, std::min<int64_t>((a.n + LT - 1) / LT, (int64_t)nsm * std::max(1, lbps)));
    k_rebuild_list_lanes_hash<Real><<<lgrid, LT, 0, st>>>(a);
  } else {
    // one warp per 32 table entries at a time: enough CTAs for every chunk of
    // a small table, at most a full wave for a large one
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&lbps, k_rebuild_list<Real, CAPMAX>, LT, 0);
    const int lgrid = (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)a.H + 32 * LIST_WARPS - 1) / (32 * LIST_WARPS),
                                                                  (int64_t)nsm * std::max(1, lbps)));
    k_rebuild_list<Real, CAPMAX><<<lgrid, LT, 0, st>>>(a);
  }
  if (a.evl) {   // pair halving: the tiles' evaluated pairs, one resident wave of warps
    int pbps = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pbps, k_rebuild_pack<Real>, PACK_WARPS * 32, 0);
    const int pgrid = (int)std::max<int64_t>(
        1, std::min<int64_t>((a.nseg + PACK_WARPS - 1) / PACK_WARPS, (int64_t)nsm * std::max(1, pbps)));
    k_rebuild_pack<Real><<<pgrid, PACK_WARPS * 32, 0, st>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace dsdna

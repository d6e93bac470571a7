// observables.cu -- FP64 reductions for the observables of one molecule:
// extension R_z (Sec. 4.1), denatured fraction (Sec. 5), twist from base-pair
// frames (Sec. 3.2, App. B) and the linking number of the closed strands by
// the Gauss integral (App. C Eq. 17, read with the vector r_R - r_B).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "obs.h"

namespace dsdna {

struct D3 {
  double x, y, z;
};
__device__ __forceinline__ D3 d3(double x, double y, double z) { return D3{x, y, z}; }
__device__ __forceinline__ D3 sub(D3 a, D3 b) { return d3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ D3 add(D3 a, D3 b) { return d3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ D3 scl(double s, D3 a) { return d3(s * a.x, s * a.y, s * a.z); }
__device__ __forceinline__ double dt3(D3 a, D3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ D3 cr3(D3 a, D3 b) { return d3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x); }
__device__ __forceinline__ D3 unit(D3 a) { return scl(1.0 / sqrt(dt3(a, a)), a); }

__device__ __forceinline__ D3 site(const ObsArgs& a, int64_t g, double sgn) {
  D3 X = d3(a.X[g], a.X[a.n + g], a.X[2 * a.n + g]);
  D3 u;
  if (a.uf) {
    const float4 v = a.uf[g];
    u = d3(v.x, v.y, v.z);
  } else {
    u = d3(a.ud[g], a.ud[a.n + g], a.ud[2 * a.n + g]);
  }
  return add(X, scl(sgn * a.h, u));
}

__device__ __forceinline__ D3 ld3(const double* p, int64_t k) { return d3(p[3 * k], p[3 * k + 1], p[3 * k + 2]); }
__device__ __forceinline__ void st3(double* p, int64_t k, D3 v) { p[3 * k] = v.x; p[3 * k + 1] = v.y; p[3 * k + 2] = v.z; }
__device__ __forceinline__ D3 shfl_down3(D3 v, int o) {
  return d3(__shfl_down_sync(0xffffffffu, v.x, o), __shfl_down_sync(0xffffffffu, v.y, o),
            __shfl_down_sync(0xffffffffu, v.z, o));
}
__device__ __forceinline__ double warp_add(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// True in every thread of the block that finished last (all blocks' earlier
// global writes are then visible to it); the counter returns to zero.
__device__ __forceinline__ bool last_block(unsigned* counter) {
  __shared__ bool s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    if (s_last) *counter = 0u;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last;
}

// Both beads and the patch midpoint of base pair k; *broken: the patches are
// further apart than rc.
struct Bp {
  D3 mid, a, b;
};
__device__ __forceinline__ Bp base_pair(const ObsArgs& o, int k, bool* broken) {
  const int64_t gA = o.g0 + 2 * (int64_t)k, gB = gA + 1;
  const D3 pA = site(o, gA, 1.0), pB = site(o, gB, 1.0);
  const D3 d = sub(pB, pA);
  if (broken) *broken = dt3(d, d) > o.rc2;
  return Bp{add(pA, scl(0.5, d)), site(o, gA, -1.0), site(o, gB, -1.0)};
}

// Closure of both curves (App. C): extensions along the end-to-end axis and a
// far return path, shared by the two strands; ext: the largest distance of a
// bead from the first midpoint.
__device__ __forceinline__ void close_curves(const ObsArgs& a, double ext) {
  const Bp b0 = base_pair(a, 0, nullptr), b1 = base_pair(a, a.N - 1, nullptr);
  D3 e = sub(b1.mid, b0.mid);
  const double le = sqrt(dt3(e, e));
  e = le < 1e-12 ? d3(0, 0, 1) : scl(1.0 / le, e);
  const D3 ax = fabs(e.x) > 0.9 ? d3(0, 1, 0) : d3(1, 0, 0);
  const D3 ep = unit(cr3(e, ax));
  const double D = ext + 5.0, F = 2.0 * ext + 10.0;
  for (int c = 0; c < 2; ++c) {
    double* p = c == 0 ? a.ca : a.cb;
    const D3 c0 = c == 0 ? b0.a : b0.b, c1 = c == 0 ? b1.a : b1.b;
    st3(p, a.N, add(c1, scl(D, e)));
    st3(p, a.N + 1, add(add(c1, scl(D, e)), scl(F, ep)));
    st3(p, a.N + 2, add(sub(c0, scl(D, e)), scl(F, ep)));
    st3(p, a.N + 3, sub(c0, scl(D, e)));
  }
}

// Per base pair: midpoint, bead curves, broken bond, and the twist increment
// alpha + gamma between the frames of steps k and k + 1 (ZYZ Euler angles;
// N - 2 increments on a linear molecule, N on a ring).  The frame of step k
// is (f, v, t): t along the axis, f the bead-bead vector of base pair k
// projected normal to t.  A warp holds 32 base pairs and 31 increments, so
// midpoints and frames pass between lanes and nothing is read back from
// memory.  FP64 runs at two lanes per clock and SM, so the work is cut into
// one-warp blocks, each on its own SM while the molecule is short (as three
// kernels of 256-thread blocks -- base pairs, twist, closure -- 600 bp took
// 4.6 + 14.6 + 11 us).  The last block adds the blocks' sums in order, closes
// the curves and writes the results.
__global__ void __launch_bounds__(32) obs_frames_kernel(const ObsArgs a, int with_lk) {
  const int lane = threadIdx.x;
  const int k = blockIdx.x * 31 + lane;
  const bool own = lane < 31 && k < a.N;
  auto wrap = [&](int q) { return q < a.N ? q : (a.ring ? q % a.N : a.N - 1); };
  bool broken = false;
  const Bp bp = base_pair(a, wrap(k), &broken);
  D3 midn = shfl_down3(bp.mid, 1);
  if (lane == 31) midn = base_pair(a, wrap(k + 1), nullptr).mid;
  const D3 t = unit(sub(midn, bp.mid));
  D3 w = sub(bp.b, bp.a);
  w = sub(w, scl(dt3(w, t), t));
  const D3 f = unit(w), v = cr3(t, f);
  const D3 f1 = shfl_down3(f, 1), v1 = shfl_down3(v, 1);
  double inc = 0.0, ext2 = 0.0;
  if (own) {
    st3(a.mid, k, bp.mid);
    st3(a.ca, k, bp.a);
    st3(a.cb, k, bp.b);
    if (a.ring || k + 2 < a.N) {
      // R_ij = e_i(k) . e_j(k+1) with e = (f, v, t)
      const double R11 = dt3(f, f1), R12 = dt3(f, v1), R21 = dt3(v, f1), R22 = dt3(v, v1);
      inc = atan2(R21 - R12, R11 + R22) / (2.0 * 3.14159265358979323846);
      if (a.inc) a.inc[k] = inc;
    }
    if (with_lk && !a.ring) {
      const D3 m0 = base_pair(a, 0, nullptr).mid;
      const D3 d1 = sub(bp.a, m0), d2 = sub(bp.b, m0);
      ext2 = fmax(dt3(d1, d1), dt3(d2, d2));
    }
  }
  double nb = own && broken ? 1.0 : 0.0;
  nb = warp_add(nb);
  inc = warp_add(inc);
  for (int o = 16; o > 0; o >>= 1) ext2 = fmax(ext2, __shfl_xor_sync(0xffffffffu, ext2, o));
  if (lane == 0) {
    double* p = a.part + 3 * (int64_t)blockIdx.x;
    p[0] = nb; p[1] = inc; p[2] = ext2;
  }
  if (!last_block(a.counter)) return;
  nb = inc = ext2 = 0.0;
  for (unsigned b = lane; b < gridDim.x; b += 32) {
    const double* p = a.part + 3 * (int64_t)b;
    nb += __ldcg(p); inc += __ldcg(p + 1); ext2 = fmax(ext2, __ldcg(p + 2));
  }
  nb = warp_add(nb);
  inc = warp_add(inc);
  for (int o = 16; o > 0; o >>= 1) ext2 = fmax(ext2, __shfl_xor_sync(0xffffffffu, ext2, o));
  if (lane == 0) {
    a.out[0] = base_pair(a, a.N - 1, nullptr).mid.z - base_pair(a, 0, nullptr).mid.z;
    a.out[1] = nb;
    a.out[2] = inc;
    a.out[4] = 0.0;
    a.out[7] = (double)*a.err;
    if (with_lk && !a.ring) close_curves(a, sqrt(ext2));
    __threadfence_system();   // out is host memory
  }
}

// Gauss double sum over all segment pairs (a_i a_i+1), (b_j b_j+1) of the
// closed curves (the bead curves of a ring are closed already; a linear
// molecule's carry the four closure points).
//
// A pair's term is the signed solid angle of the quadrilateral its ends span
// seen from the origin of their differences, cut into two triangles whose
// half solid angles are the arguments of
//   z1 = l13 l14 l24 + (r13.r14) l24 + (r14.r24) l13 + (r24.r13) l14 + i T
//   z2 = l13 l24 l23 + (r13.r24) l23 + (r24.r23) l13 + (r23.r13) l24 + i T
// (the solid-angle formula of Van Oosterom and Strackee, 1983) with
// r13 = b_j - a_i and so on, l their lengths and T = r13 . (d x e) the same
// for both, d and e the segments.  The scalar products follow from the
// squared lengths and the segments alone, so a pair needs one new length: the
// others come from the previous j and, by shuffle, from the next lane's i.
// arg z1 + arg z2 stays within (-pi, pi), because T r^-3 keeps its sign over
// two straight segments; so a lane multiplies its pairs' z1 z2 into one
// complex number, counts its turns by the signs of the imaginary parts, and
// takes one arctangent at the end.  That is about 50 FP64 operations per pair
// against about 500 for four normalised cross products and four arcsines, and
// it is exact to rounding (Lk of a closed duplex is an integer to 1e-13)
// where the arcsine near +-1 lost half the digits.
//
// FP64 bound: two lanes per clock and SM.  A warp holds 31 segments i; work
// items of 4 x 31 segments times a run of `len` segments j are dealt to the
// blocks in order, `len` chosen so that a short molecule still fills the SMs
// (600 bp: 5 x 121 items of 5 j, about four blocks per SM).  One call for a
// 600 bp molecule, launches and wait included: 84 us, against 7280 us as one
// thread per i with all j (five blocks of 128).
constexpr int LK_WARPS = 4, LK_I = 31 * LK_WARPS, LK_J = 64;
__global__ void __launch_bounds__(32 * LK_WARPS) obs_lk_kernel(const ObsArgs a, int M, int nig, int len, int64_t items) {
  __shared__ double sb[LK_J + 1][3], se[LK_J][4];
  __shared__ double red[LK_WARPS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double zr = 1.0, zi = 0.0;
  int turns = 0;
  for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const int j0 = (int)(it / nig) * len, nj = min(len, M - j0);
    const int i = (int)(it % nig) * LK_I + warp * 31 + lane;
    __syncthreads();
    for (int q = threadIdx.x; q <= nj; q += blockDim.x) {
      const int j = j0 + q;
      const D3 p = ld3(a.cb, j < M ? j : 0);
      sb[q][0] = p.x; sb[q][1] = p.y; sb[q][2] = p.z;
      if (q < nj) {
        const D3 e = sub(ld3(a.cb, j + 1 < M ? j + 1 : 0), p);
        se[q][0] = e.x; se[q][1] = e.y; se[q][2] = e.z; se[q][3] = dt3(e, e);
      }
    }
    __syncthreads();
    const bool live = lane < 31 && i < M;
    const int i0 = i < M ? i : 0, i1 = i0 + 1 < M ? i0 + 1 : 0;
    const D3 p = ld3(a.ca, i0), d = sub(ld3(a.ca, i1), p);
    const double dd = dt3(d, d);
    const D3 d2 = scl(2.0, d);
    // column j0: r13 and its length here, r23's from the next lane
    D3 r = d3(sb[0][0] - p.x, sb[0][1] - p.y, sb[0][2] - p.z);
    double s13 = dt3(r, r), l13 = sqrt(s13);
    double s23 = __shfl_down_sync(0xffffffffu, s13, 1), l23 = __shfl_down_sync(0xffffffffu, l13, 1);
    double p23 = s13 + s23 - dd;                       // 2 r23.r13
    for (int q = 0; q < nj; ++q) {
      const D3 e = d3(se[q][0], se[q][1], se[q][2]);
      const double ee = se[q][3];
      const D3 rn = d3(sb[q + 1][0] - p.x, sb[q + 1][1] - p.y, sb[q + 1][2] - p.z);
      const double s14 = dt3(rn, rn), l14 = sqrt(s14);
      const double s24 = __shfl_down_sync(0xffffffffu, s14, 1), l24 = __shfl_down_sync(0xffffffffu, l14, 1);
      const double p34 = s13 + s14 - ee;               // 2 r13.r14
      const double p34n = __shfl_down_sync(0xffffffffu, p34, 1);   // 2 r23.r24
      const double p14 = s14 + s24 - dd;               // 2 r14.r24
      // 2 r13.r24 = s13 + s24 - |e - d|^2
      const double px = fma(d2.x, e.x, fma(d2.y, e.y, fma(d2.z, e.z, (s13 + s24) - (ee + dd))));
      const double g = fma(2.0 * l13, l24, px);
      const double D1 = fma(g, l14, fma(p34, l24, p14 * l13));
      const double D2 = fma(g, l23, fma(p34n, l13, p23 * l24));
      const double T = dt3(r, cr3(d2, e));
      double xr = fma(D1, D2, -(T * T)), xi = T * (D1 + D2);
      if (!live || T == 0.0) { xr = 1.0; xi = 0.0; }   // coplanar segments span no solid angle
      const double nr = fma(zr, xr, -(zi * xi)), ni = fma(zr, xi, zi * xr);
      // the argument passed +-pi: upper times upper half plane gives lower, or the reverse
      const int sx = __double2hiint(xi) >> 31, so = __double2hiint(zi) >> 31, sn = __double2hiint(ni) >> 31;
      turns += (~sx & ~so & sn & 1) - (sx & so & ~sn & 1);
      zr = nr; zi = ni;
      if ((q & 3) == 3 || q + 1 == nj) {   // a pair multiplies |z| by up to about 64 l^6: back to 1 by a power of two
        const int h = max(__double2hiint(zr) & 0x7fffffff, __double2hiint(zi) & 0x7fffffff) >> 20;
        const double sc = __hiloint2double(max(1, 2046 - h) << 20, 0);
        zr *= sc; zi *= sc;
      }
      r = rn; s13 = s14; l13 = l14; s23 = s24; l23 = l24; p23 = p14;
    }
  }
  double acc = warp_add(atan2(zi, zr) + 6.28318530717958647693 * (double)turns);
  if (lane == 0) red[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < LK_WARPS; ++w) acc += red[w];
    a.part[blockIdx.x] = acc;
  }
  if (!last_block(a.counter) || warp != 0) return;
  acc = 0.0;
  for (unsigned b = lane; b < gridDim.x; b += 32) acc += __ldcg(a.part + b);
  acc = warp_add(acc);
  if (lane == 0) {
    a.out[4] = acc * (-1.0 / 6.28318530717958647693);
    __threadfence_system();
  }
}

int64_t obs_partials(int maxN) { return 3 * ((int64_t)maxN / 31 + 1) + OBS_MAX_GRID; }

cudaError_t obs_launch(const ObsArgs& a, unsigned flags, int nsm, cudaStream_t st) {
  const bool lk = (flags & 8u) && a.N >= 2;
  obs_frames_kernel<<<(a.N + 30) / 31, 32, 0, st>>>(a, lk ? 1 : 0);
  if (lk) {
    const int M = a.ring ? a.N : a.N + 4;
    const int nig = (M + LK_I - 1) / LK_I;
    const int grid_most = std::min(4 * std::max(1, nsm), OBS_MAX_GRID);
    // j segments per item: enough items for every block, at most LK_J
    const int runs = (grid_most + nig - 1) / nig;
    const int len = std::min(LK_J, std::max(4, (M + runs - 1) / runs));
    const int64_t items = (int64_t)nig * ((M + len - 1) / len);
    obs_lk_kernel<<<(int)std::min<int64_t>(items, grid_most), 32 * LK_WARPS, 0, st>>>(a, M, nig, len, items);
  }
  return cudaGetLastError();
}

}  // namespace dsdna

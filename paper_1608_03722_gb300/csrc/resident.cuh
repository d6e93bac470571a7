// resident.cuh -- step kernel of small systems: every CTA keeps its stretch of
// the chain in shared memory and registers from step to step.  Included by
// kern_launch.cuh after engine_kernels.cuh and chainlist.cuh.
//
// Up to 512 nucleotides per SM (256 in FP64) the strip kernel (engine_kernel)
// waits rather than works: a warp walks one tile by itself through a chain of
// memory latencies and two passes of bonded terms (its prologue's and its
// own), reloads the whole state every step, and a stale list costs five more
// grid barriers and a cell walk.  Here
//  * the CTAs split the chain into stretches of whole 16-slot segments, one
//    CTA per SM; positions and flags of the stretch live in shared memory,
//    X, V, Omega and the rebuild reference of a nucleotide in its thread's
//    registers, so a step reads only the few slots beyond its ends and the
//    list partners of other stretches;
//  * owners and list pairs are dealt to the warps together (they need only
//    positions), one block barrier later every nucleotide adds its forces and
//    moves;
//  * positions pass between CTAs as 16-byte records that carry the step they
//    belong to, stored and polled as single 128-bit accesses: a reader waits
//    for the slots it needs and for nothing else;
//  * the grid-wide agreement that no bead has outrun the list (and that no
//    error happened) is needed only before the pair forces are used, so a
//    warp of its own publishes the CTA's word and polls the others' while the
//    rest evaluate the next step's owners and pairs; a stale list throws away
//    the pair forces only.  As a barrier after every step (a release add on
//    one word, polled by all) it took 2.6 us of the 5.9 us of a 10 kbp step;
//  * a rebuild is one phase that bins the beads and threads each 16-slot
//    segment into a hash of cells (linked lists, no table scan), one grid
//    barrier, and the chain-window list build of the CTA's own beads, whose
//    result stays in shared memory.
// All forces, sums and updates are those of engine_kernel, term by term in the
// same order, so trajectories agree bit for bit.  100 steps and one state
// download, strip kernel with in-kernel rebuild -> this kernel: 10 kbp 1953 ->
// 677 us, periodic walk of 30 kbp 2232 -> 1117 us, 64 rings of 500 bp 3435 ->
// 1151 us, melting 16 x 1000 bp 1807 -> 739 us; 50 FP64 steps of 200 bp 3722
// -> 1188 us (a warp per SM instead of eight sharing one SM's FP64 pipe).
//
// Cycles of a step by clock stamps on every CTA (profiles/resident_kernel.md):
// 10 kbp 6800 (3800 until all forces and the agreement are there, 2850 to gather
// and update) and 20,000 per rebuild; 200 bp in FP64 40,900 (27,500 for one pass
// of the owners' terms, 13,400 to gather and update).  Dealing the FP64 work in
// groups of few lanes over all schedulers was slower (24 -> 38 us).
#pragma once
#include "../../include/dsdna.h"
#include "cell_heads.h"
#include "chainlist.cuh"
#include "engine_kernels.cuh"

namespace dsdna {

template <class Real> __host__ __device__ constexpr int res_max_len() { return sizeof(Real) == 4 ? 512 : 256; }
template <class Real> __host__ __device__ constexpr int res_max_threads() { return res_max_len<Real>(); }
constexpr int RES_PAIRS_PER_SLOT = 4;   // list entries kept in shared memory per slot (else the lists are walked in memory)

// Shared-memory layout of a CTA whose stretch holds at most `len` slots.
constexpr int RES_HALO = 8;   // slots staged beyond either end of a stretch (the neighbourhoods of its owners)
struct ResLayout {
  int len, own, pairs, warps;
  size_t pos, flg, cs, cn, cp, pf, ent, off, po, jx, xo, xw, load, list, win, gi, gc, bytes;
};
template <class Real>
__host__ __device__ inline ResLayout res_layout(int len, int rings, int T) {
  ResLayout l;
  l.len = len;
  l.own = len + 4 + (rings ? len / 3 + 8 : 0);   // owners of a stretch, and those across the junctions of its rings
  l.pairs = RES_PAIRS_PER_SLOT * len + 64;
  l.warps = T / 32;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = (o + bytes + 15) & ~(size_t)15;
    return at;
  };
  l.pos = take(2 * sizeof(SPos<Real>) * (len + 2 * RES_HALO));   // this step's and the next one's
  l.cs = take(sizeof(Real) * 6 * l.own);
  l.cn = take(sizeof(Real) * 6 * l.own);
  l.cp = take(sizeof(Real) * 3 * l.own);
  l.pf = take(sizeof(Real) * 3 * l.pairs);
  l.load = take(sizeof(Real) * 6 * len);
  l.win = take(sizeof(float4) * (CL_WIN + CL_WIN / 16) * l.warps);
  l.gc = take(sizeof(float4) * 4 * l.warps);
  l.gi = take(sizeof(int) * 4 * l.warps);
  l.flg = take(sizeof(int) * (len + 2 * RES_HALO));
  l.ent = take(sizeof(int) * l.pairs);
  l.off = take(sizeof(int) * (len + 33));
  l.xo = take(sizeof(int) * (rings ? l.own : 0));
  l.xw = take(sizeof(short) * (rings ? l.own : 0));
  l.list = take(sizeof(int) * 32 * LIST_CAP * l.warps);
  l.po = take(sizeof(unsigned short) * l.pairs);
  l.jx = take(sizeof(short) * len);
  l.bytes = o;
  return l;
}

// ---------------------------------------------------------------- exchange between CTAs
// A slot's position and orientation as records of three words and a tag: the
// sequence number of the step (rs_seq + steps of this launch, so that records
// of earlier launches never match; 30 bits) and the slot's removed terms
// (bubble rule 2, two bits); double-buffered by step parity.  A CTA
// overwrites the records of step t when it finishes step t + 1, after every
// CTA's word for step t, and so after every read of them.
constexpr unsigned RES_SEQ = 0x3fffffffu;
template <class Real> __host__ __device__ constexpr int res_records() { return (int)sizeof(SPos<Real>) / 12; }

__device__ __forceinline__ void st128(uint4* p, uint4 v) {
  asm volatile("{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}\n" ::"l"(p),
               "l"((unsigned long long)v.x | ((unsigned long long)v.y << 32)),
               "l"((unsigned long long)v.z | ((unsigned long long)v.w << 32))
               : "memory");
}
__device__ __forceinline__ uint4 ld128(const uint4* p) {
  unsigned long long lo, hi;
  asm volatile("{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}\n"
               : "=l"(lo), "=l"(hi)
               : "l"(p)
               : "memory");
  return make_uint4((unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32));
}

template <class Real>
__device__ __forceinline__ void rec_store(const KArgs<Real>& a, int cur, unsigned g, unsigned seq, int flags, const SPos<Real>& s) {
  constexpr int R = res_records<Real>();
  uint4* p = a.rs_xch + R * ((size_t)cur * a.ns + g);
  unsigned w[3 * R];
  memcpy(w, &s, sizeof(s));
  const unsigned tag = (seq & RES_SEQ) | ((unsigned)(flags >> RM_SHIFT) << 30);
#pragma unroll
  for (int r = 0; r < R; ++r) st128(p + r, make_uint4(w[3 * r], w[3 * r + 1], w[3 * r + 2], tag));
}

// Waits for slot g's records of step seq, at most the launch's clock budget;
// then *timeout is set and the records are returned as they are.  *removed: the
// slot's removed terms.
template <class Real>
__device__ __forceinline__ SPos<Real> rec_load(const KArgs<Real>& a, int cur, unsigned g, unsigned seq, unsigned* timeout,
                                              unsigned* removed = nullptr) {
  constexpr int R = res_records<Real>();
  const uint4* p = a.rs_xch + R * ((size_t)cur * a.ns + g);
  unsigned w[3 * R];
  const unsigned long long t0 = clock64();
  for (;;) {
    bool ok = true;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint4 v = ld128(p + r);
      w[3 * r] = v.x; w[3 * r + 1] = v.y; w[3 * r + 2] = v.z;
      ok = ok && ((v.w ^ seq) & RES_SEQ) == 0u;
      if (removed) *removed = v.w >> 30;
    }
    if (ok) break;
    if ((unsigned long long)(clock64() - t0) > a.spin_budget) { *timeout = 1u; break; }
  }
  SPos<Real> s;
  memcpy(&s, w, sizeof(s));
  return s;
}

// The same for three slots together; slots of the stretch come from spos.
template <class Real>
__device__ __forceinline__ void rec_load3(const KArgs<Real>& a, int cur, const int* slot, unsigned seq, unsigned* timeout,
                                          const SPos<Real>* spos, int s0, int len, SPos<Real>* out) {
  constexpr int R = res_records<Real>();
  unsigned w[3][3 * R];
  bool out_of[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) out_of[k] = (unsigned)(slot[k] - s0) >= (unsigned)len;
  const unsigned long long t0 = clock64();
  for (;;) {
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (out_of[k]) {
        const uint4* p = a.rs_xch + R * ((size_t)cur * a.ns + (unsigned)slot[k]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const uint4 v = ld128(p + r);
          w[k][3 * r] = v.x; w[k][3 * r + 1] = v.y; w[k][3 * r + 2] = v.z;
          ok = ok && ((v.w ^ seq) & RES_SEQ) == 0u;
        }
      }
    if (ok) break;
    if ((unsigned long long)(clock64() - t0) > a.spin_budget) { *timeout = 1u; break; }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (out_of[k]) memcpy(&out[k], w[k], sizeof(SPos<Real>));
    else out[k] = spos[slot[k] - s0];
  }
}

// Agreement number p of a launch (step agreements and rebuild barriers share
// one count) on word p mod 3 of bar->res: arrivals in bits 0-9, stale
// stretches in bits 10-19, stretches with an error in bits 20-29 (their bits
// are in bar->gen).  The word of p - 1 is cleared after p by block 0, two
// agreements before it is used again.  Publishing releases the CTA's writes
// (after a block barrier), reading acquires the others'.  One word and one
// release add take 1.28 us over 152 CTAs; a word per CTA, polled by all, took
// 2.8 to 5 us, the polls queueing behind one another and the stores.
template <class Real>
__device__ __forceinline__ void res_publish(const KArgs<Real>& a, unsigned p, unsigned fl) {
  if (fl & B_ERRMASK) atomicOr(&a.bar->gen, fl & B_ERRMASK);
  const unsigned v = 1u | ((fl & B_STALE) ? 1u << 10 : 0u) | ((fl & B_ERRMASK) ? 1u << 20 : 0u);
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(a.bar->res[p % 3]), "r"(v) : "memory");
}
// All CTAs' flags of agreement p (one thread); B_ETIMEOUT when the clock budget
// runs out.
template <class Real>
__device__ __forceinline__ unsigned res_agree(const KArgs<Real>& a, unsigned p) {
  const unsigned long long t0 = clock64();
  unsigned v;
  while (((v = ld_acquire(a.bar->res[p % 3])) & 1023u) != gridDim.x)
    if ((unsigned long long)(clock64() - t0) > a.spin_budget) return B_ETIMEOUT;
  if (blockIdx.x == 0) a.bar->res[(p + 2) % 3][0] = 0u;
  unsigned r = ((v >> 10) & 1023u) ? B_STALE : 0u;
  if (v >> 20) r |= ld_acquire(&a.bar->gen);
  return r;
}

// ---------------------------------------------------------------- neighbourhood of an owner
// ResSrc: the stretch and its halo in shared memory (every owner but those
// next to the junction of a circular molecule; spos and flg point at the first
// slot of the stretch).
template <class Real>
struct ResSrc {
  const SPos<Real>* spos;
  const int* flg;
  int s0;
  __device__ __forceinline__ SPos<Real> pos(int64_t g) const { return spos[(int)g - s0]; }
  __device__ __forceinline__ int64_t step(int64_t g, int d) const { return (int)g + d; }
  __device__ __forceinline__ bool open(int64_t k, int mol) const {
    const int f = flg[2 * (int)k - s0];
    return (f & F_OPEN) && (f >> MOL_SHIFT) == mol;
  }
};

// ResJunc: an owner next to a junction, whose neighbours are taken modulo the
// molecule (base pairs off .. off + N - 1): its three slots, waited for
// together; the base pairs of the bubble rule one by one.
template <class Real>
struct ResJunc {
  const KArgs<Real>& a;
  const SPos<Real>* spos;
  const int* flg;
  unsigned* timeout;
  int cur;
  unsigned seq;
  int s0, len, off, N;
  int slot[3];        // the owner, the next and the previous nucleotide of its strand
  SPos<Real> p3[3];
  __device__ __forceinline__ int bp(int k) const {   // at most three base pairs outside the molecule
    return k < off ? k + N : (k >= off + N ? k - N : k);
  }
  __device__ __forceinline__ void load(int o) {
    const int dir = (o & 1) ? -2 : 2;
    slot[0] = o;
    slot[1] = (int)step(o, dir);
    slot[2] = (int)step(o, -dir);
    rec_load3(a, cur, slot, seq, timeout, spos, s0, len, p3);
  }
  __device__ __forceinline__ SPos<Real> at(int g) const {
    const unsigned l = (unsigned)(g - s0);
    if (l < (unsigned)len) return spos[l];
    return rec_load(a, cur, (unsigned)g, seq, timeout);
  }
  __device__ __forceinline__ SPos<Real> pos(int64_t g) const {
    return (int)g == slot[0] ? p3[0] : ((int)g == slot[1] ? p3[1] : p3[2]);
  }
  __device__ __forceinline__ int64_t step(int64_t g, int d) const {
    return 2 * bp(((int)g >> 1) + d / 2) + ((int)g & 1);
  }
  __device__ __forceinline__ bool open(int64_t k64, int /*mol*/) const {
    const int k = bp((int)k64);
    const unsigned l = (unsigned)(2 * k - s0);
    if (l < (unsigned)len) return (flg[l] & F_OPEN) != 0;
    const SPos<Real> pa = at(2 * k), pb = at(2 * k + 1);
    const V3<Real> d = rel(pa, pb, a.fixq) + a.c.h * (uvec(pb) - uvec(pa));
    return dot(d, d) > a.c.rchb2;
  }
};

// Typed WCA force of list entry e on bead b of the stretch (record me, partner
// q with flags fj).
template <class Real>
__device__ __forceinline__ V3<Real> res_pair(const KArgs<Real>& a, int s0, int b, const SPos<Real>& me, int fb, int e,
                                             const SPos<Real>& q, int fj) {
  const int j = e & ENT_JMASK;
  V3<Real> R = rel(me, q, a.fixq);
  if constexpr (sizeof(Real) == 8) {
    if (a.periodic) {
      const int wi = a.img[s0 + b], wj = a.img[j];
      R.x += (double)(img_comp(wi, 0) - img_comp(wj, 0) + ent_shift(e, 0)) * a.L[0];
      R.y += (double)(img_comp(wi, 1) - img_comp(wj, 1) + ent_shift(e, 1)) * a.L[1];
      R.z += (double)(img_comp(wi, 2) - img_comp(wj, 2) + ent_shift(e, 2)) * a.L[2];
    }
  }
  return pair_core(a, R, uvec(me), uvec(q), ((s0 + b) ^ j) & 1, (fb & fj & F_STERIC) != 0, (V3<Real>*)nullptr,
                   (Real*)nullptr);
}

// ---------------------------------------------------------------- list build
// The segment grid of the resident kernel: cells of the wide kernel's segment
// grid in a periodic box; in an open box wider ones that keep segments of up to
// DSDNA_RES_RCAP whole (a molten stretch spreads its 16 slots over 2 nm and
// more, and bead by bead they cost four times a whole segment), hashed by
// molecule and cell.
template <class Real>
__device__ __forceinline__ void res_cell(const KArgs<Real>& a, const float* p, int* ci) {
  if (a.periodic) {
    seg_cell(a, p[0], p[1], p[2], ci);
  } else {
    for (int c = 0; c < 3; ++c) ci[c] = (int)floorf(p[c] * a.rs_invh);
  }
}
// Bucket of neighbour q (0..26; 13 is the cell itself) of cell ci.
template <class Real>
__device__ __forceinline__ unsigned res_key(const KArgs<Real>& a, int mol, const int* ci, int q) {
  int cc[3] = {ci[0] + q % 3 - 1, ci[1] + (q / 3) % 3 - 1, ci[2] + q / 9 - 1};
  if (a.periodic)
    for (int c = 0; c < 3; ++c) cc[c] = cc[c] < 0 ? cc[c] + a.sg_nc[c] : (cc[c] >= a.sg_nc[c] ? cc[c] - a.sg_nc[c] : cc[c]);
  return hash_block(mol, cc[0], cc[1], cc[2]) & a.rs_mask;
}

// A grid item is a segment, or its first part when it spans two molecules (id:
// the segment), the second part (id: nseg16 + its first slot), or a bead of a
// wide segment (nseg16 + its slot).  Into the front of its cell's list; a head
// of an earlier rebuild (another epoch) is an empty list.
template <class Real>
__device__ __forceinline__ void res_insert(const KArgs<Real>& a, int mol, const float* p, unsigned id, unsigned long long epoch) {
  int ci[3];
  res_cell(a, p, ci);
  const unsigned long long old =
      atomicExch(a.rs_head + res_key(a, mol, ci, 13), res_head(epoch, id));
  a.rs_next[id] = res_first(old, epoch);
}
// Sphere and slot range (first slot | (beads - 1) << ENT_J_BITS) of item id.
template <class Real>
__device__ __forceinline__ int res_item(const KArgs<Real>& a, unsigned id, float4& sph) {
  const unsigned nseg = (unsigned)a.nseg16;
  if (id < nseg) {
    sph = a.segc[id];
    const int nb = a.n_mol > 1 ? a.rs_part[id] : min(SEG_W, (int)a.n - (int)(id * SEG_W));
    return (int)(id * SEG_W) | ((nb - 1) << ENT_J_BITS);
  }
  const unsigned j = id - nseg, s = j / SEG_W;
  const float4 whole = a.segc[s], second = a.rs_sph1[s], p = a.wpos[j];
  if (whole.w < 0.0f) {
    sph = make_float4(p.x, p.y, p.z, 0.0f);
    return (int)j;
  }
  sph = second;
  return (int)j | ((min((int)((s + 1) * SEG_W), (int)a.n) - (int)j - 1) << ENT_J_BITS);
}

// Bead g of a wide segment (wrapped position mp) against the items of its own 27
// cells; returns (cnt, total).  Out of line: wide segments are rare.
template <class Real>
__device__ __noinline__ int2 res_list_bead(const KArgs<Real>& a, int g, float4 mp, bool st_g, unsigned long long epoch, int* list,
                                           int cnt, int total) {
  const int s = g / SEG_W;
  int ci[3];
  const float p3[3] = {mp.x, mp.y, mp.z};
  res_cell(a, p3, ci);
  const int pmol = __float_as_int(mp.w);
  const int plo = a.n_mol > 1 ? 2 * (int)a.mol_off[pmol] : 0, phi = a.n_mol > 1 ? 2 * (int)a.mol_off[pmol + 1] : (int)a.n;
  const float4 pt = make_float4(mp.x, mp.y, mp.z, 0.0f);
  const unsigned most = (unsigned)(a.nseg16 + a.n);   // items there are at most
  // the buckets first, all heads in flight together; a bucket two cells share is walked once
  unsigned keys[27], hd[27];
#pragma unroll
  for (int q = 0; q < 27; ++q) {
    keys[q] = res_key(a, pmol, ci, q);
    hd[q] = res_first(a.rs_head[keys[q]], epoch);
  }
#pragma unroll
  for (int q = 1; q < 27; ++q)
#pragma unroll
    for (int o = 0; o < q; ++o)
      if (keys[o] == keys[q]) hd[q] = RES_NONE;
#pragma unroll 1
  for (int q = 0; q < 27; ++q) {
    unsigned walked = 0;
    for (unsigned e = hd[q]; e != RES_NONE && walked <= most; e = a.rs_next[e], ++walked) {
      float4 it;
      const int ir = res_item(a, e, it);
      const int j0 = ir & ENT_JMASK, js = j0 / SEG_W;
      if (j0 < plo || j0 >= phi || (js <= s + 1 && js >= s - 1)) continue;
      if (cl_spheres_meet(a, pt, it)) cl_item_pairs(a, g, mp, st_g, ir, list, cnt, total);
    }
  }
  return make_int2(cnt, total);
}

// Cell lists around the lanes' parts sc of segments sA, sA + 1 (radius < 0:
// none) of molecules qmol: first item of the cell each lane walks for either
// (a bucket that a lower lane of the same part also reads is dropped), and the
// slot ranges of the molecules.
struct ResQuery {
  unsigned id[2];
  int slo[2], shi[2];
};
template <class Real>
__device__ __forceinline__ void res_query(const KArgs<Real>& a, const float4* sc, const int* qmol, unsigned long long epoch,
                                          ResQuery& q) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    unsigned key = RES_NONE;
    if (lane < 27 && sc[h].w >= 0.0f) {
      int ci[3];
      const float p[3] = {sc[h].x, sc[h].y, sc[h].z};
      res_cell(a, p, ci);
      key = res_key(a, qmol[h], ci, lane);
    }
    q.id[h] = RES_NONE;
    const unsigned same = __match_any_sync(0xffffffffu, key);
    if (key != RES_NONE && __ffs(same) - 1 == lane) q.id[h] = res_first(a.rs_head[key], epoch);
    q.slo[h] = 0;
    q.shi[h] = (int)a.n;
    if (a.n_mol > 1 && sc[h].w >= 0.0f) {
      q.slo[h] = 2 * (int)a.mol_off[qmol[h]];
      q.shi[h] = 2 * (int)a.mol_off[qmol[h] + 1];
    }
  }
}
// Pairs of the lanes' beads (`in`) with the items of those lists.
template <class Real>
__device__ __forceinline__ void res_walk(const KArgs<Real>& a, ResQuery& q, const float4* sc, int sA, int g, bool in,
                                         bool st_g, float4 mp, float4* win, int* gi, float4* gc, int* list, int& cnt,
                                         int& total) {
  const int lane = threadIdx.x & 31;
  const unsigned most = (unsigned)(a.nseg16 + a.n);   // items there are at most
  for (unsigned walked = 0; walked <= most && __any_sync(0xffffffffu, q.id[0] != RES_NONE || q.id[1] != RES_NONE); ++walked) {
    const int hq = q.id[0] != RES_NONE ? 0 : 1;
    const unsigned e = hq ? q.id[1] : q.id[0];
    bool acc = false;
    int ir = 0;
    float4 it = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (e != RES_NONE) {
      const unsigned nx = a.rs_next[e];
      ir = res_item(a, e, it);
      if (hq) q.id[1] = nx; else q.id[0] = nx;
      const int j0 = ir & ENT_JMASK, js = j0 / SEG_W, s = sA + hq;
      const int lo_h = hq ? q.slo[1] : q.slo[0], hi_h = hq ? q.shi[1] : q.shi[0];
      if (j0 >= lo_h && j0 < hi_h && (js > s + 1 || js < s - 1)) acc = cl_spheres_meet(a, hq ? sc[1] : sc[0], it);
    }
    cl_items(a, lane, g, in, st_g, sc, mp, acc, hq, ir, it, win, gi, gc, list, cnt, total);
  }
}
// The second parts (slots n0 on) of segments that span two molecules.  Out of
// line: they are rare.
template <class Real>
__device__ __noinline__ int2 res_list_second(const KArgs<Real>& a, int sA, float4 scA, float4 scB, int n0A, int n0B, int g,
                                             bool in, bool st_g, float4 mp, unsigned long long epoch, float4* win, int* gi,
                                             float4* gc, int* list, int cnt, int total) {
  const float4 sc[2] = {scA, scB};
  const int qmol[2] = {scA.w >= 0.0f ? __float_as_int(a.wpos[SEG_W * sA + n0A].w) : 0,
                       scB.w >= 0.0f ? __float_as_int(a.wpos[SEG_W * (sA + 1) + n0B].w) : 0};
  ResQuery q;
  res_query(a, sc, qmol, epoch, q);
  res_walk(a, q, sc, sA, g, in, st_g, mp, win, gi, gc, list, cnt, total);
  return make_int2(cnt, total);
}

// Lists of the `nb` (16 or 32) beads from slot g0 on, one lane per bead.
template <class Real>
__device__ __forceinline__ void res_list(const KArgs<Real>& a, int g0, int nb, unsigned long long epoch, float4* win, int* gi,
                                         float4* gc, int* list, int& cnt, int& total) {
  const int lane = threadIdx.x & 31;
  const int g = g0 + lane;
  const bool in = lane < nb && g < (int)a.n;
  float4 raw[2];
  int word[2];
  bool val[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int j = g0 - 16 + lane + 32 * h;
    val[h] = j >= 0 && j < (int)a.n;
    raw[h] = val[h] ? a.wpos[j] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    word[h] = val[h] ? ((a.topo[j] & F_STERIC) | CL_VALID) : 0;
  }
  const int sA = g0 / SEG_W;
  const bool hasB = nb > 16 && sA + 1 < (int)a.nseg16;
  const float4 none = make_float4(0.0f, 0.0f, 0.0f, -1.0f);
  const float4 sc[2] = {a.segc[sA], hasB ? a.segc[sA + 1] : none};
  // slots of the first parts
  const int n0A = a.n_mol > 1 ? a.rs_part[sA] : SEG_W, n0B = a.n_mol > 1 && hasB ? a.rs_part[sA + 1] : SEG_W;
  const float4 mp = in ? a.wpos[g] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  // molecule of each segment's first slot (staged slots 16 and 32)
  const int qmol[2] = {__shfl_sync(0xffffffffu, __float_as_int(raw[0].w), 16),
                       __shfl_sync(0xffffffffu, __float_as_int(raw[1].w), 0)};
  ResQuery q;
  res_query(a, sc, qmol, epoch, q);
  const bool fast = cl_stage(a, lane, raw, word, val, win);   // while the heads load
  bool st_g = false;
  cl_window(a, g0, lane, in, fast, win, st_g, list, cnt, total);
  __syncwarp();
  const bool second = (lane & 15) >= ((lane >> 4) ? n0B : n0A);   // of the segment's second molecule
  res_walk(a, q, sc, sA, g, in && !second, st_g, mp, win, gi, gc, list, cnt, total);
  const bool spA = sc[0].w >= 0.0f && n0A < min(SEG_W, (int)a.n - g0);
  const bool spB = sc[1].w >= 0.0f && n0B < min(SEG_W, (int)a.n - g0 - SEG_W);
  if (spA || spB) {
    const int2 r = res_list_second(a, sA, spA ? a.rs_sph1[sA] : none, spB ? a.rs_sph1[sA + 1] : none, n0A, n0B, g,
                                   in && second, st_g, mp, epoch, win, gi, gc, list, cnt, total);
    cnt = r.x;
    total = r.y;
  }
  // a wide segment: each of its beads queries its own 27 cells
  const int lh = lane >> 4;
  if (in && (lh == 0 || hasB) && (lh ? sc[1].w : sc[0].w) < 0.0f) {
    const int2 r = res_list_bead(a, g, mp, st_g, epoch, list, cnt, total);
    cnt = r.x;
    total = r.y;
  }
  __syncwarp();
}

// Arguments of a single force evaluation (ONCE).
template <bool ONCE>
struct ResOnce {};
template <>
struct ResOnce<true> {
  const double* X;              // [n][3] centres
  const double* u;              // [n][3] orientations
  double* Fb;                   // [n][3] bead and patch forces
  double* Fp;
  unsigned* err;                // error bits (host memory, mapped)
  int steric_phase;
  unsigned call;                // number of the call (once_calls.h)
  int off[DSDNA_NOALLOC_MAX_MOL + 1];   // base-pair offsets of the molecules
};

// ---------------------------------------------------------------- the kernel
// Bound by latency: a step is the grid barrier, one pass of owners and pairs
// out of shared memory and one pass of updates.
// ONCE: one force evaluation of a configuration given in device memory instead
// of steps (linear molecules, no loads): flags, mirror and lists are made from
// it on the way, and the site forces go straight to the caller's arrays.
template <class Real, bool EXT, bool ONCE = false>
__global__ void __launch_bounds__(res_max_threads<Real>(), 1)
    resident_kernel(const __grid_constant__ KArgs<Real> a, const __grid_constant__ ResLayout lay,
                    const __grid_constant__ ResOnce<ONCE> once) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ unsigned s_fl[2], s_word, s_to;
  __shared__ int s_scan[33], s_nx, s_nj;
  SPos<Real>* const spos2[2] = {reinterpret_cast<SPos<Real>*>(sm + lay.pos) + RES_HALO,
                                reinterpret_cast<SPos<Real>*>(sm + lay.pos) + lay.len + 3 * RES_HALO};
  int* const flg = reinterpret_cast<int*>(sm + lay.flg) + RES_HALO;
  Real* const cs = reinterpret_cast<Real*>(sm + lay.cs);
  Real* const cn = reinterpret_cast<Real*>(sm + lay.cn);
  Real* const cp = reinterpret_cast<Real*>(sm + lay.cp);
  Real* const pf = reinterpret_cast<Real*>(sm + lay.pf);
  int* const ent = reinterpret_cast<int*>(sm + lay.ent);
  int* const off = reinterpret_cast<int*>(sm + lay.off);
  unsigned short* const po = reinterpret_cast<unsigned short*>(sm + lay.po);
  short* const jx = reinterpret_cast<short*>(sm + lay.jx);
  int* const xo = reinterpret_cast<int*>(sm + lay.xo);
  short* const xw = reinterpret_cast<short*>(sm + lay.xw);
  Real* const ext = reinterpret_cast<Real*>(sm + lay.load);   // applied loads of last base pairs: [6][len]
  const int OC = lay.own;
  const unsigned ns = (unsigned)a.ns;
  const int i = threadIdx.x, lane = i & 31, warp = i >> 5, nwarp = (int)(blockDim.x >> 5);
  const int nwork = nwarp - 1;          // the last warp agrees with the other CTAs while these evaluate forces
  const bool sync_warp = warp == nwork;
  int* const list = reinterpret_cast<int*>(sm + lay.list) + (warp * 32 + lane) * LIST_CAP;
  float4* const win = reinterpret_cast<float4*>(sm + lay.win) + warp * (CL_WIN + CL_WIN / 16);
  int* const gi = reinterpret_cast<int*>(sm + lay.gi) + warp * 4;
  float4* const gc = reinterpret_cast<float4*>(sm + lay.gc) + warp * 4;

  // the CTA's stretch, and the nucleotide of this thread
  const int s0 = SEG_W * (int)((int64_t)blockIdx.x * a.nseg16 / gridDim.x);
  const int s1 = min((int)a.n, SEG_W * (int)((int64_t)(blockIdx.x + 1) * a.nseg16 / gridDim.x));
  const int len = s1 - s0;
  const bool mine = i < len;
  const int g = s0 + i;
  const unsigned gu = (unsigned)(mine ? g : s0);

  const int64_t step0 = ONCE ? 0 : *a.step;
  int64_t budget = ONCE ? 1 : (a.steps_left ? *a.steps_left : a.nsteps);
  if (!ONCE && (*a.err & B_ERRMASK)) budget = 0;
  unsigned seq0, phase = 0u;
  unsigned long long epoch;
  if constexpr (ONCE) {
    phase = once.call;
    epoch = once.call;
    seq0 = once.call + 1u;
  } else {
    seq0 = *a.rs_seq;
    epoch = *a.nrebuild;
  }
  int cur = (int)(step0 & 1);

  // state into registers and shared memory
  double Xd[3] = {0, 0, 0}, Vd[3] = {0, 0, 0};
  V3<Real> Om{0, 0, 0};
  int kr[3] = {0, 0, 0}, packed = 0, f = 0;
  if constexpr (ONCE) {
    if (blockIdx.x == 0)
      for (int m = i; m <= a.n_mol; m += blockDim.x) const_cast<int64_t*>(a.mol_off)[m] = once.off[m];
    if (mine) {
      int lo = 0, hi = a.n_mol - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (once.off[mid] <= g >> 1) lo = mid; else hi = mid - 1;
      }
      const int N = once.off[lo + 1] - once.off[lo], k = (g >> 1) - once.off[lo], q = (g & 1) ? N - 1 - k : k;
      f = (q % 3 == once.steric_phase ? F_STERIC : 0) | (q > 0 ? F_PREV : 0) | (q < N - 1 ? F_NEXT : 0) | (lo << MOL_SHIFT);
      double w[3];
      for (int c = 0; c < 3; ++c) { Xd[c] = once.X[3 * gu + c]; w[c] = once.u[3 * gu + c]; }
      const double l2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
      if (fabs(l2 - 1.0) > 1e-6) { const double l = sqrt(l2); w[0] /= l; w[1] /= l; w[2] /= l; }
      const SPos<Real> me{fixs(Xd[0], a.fixS[0]), fixs(Xd[1], a.fixS[1]), fixs(Xd[2], a.fixS[2]),
                          (Real)w[0], (Real)w[1], (Real)w[2]};
      spos2[0][i] = me;
      a.topo[gu] = f;
      flg[i] = f;
      rec_store(a, cur, gu, seq0, f, me);
    }
  } else if (mine) {
    SPos<Real> me;
    load_slot(a, cur, g, me);
    spos2[0][i] = me;
    f = a.topo[gu];
    rec_store(a, cur, gu, seq0, f, me);
    flg[i] = f;
    if constexpr (sizeof(Real) == 4) {
      Xd[0] = a.X[gu]; Xd[1] = a.X[ns + gu]; Xd[2] = a.X[2 * ns + gu];
      packed = a.Kw[(unsigned)cur * ns + gu].w;
    } else {
      Xd[0] = me.x; Xd[1] = me.y; Xd[2] = me.z;
    }
    Vd[0] = a.V[gu]; Vd[1] = a.V[ns + gu]; Vd[2] = a.V[2 * ns + gu];
    Om = V3<Real>{a.Om[gu], a.Om[ns + gu], a.Om[2 * ns + gu]};
    kr[0] = a.kref[gu]; kr[1] = a.kref[ns + gu]; kr[2] = a.kref[2 * ns + gu];
    if (f & F_TOP) {
      V3<Real> Fe, Tq;
      read_load(a, f >> MOL_SHIFT, Fe, Tq);
      ext[i] = Fe.x; ext[lay.len + i] = Fe.y; ext[2 * lay.len + i] = Fe.z;
      ext[3 * lay.len + i] = Tq.x; ext[4 * lay.len + i] = Tq.y; ext[5 * lay.len + i] = Tq.z;
    }
  }
  const int mol = f >> MOL_SHIFT;
  const bool frozen = (f & F_FROZEN) != 0;
  const uint32_t local = mine && !ONCE ? (uint32_t)(g - 2 * (int)a.mol_off[mol]) : 0u;
  if (i == 0) { s_fl[0] = 0u; s_fl[1] = 0u; s_nx = 0; s_nj = 0; s_to = 0u; s_word = 0u; }
  __syncthreads();
  if constexpr (EXT) {
    // circular molecules: the owners next to a junction, listed apart (slot xo,
    // place xw in the owner table); the end nucleotides of a strand also take
    // the forces of the owner across the junction, evaluated here a second time
    // (places len + 4 + jx)
    if (a.n_junc) {
      for (int w = i; w < len + 4; w += blockDim.x) {
        const int o = s0 - 2 + w;
        if (o < 0 || o >= (int)a.n || !(a.topo[o] & F_JUNC)) continue;
        const int x = atomicAdd(&s_nj, 1);
        xo[x] = o;
        xw[x] = (short)w;
      }
      if (mine) {
        jx[i] = -1;
        if (f & F_JUNC) {
          const int k0 = (int)a.mol_off[mol], k1 = (int)a.mol_off[mol + 1] - 1, k = g >> 1;
          if (k == k0 || k == k1) {
            const int x = atomicAdd(&s_nj, 1), y = atomicAdd(&s_nx, 1);
            jx[i] = (short)y;
            xo[x] = 2 * (k == k0 ? k1 : k0) + (g & 1);
            xw[x] = (short)(len + 4 + y);
          }
        }
      }
    }
    if (a.bubble && mine && !(i & 1)) {
      const SPos<Real> pa = spos2[0][i], pb = spos2[0][i + 1];
      const V3<Real> d = rel(pa, pb, a.fixq) + a.c.h * (uvec(pb) - uvec(pa));
      if (dot(d, d) > a.c.rchb2) flg[i] = f | F_OPEN;
    }
  }

  // offsets of the nucleotides' list entries in the CTA's pair table (block scan)
  int npair = 0;
  auto number_pairs = [&](int cnt) {
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_scan[warp] = incl;
    __syncthreads();
    int before = 0, tot = 0;
    for (int w = 0; w < nwarp; ++w) {
      if (w == warp) before = tot;
      tot += s_scan[w];
    }
    if (mine) off[i] = before + incl - cnt;
    if (i == 0) off[len] = tot;
    npair = tot;
    __syncthreads();
  };
  auto keep_entry = [&](int q, int e) {
    const int p = off[i] + q;
    if (p < lay.pairs) { ent[p] = e; po[p] = (unsigned short)i; }
  };
  if constexpr (!ONCE) {
    const int cnt = mine ? a.ncnt[gu] : 0;
    number_pairs(cnt);
    for (int q = 0; q < cnt; ++q) keep_entry(q, a.nbr[(unsigned)q * ns + gu]);
  }
  const int njo = EXT ? s_nj : 0;
  // halo slot of this lane (edge_chunk), its static flags
  const int hl = lane < RES_HALO ? lane - RES_HALO : len + lane - RES_HALO, hs = s0 + hl;
  const bool halo = lane < 2 * RES_HALO && hs >= 0 && hs < (int)a.n;
  int hf = !ONCE && halo ? a.topo[hs] : 0;
  __syncthreads();

  unsigned errbits = 0, seq = seq0;
  SPos<Real>* spos = spos2[0];
  unsigned fl = 0;   // this thread's flags of the step
  // owners within `edge` slots of an end read the halo (five base pairs with the bubble rule)
  const int edge = EXT && a.bubble ? 6 : 2;
  const int e0 = min(edge, len), e1 = max(len - edge, e0);   // interior: local slots [e0, e1)

  auto store_out = [&](int w, const OwnerOut<Real>& out) {
    cs[0 * OC + w] = out.sb.x; cs[1 * OC + w] = out.sb.y; cs[2 * OC + w] = out.sb.z;
    cs[3 * OC + w] = out.sp.x; cs[4 * OC + w] = out.sp.y; cs[5 * OC + w] = out.sp.z;
    cn[0 * OC + w] = out.nb.x; cn[1 * OC + w] = out.nb.y; cn[2 * OC + w] = out.nb.z;
    cn[3 * OC + w] = out.np.x; cn[4 * OC + w] = out.np.y; cn[5 * OC + w] = out.np.z;
    cp[0 * OC + w] = out.pp.x; cp[1 * OC + w] = out.pp.y; cp[2 * OC + w] = out.pp.z;
  };
  // owner of local slot l (-2 .. len + 1; lanes with `on`)
  auto owner = [&](int l, bool on) {
    const int fo = on ? flg[l] : 0;
    if (!on || (EXT && (fo & F_JUNC))) return;
    OwnerOut<Real> out{{0, 0, 0}, {0, 0, 0}, {0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    if (fo & F_NEXT) {
      const ResSrc<Real> src{spos, flg, s0};
      unsigned rm = 0u;
      if constexpr (EXT) {
        if (a.bubble) {
          const bool home = l >= 0 && l < len;
          rm = bubble_bits(a, src, s0 + l, fo, home);
          if (home && rm) atomicOr(&flg[l], (int)(rm << RM_SHIFT));   // as in the topology word
        }
      }
      owner_eval<Real>(a, src, s0 + l, fo, rm, fl, (Real*)nullptr, (Real*)nullptr, out);
    }
    store_out(l + 2, out);
  };
  // the halo into shared memory, then the owners near both ends
  auto edge_chunk = [&] {
    int fh = 0;
    if (halo) {
      unsigned rm0 = 0u;
      spos[hl] = rec_load(a, cur, (unsigned)hs, seq, &s_to, &rm0);
      fh = (hf & ~(3 << RM_SHIFT)) | (int)(rm0 << RM_SHIFT);
    }
    __syncwarp();
    if (lane < 2 * RES_HALO) {
      if (EXT && a.bubble && halo && !(lane & 1)) {
        const SPos<Real> pa = spos[hl], pb = spos[hl + 1];
        const V3<Real> d = rel(pa, pb, a.fixq) + a.c.h * (uvec(pb) - uvec(pa));
        if (dot(d, d) > a.c.rchb2) fh |= F_OPEN;
      }
      flg[hl] = fh;
    }
    __syncwarp();
    const int lo = 2 + e0, hi = len + 2 - e1;   // owners at either end
    owner(lane < lo ? lane - 2 : e1 + lane - lo, lane < lo + hi);
    __syncwarp();
  };
  // owners next to junctions of circular molecules
  auto junction_chunk = [&](int c) {
    const int x = 32 * c + lane;
    const bool on = x < njo;
    ResJunc<Real> src{a, spos, flg, &s_to, cur, seq, s0, len, 0, 0, {}, {}};
    int o = 0;
    if (on) {
      o = xo[x];
      const int m = a.topo[o] >> MOL_SHIFT;
      src.off = (int)a.mol_off[m];
      src.N = (int)a.mol_off[m + 1] - src.off;
      src.load(o);
    }
    __syncwarp();   // the lanes that waited for a record join the others
    if (on) {
      const int w = xw[x];
      const unsigned l = (unsigned)(o - s0);
      const bool home = w >= 2 && w < len + 2;
      int fo = (l < (unsigned)len ? flg[l] : a.topo[o]) | F_PREV | F_NEXT;   // both neighbours exist on a ring
      unsigned rm = 0u;
      if constexpr (EXT) {
        if (a.bubble) {
          if (l >= (unsigned)len) {   // removed terms as of this step: the topology word may be a step ahead
            unsigned rm0 = 0u;
            rec_load(a, cur, (unsigned)o, seq, &s_to, &rm0);
            fo = (fo & ~(3 << RM_SHIFT)) | (int)(rm0 << RM_SHIFT);
          }
          rm = bubble_bits(a, src, o, fo, home);
          if (home && rm) atomicOr(&flg[l], (int)(rm << RM_SHIFT));
        }
      }
      OwnerOut<Real> out{{0, 0, 0}, {0, 0, 0}, {0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
      owner_eval<Real>(a, src, o, fo, rm, fl, (Real*)nullptr, (Real*)nullptr, out);
      store_out(w, out);
    }
    __syncwarp();
  };
  // partner of list entry e: from shared memory, or its records
  auto partner = [&](int e, int& fj) {
    const int j = e & ENT_JMASK;
    const unsigned l = (unsigned)(j - s0);
    if (l < (unsigned)len) {
      fj = flg[l];
      return spos[l];
    }
    fj = a.topo[j];
    return rec_load(a, cur, (unsigned)j, seq, &s_to);
  };
  // pairs 32 c .. of the table
  auto pair_chunk = [&](int c) {
    const int p = 32 * c + lane;
    const bool on = p < npair;
    int b = 0, e = 0, fj = 0;
    SPos<Real> q{};
    if (on) {
      b = po[p];
      e = ent[p];
      q = partner(e, fj);
    }
    __syncwarp();   // the lanes that waited for a record join the others
    if (on) {
      const V3<Real> fw = res_pair(a, s0, b, spos[b], flg[b], e, q, fj);
      Real* o = pf + 3 * p;
      o[0] = fw.x; o[1] = fw.y; o[2] = fw.z;
    }
  };
  // the sync warp: this CTA's flags out, every CTA's in (to s_word)
  auto agree = [&](unsigned* flags, auto meanwhile) {
    ++phase;
    if (sync_warp) {
      if (lane == 0) {
        res_publish(a, phase, *flags);
        *flags = 0u;
      }
      meanwhile();
      if (lane == 0) s_word = res_agree(a, phase);
    }
  };
  // A list beyond its capacity is agreed on one step after its build, and that
  // step, without the pairs left out, is not kept: positions and velocities at
  // the build wait in the list buffer (free until the next build; the lanes'
  // words side by side), orientations in the other position buffer.  Written to
  // memory instead, they had to arrive before the next agreement: 10 kbp 652 ->
  // 664 us per 100 steps, here 660.
  int* const kept = reinterpret_cast<int*>(sm + lay.list) + warp * 32 * LIST_CAP + lane;
  auto keep_state = [&](bool back) {
    int w = 0;
    auto word = [&](int& x) {
      if (back) x = kept[32 * w]; else kept[32 * w] = x;
      ++w;
    };
    auto real = [&](auto& x) {
      int p[sizeof(x) / 4];
      memcpy(p, &x, sizeof(x));
      for (unsigned q = 0; q < sizeof(x) / 4; ++q) word(p[q]);
      memcpy(&x, p, sizeof(x));
    };
    static_assert(LIST_CAP >= 18, "the words of a state fit its lane's share of the list buffer");
    for (int c = 0; c < 3; ++c) { real(Xd[c]); real(Vd[c]); }
    real(Om.x); real(Om.y); real(Om.z);
  };
  // bin the beads, thread the segments into the hash, wait for all, build the
  // CTA's own lists
  auto rebuild = [&](unsigned* flags) {
    ++epoch;
    const int nw_i = (len + 31) & ~31;
    unsigned e = 0;
    if (i < nw_i) {   // whole warps
      float pw[3] = {0.0f, 0.0f, 0.0f};
      if (mine) {
        const float hf = (float)a.c.h;
        const SPos<Real> me = spos[i];
        float b[3];
        if constexpr (sizeof(Real) == 4) {
          b[0] = d2f_words(Xd[0]) - hf * me.ux;
          b[1] = d2f_words(Xd[1]) - hf * me.uy;
          b[2] = d2f_words(Xd[2]) - hf * me.uz;
          kr[0] = me.kx + bead_off(hf * me.ux, a.fixSf[0]);
          kr[1] = me.ky + bead_off(hf * me.uy, a.fixSf[1]);
          kr[2] = me.kz + bead_off(hf * me.uz, a.fixSf[2]);
        } else {
          const double uu[3] = {me.ux, me.uy, me.uz};
          for (int c = 0; c < 3; ++c) {
            b[c] = (float)(Xd[c] - (double)hf * uu[c]);
            kr[c] = fixs(Xd[c], a.fixS[c]) + bead_off(hf * (float)uu[c], a.fixSf[c]);
          }
        }
        int wi[3] = {0, 0, 0};
        for (int c = 0; c < 3; ++c) {
          float x = b[c];
          if (a.periodic) {
            const float qf = floorf(x * a.invLf[c]);
            wi[c] = (int)qf;
            x = fmaf(-qf, a.Lf[c], x);
            if (wi[c] > 511 || wi[c] < -512) e |= B_EIMG;
          }
          pw[c] = x;
        }
        packed = (wi[0] & 0x3ff) | ((wi[1] & 0x3ff) << 10) | ((wi[2] & 0x3ff) << 20) | ((f & F_STERIC) << IMG_STERIC_SHIFT);
        a.wpos[gu] = make_float4(pw[0], pw[1], pw[2], __int_as_float(mol));
        if constexpr (sizeof(Real) == 8) a.img[gu] = packed;
      }
      // the segment's parts: one molecule, or two of them
      int mlo = mine ? mol : INT_MAX, mhi = mine ? mol : INT_MIN;
      if (a.n_mol > 1)
        for (int o = 8; o > 0; o >>= 1) {
          mlo = min(mlo, __shfl_xor_sync(0xffffffffu, mlo, o, 16));
          mhi = max(mhi, __shfl_xor_sync(0xffffffffu, mhi, o, 16));
        }
      const unsigned half = 0xffffu << (lane & 16);
      const bool first = mine && mol == mlo, second = mine && mol == mhi && mhi != mlo;
      const int n0 = __popc(__ballot_sync(0xffffffffu, first) & half);
      const bool more = (__ballot_sync(0xffffffffu, mine && !first && !second) & half) != 0u;   // a third molecule
      const bool two = (__ballot_sync(0xffffffffu, second) & half) != 0u;
      float c3[3], d3[3] = {0.0f, 0.0f, 0.0f};
      const float R = seg_sphere(a, first, 0, pw, c3);
      float R1 = 0.0f;
      if (__any_sync(0xffffffffu, two)) R1 = seg_sphere(a, second, n0 & 15, pw, d3);
      const bool wide = more || !(R <= a.rs_rcap) || (two && !(R1 <= a.rs_rcap));
      if (mine && (lane & 15) == 0) {
        a.segc[g >> 4] = make_float4(c3[0], c3[1], c3[2], wide ? -1.0f : R);
        a.rs_part[g >> 4] = n0;
        if (!wide) res_insert(a, mol, c3, (unsigned)(g >> 4), epoch);
      }
      if (two && second && !wide && (lane & 15) == n0) {
        a.rs_sph1[g >> 4] = make_float4(d3[0], d3[1], d3[2], R1);
        res_insert(a, mol, d3, (unsigned)a.nseg16 + gu, epoch);
      }
      if (mine && wide) res_insert(a, mol, pw, (unsigned)a.nseg16 + gu, epoch);
    }
    e = __reduce_or_sync(0xffffffffu, e);
    if (lane == 0 && e) atomicOr(flags, e);
    __syncthreads();
    agree(flags, [] {});
    __syncthreads();
    if (s_word & B_ERRMASK) return false;
    int cnt = 0, total = 0;
    if (i < nw_i) {
      const int g0 = s0 + 32 * warp;
      res_list(a, g0, min(32, SEG_W * ((s1 - g0 + SEG_W - 1) / SEG_W)), epoch, win, gi, gc, list, cnt, total);
      if (mine) {
        if (total > a.cap) fl |= B_EOVF;
        for (int q = 0; q < cnt; ++q) a.nbr[(unsigned)q * ns + gu] = list[q];
        a.ncnt[gu] = cnt;
      }
    }
    number_pairs(mine ? cnt : 0);
    for (int q = 0; q < cnt; ++q) keep_entry(q, list[q]);
    if constexpr (!ONCE) {
      __syncwarp();   // the lanes' lists are read
      keep_state(false);
    }
    if (blockIdx.x == 0 && i == 0) *a.nrebuild += 1;
    __syncthreads();
    return true;
  };

  int64_t it = 0;   // steps taken
  if constexpr (ONCE) {
    if (!rebuild(&s_fl[1])) {
      budget = 0;
      errbits = s_word;
    }
    if (halo) hf = a.topo[hs];
  }
  for (;; ++it) {
    const bool end = it == budget;
    const int64_t step = step0 + it;
    cur = (int)(step & 1);
    const int nxt = cur ^ 1;
    spos = (it & 1) ? spos2[1] : spos2[0];
    SPos<Real>* const snxt = (it & 1) ? spos2[0] : spos2[1];
    seq = seq0 + (unsigned)it;
    V3<Real> eb{0, 0, 0}, ep{0, 0, 0};
    unsigned* const before = &s_fl[(it + 1) & 1];   // flags of the step before
    auto draw_noise = [&] {
      if (!ONCE && mine && !frozen && !end) nucleotide_noise(a, local, step, mol, eb, ep);
    };
    if (!sync_warp && !end) {
      // owners and list pairs, 32 at a time: the ends, which wait for the
      // neighbours, to the last warp alone, then owners to the last warps first,
      // so that the first ones, whose threads also draw the noise, hold pairs
      const int nj = (njo + 31) >> 5, nco = nj + ((e1 - e0 + 31) >> 5);
      const int ncp = npair <= lay.pairs ? (npair + 31) >> 5 : 0;
      const int nrest = nwork > 1 ? nwork - 1 : 1;
      // a warp with a junction chunk, which waits for other stretches too, gets
      // no other chunk while these are at most half of the warps: with a share of
      // the others it was last by 2000 of a step's 13,000 cycles (100 steps of 64
      // rings of 500 bp 1185 -> 1129 us).  Up to three tiles there are warps for
      // all chunks at once (kern_launch.cuh) and none is kept free (1% slower).
      const int jw = lay.len > 96 && 2 * nj <= nrest ? nj : 0, w0 = nrest - 1 - warp;
      if (warp == nwork - 1) edge_chunk();
      if (warp < nrest)
        for (int c = w0; c < (w0 < jw ? nj : nco + ncp); c += w0 < jw ? nj : nrest - jw) {
          if (c < nj) junction_chunk(c);
          else if (c < nco) owner(e0 + 32 * (c - nj) + lane, e0 + 32 * (c - nj) + lane < e1);
          else pair_chunk(c - nco);
        }
    }
    if (it > 0) agree(before, [&] { if (sync_warp) draw_noise(); });
    if (!sync_warp || it == 0) draw_noise();
    __syncthreads();
    if (it > 0) {
      const unsigned r = s_word;
      if (r & B_ERRMASK) {   // the last step was not taken
        errbits = r;
        --it;
        if (r & B_EOVF) {
          keep_state(true);
          spos = snxt;
        }
        break;
      }
      if (r & B_STALE) {
        if (!rebuild(before)) { errbits = s_word; break; }
        if (!end) {   // the pair forces once more, from the new lists
          const int ncp = npair <= lay.pairs ? (npair + 31) >> 5 : 0;
          for (int c = warp; c < ncp; c += nwarp) pair_chunk(c);
          __syncthreads();
        }
      }
    }
    if (end) break;
    // every nucleotide: forces in the order of nucleotide_pass, then its step
    if (mine) {
      const SPos<Real> me = spos[i], q = spos[i ^ 1];
      const Real h = a.c.h;
      const V3<Real> um = uvec(me);
      const int w = i + 2, dir = (i & 1) ? -2 : 2;
      V3<Real> Fb{cs[0 * OC + w], cs[1 * OC + w], cs[2 * OC + w]};
      V3<Real> Fp{cs[3 * OC + w], cs[4 * OC + w], cs[5 * OC + w]};
      if constexpr (EXT) {
        if ((f & F_JUNC) && jx[i] >= 0) {   // the owner across the junction: the previous or the next one
          const int x = len + 4 + jx[i];
          const bool first = (i & 1) ? g >> 1 != (int)a.mol_off[mol] : g >> 1 == (int)a.mol_off[mol];
          if (first) {
            Fb += V3<Real>{cn[0 * OC + x], cn[1 * OC + x], cn[2 * OC + x]};
            Fp += V3<Real>{cn[3 * OC + x], cn[4 * OC + x], cn[5 * OC + x]};
          } else {
            Fp += V3<Real>{cp[0 * OC + x], cp[1 * OC + x], cp[2 * OC + x]};
          }
        }
      }
      if (f & F_PREV) {
        const int op = w - dir;
        Fb += V3<Real>{cn[0 * OC + op], cn[1 * OC + op], cn[2 * OC + op]};
        Fp += V3<Real>{cn[3 * OC + op], cn[4 * OC + op], cn[5 * OC + op]};
      }
      if (f & F_NEXT) {
        const int on = w + dir;
        Fp += V3<Real>{cp[0 * OC + on], cp[1 * OC + on], cp[2 * OC + on]};
      }
      {
        V3<Real> d;
        Real r2, k2;
        if (hbond(a, me, q, um, f, d, r2, k2)) Fp += k2 * d;
      }
      if (npair <= lay.pairs) {
        for (int p = off[i], p1 = off[i + 1]; p < p1; ++p) Fb += V3<Real>{pf[3 * p], pf[3 * p + 1], pf[3 * p + 2]};
      } else {   // more entries than the table holds: this nucleotide's list, from memory
        for (int p = 0, nn = off[i + 1] - off[i]; p < nn; ++p) {
          const int e = a.nbr[(unsigned)p * ns + gu];
          int fj;
          const SPos<Real> qj = partner(e, fj);
          Fb += res_pair(a, s0, i, me, f, e, qj, fj);
        }
      }
      if constexpr (ONCE) {
        double *ob = once.Fb + 3 * gu, *op = once.Fp + 3 * gu;
        ob[0] = Fb.x; ob[1] = Fb.y; ob[2] = Fb.z;
        op[0] = Fp.x; op[1] = Fp.y; op[2] = Fp.z;
      } else {
      if (f & F_TOP)
        add_load(a, V3<Real>{ext[i], ext[lay.len + i], ext[2 * lay.len + i]},
                 V3<Real>{ext[3 * lay.len + i], ext[4 * lay.len + i], ext[5 * lay.len + i]}, me, q, Fb, Fp);
      const V3<Real> F = Fb + Fp;
      const V3<Real> Tc = h * cross(um, Fp - Fb);
      V3<Real> un = um;
      if (!frozen) {
        V3<Real> Ft, Tt;
        langevin(a, F, Tc, Vd, Om, um, eb, ep, Ft, Tt);
        kick_drift(a, Ft, Tt, um, Xd, Vd, Om, un, fl);
      }
      const int k0 = fixs(Xd[0], a.fixS[0]), k1 = fixs(Xd[1], a.fixS[1]), k2 = fixs(Xd[2], a.fixS[2]);
      SPos<Real> nw;
      if constexpr (sizeof(Real) == 4) nw = SPos<Real>{k0, k1, k2, un.x, un.y, un.z};
      else nw = SPos<Real>{Xd[0], Xd[1], Xd[2], un.x, un.y, un.z};
      rec_store(a, nxt, gu, seq0 + (unsigned)it + 1u, EXT ? flg[i] : 0, nw);
      snxt[i] = nw;
      if (moved(a, k0, k1, k2, un, kr)) fl |= B_STALE;
      }
    }
    if constexpr (ONCE) break;
    if constexpr (EXT) {
      if (a.bubble) {
        __syncwarp();
        if (mine && !(i & 1)) {
          const SPos<Real> pa = snxt[i], pb = snxt[i + 1];
          const V3<Real> d = rel(pa, pb, a.fixq) + a.c.h * (uvec(pb) - uvec(pa));
          const int fi = flg[i] & ~F_OPEN;
          flg[i] = dot(d, d) > a.c.rchb2 ? fi | F_OPEN : fi;
        }
      }
    }
    if (i == 0 && s_to) fl |= B_ETIMEOUT;
    fl = __reduce_or_sync(0xffffffffu, fl);
    if (lane == 0 && fl) atomicOr(&s_fl[it & 1], fl);
    fl = 0;
    __syncthreads();   // the next step's positions and this step's flags are complete
  }
  if constexpr (ONCE) {
    if (i == 0 && s_to) fl |= B_ETIMEOUT;
    fl = (__reduce_or_sync(0xffffffffu, fl) | errbits) & B_ERRMASK;
    if (lane == 0 && fl) atomicOr_system(once.err, fl);
    return;
  }
  const int64_t done = it;
  // state back to memory: orientation and mirror into the buffer of the step
  // the launch ends at, into both after an error
  if (mine) {
    const SPos<Real> me = spos[i];
    for (int o = 0; o < (errbits ? 2 : 1); ++o) {
      const int buf = (int)((step0 + done + o) & 1);
      if constexpr (sizeof(Real) == 4) {
        const double none[3] = {0, 0, 0};
        store_state(a, buf, (int64_t)gu, me.kx, me.ky, me.kz, none, uvec(me), packed);
      } else {
        store_state(a, buf, (int64_t)gu, 0, 0, 0, Xd, uvec(me), 0);
      }
    }
    if (sizeof(Real) == 4 && !frozen) { a.X[gu] = Xd[0]; a.X[ns + gu] = Xd[1]; a.X[2 * ns + gu] = Xd[2]; }
    a.V[gu] = Vd[0]; a.V[ns + gu] = Vd[1]; a.V[2 * ns + gu] = Vd[2];
    a.Om[gu] = Om.x; a.Om[ns + gu] = Om.y; a.Om[2 * ns + gu] = Om.z;
    a.kref[gu] = kr[0]; a.kref[ns + gu] = kr[1]; a.kref[2 * ns + gu] = kr[2];
  }
  if (__syncthreads_or((int)(fl & B_EOVF))) errbits |= B_EOVF;   // of a rebuild after the last step
  if (i == 0) {
    if (errbits & B_ERRMASK) atomicOr(a.err, errbits & B_ERRMASK);
    if (blockIdx.x == 0) {
      *a.step = step0 + done;
      *a.rs_seq = seq0 + (unsigned)budget + 2u;
      const int64_t left = budget - done;
      if (a.steps_left) *a.steps_left = left;
      if (a.use_cond) cudaGraphSetConditional(a.h_while, left > 0 && done > 0 && (errbits & B_ERRMASK) == 0 ? 1u : 0u);
    }
  }
}

}  // namespace dsdna

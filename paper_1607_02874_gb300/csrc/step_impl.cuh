// Fused collide-stream-boundary kernel and state readers, templated on the
// population storage. Included once per storage type and variant
// (step_f32.cu, step_f16.cu, step_bf16.cu, ...) so the units compile in
// parallel.
//
// Time stepping follows the lattice BGK equation of the paper's Appendix
// (Eq. LBE, Eq. feq, one omega for every species), with species relaxed
// towards an equilibrium built on the carrier velocity, halfway bounce-back
// of the carrier at solid links, and the sputtering law (Appendix,
// Eq. f_P_in) with S_ij = 1/b(x) at catalytic nodes.
//
// Streaming is in place (AA pattern): one population array per kind. Each
// cell owns 19 pointer slots per array, P_k, and a step loads the 19 values
// behind them and stores 19 new values to the same places:
//   - even step: P_k = own slot k. The load is the incoming population of
//     direction k; the store is the outgoing f*_opp(k) (so f*_i lands in own
//     slot opp(i));
//   - odd step: P_k = slot k of the neighbour x + c_k. The load is the
//     incoming population of direction opp(k) (the neighbour's even-step
//     output f*_opp(k)(x - c_opp(k))); the store is the outgoing f*_k, which
//     the neighbour reads as its incoming k after the step. After an odd
//     step the arrays hold the streamed populations in natural order again.
//   - when x + c_k is solid (or, on an inlet/outlet plane, outside the box)
//     the odd step's P_k is the cell's own slot opp(k): the store of f*_k
//     there is the halfway bounce-back that the next step reads as incoming
//     opp(k); the even step's own-slot pointers give the same by
//     construction.
//   - species leaving towards a catalytic solid stay in the slot of the link,
//     as the carrier does; after the cell updates the node kernels sum them per
//     node into the step's wall hits (A_cur) and overwrite the slots with what
//     the sputtering law returns, from the hits of the step before (A_prev).
//     So the wall re-emits one step after the hit, the timing of bounce-back,
//     with no grid-wide synchronisation.
//   - inlet plane z=0 / outlet plane z=nz-1: equilibrium with the velocity of
//     plane 1 / nz-2 from the previous step (and, at the outlet, the species
//     densities of plane nz-2), passed through a double-buffered plane cache.
//
// All arithmetic is on the stored scaled deviations d_i = (f_i - w_i rho_ref)
// / w_i (rho_ref = 1 for the carrier, 0 for the species): drho = sum w d,
// j = sum w c d (the w_i rho_ref parts cancel since sum w c = 0),
// rho = rho_ref + drho, u = j / rho. With P_i = 3 c.u + 4.5 (c.u)^2 - 1.5 u^2,
// the same for every array that relaxes towards the same u, the equilibria
// are deq_i = drho + rho P_i (carrier) and rho_s + rho_s P_i (species), and
// d*_i = (1 - omega) d_i + omega deq_i. The reactant and product of a slot
// move as one pair and relax with packed FP32x2 arithmetic.
#pragma once

#include <cooperative_groups.h>

#include <algorithm>

#include "lbm_internal.h"

namespace lbm {

// Population layout: two warp-blocked arrays (carrier a.f, species a.fs).
// Entry e, slot k lives at element (e / 32) 608 + 32 k + e % 32 of each
// (608 = 19 x 32): a warp's 32 consecutive entries are contiguous for every
// slot, and all slots of an entry are compile-time offsets from one base.
__device__ __forceinline__ int64_t ent_off(int32_t e) { return (int64_t)(e >> 5) * (kQ * 32) + (e & 31); }
// ent_off modulo 2^32: the difference of two of these is the exact element
// distance between two entries whenever that distance is below 2^31
__device__ __forceinline__ uint32_t ent_off32(int32_t e) { return (uint32_t)e + ((uint32_t)e >> 5) * (uint32_t)(kQ * 32 - 32); }

// The step's kernels follow one another on a stream with programmatic
// dependent launch: each lets the next one be scheduled as soon as all its
// own blocks have started (chain_next), and reads what earlier kernels wrote
// only after they have completed (chain_wait). Before the wait a kernel may
// read the lists and the geometry alone, which never change once a simulation
// exists; so a launch's latency and the index loads overlap the kernel before
// it. (Without the launch attribute both are no-ops.)
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// slots whose neighbour lies below / above the cell in z
constexpr uint32_t kDownBits = (1u << 6) | (1u << 12) | (1u << 13) | (1u << 16) | (1u << 17);
constexpr uint32_t kUpBits = (1u << 5) | (1u << 11) | (1u << 14) | (1u << 15) | (1u << 18);

// Population loads name their cache operator (ld.global.ca): never the
// non-coherent read-only path, which a const __restrict__ pointer would
// allow. Within one multi-step batched launch a CTA reads populations that
// other CTAs wrote earlier in the same launch; ordinary loads observe them
// after the step-ordering acquire, non-coherent loads need not.
// Population stores are streaming stores (st.global.cs): each stored value
// is read once, by the next step; coherence is unchanged.
template <typename T>
__device__ __forceinline__ T ld_pop(const T *p) {
  return __ldca(p);
}

// Wall hits of the previous step at node k, species row sp (0 R, 1 P): the
// node's total, or, under the random sputtering matrix, the sum over its
// link slots. And what the node re-emits along its outgoing link i: a share
// of the hits times 1/b (uniform matrix) or the link's own slot, whose rank
// is the number of active links below i (random matrix, factor 1).
template <bool DET>
__device__ __forceinline__ double hits_d(const StepArgs &a, int sp, int64_t k) {
  if (!a.rs) return acc_get_d<DET>(a.A_prev, LBM_OFF(a, kChkAcc, 0, sp * a.acc_row + k, LBM_NACC(a)));
  double h = 0.0;
  for (int32_t l = __ldg(a.node_off + LBM_OFF(a, kChkNode, 0, k, a.n_nodes + 1));
       l < __ldg(a.node_off + LBM_OFF(a, kChkNode, 0, k + 1, a.n_nodes + 1)); ++l)
    h += acc_get_d<DET>(a.A_prev, LBM_OFF(a, kChkAcc, 0, sp * a.acc_row + l, LBM_NACC(a)));
  return h;
}
// (rs: the random matrix, fixed at compile time on the step path; the
// observables' readers pass the simulation's runtime flag)
__device__ __forceinline__ int64_t emit_index(bool rs, const StepArgs &a, int i, int32_t node, int32_t node_cell) {
  if (!rs) return (int64_t)node;
  return (int64_t)__ldg(a.node_off + LBM_OFF(a, kChkNode, 0, node, a.n_nodes + 1)) +
         __popc(__ldg(a.cell_bits + LBM_OFF(a, kChkIdx, 0, node_cell, LBM_NCELLS(a))) & ((1u << i) - 1u));
}
__device__ __forceinline__ float emit_scale(bool rs, const StepArgs &a, int32_t node) {
  return rs ? 1.0f : __ldg(a.inv_b + LBM_OFF(a, kChkNode, 0, node, a.n_nodes));
}
// What a node that gathered AR and AP re-emits along its outgoing link i, in
// the units of the stored species (scaled deviations d = f / w); scale: the
// link's share (1/b, or 1 under the random matrix, whose slots are per link).
template <int ST, int NS>
__device__ __forceinline__ float2 emission_of(const StepArgs &a, int i, float AR, float AP, float scale) {
  const float ib = __fmul_rn(scale, inv_wq(i) * Pop<ST, NS>::kSp);
  float2 v;
  v.x = __fmul_rn(__fmul_rn(a.em_R, AR), ib);
  v.y = 0.0f;
  if (NS > 2) v.y = __fmul_rn(fmaf(a.em_PR, AR, __fmul_rn(a.em_P, AP)), ib);
  return v;
}

// Species (R, P) re-emitted by the catalytic node `node` along its outgoing
// link i (the incoming population of direction i of the fluid cell behind
// it), from the hits of the previous step.
template <int ST, int NS, bool DET>
__device__ __forceinline__ float2 emission(bool rs, const StepArgs &a, int i, int32_t node, int32_t node_cell) {
  const int64_t e = emit_index(rs, a, i, node, node_cell);
  const float AR = acc_get<DET>(a.A_prev, LBM_OFF(a, kChkAcc, 0, e, LBM_NACC(a)));
  const float AP = NS > 2 ? acc_get<DET>(a.A_prev, LBM_OFF(a, kChkAcc, 0, a.acc_row + e, LBM_NACC(a))) : 0.0f;
  return emission_of<ST, NS>(a, i, AR, AP, emit_scale(rs, a, node));
}

// Populations of lattice entry L at the current time, as a two-lattice scheme
// would hold them (natural order), in the stored form (scaled deviations d,
// species in the stored units; w d is the deviation g = f - w rho_ref), for a state of parity ODD (ODD = 1: the last
// completed step was an even one). For the observables and exports. C, S: load
// the carrier's, the species' (a reader of one of them moves 1/3 or 2/3 of
// the bytes); what is not loaded is 0.
//
// Every address is formed without a branch and all loads are issued together;
// a cell next to a catalytic solid then replaces the species that the wall
// re-emits.
template <int ST, int LAYOUT, int NS, int ODD, bool DET, bool C = true, bool S = true>
__device__ __forceinline__ void load_cell(const StepArgs &a, int32_t L, int32_t cell, uint32_t nbm,
                                          float (&d)[NS][kQ]) {
  using P = Pop<ST, NS>;
  const typename P::C *Cb = static_cast<const typename P::C *>(a.f);
  const typename P::S *Sb = static_cast<const typename P::S *>(a.fs);
  Nbr nb;
  if (ODD || (S && NS > 1 && nbm)) {
    const int z = (int)fast_div((uint32_t)cell, a.div_plane_m, a.div_sh & 0xffu, (a.div_sh >> 8) & 0xffu);
    const int32_t xy = cell - z * a.nx * a.ny;
    const int y = (int)fast_div((uint32_t)xy, a.div_nx_m, (a.div_sh >> 16) & 0xffu, a.div_sh >> 24);
    nb = Nbr(cell, xy - y * a.nx, y, z, a.nx, a.ny, a.nz, a.periodic_z);
  }
  // the entry whose slot holds the population of direction i: odd states, the
  // upwind one, unless it is solid; then, as on even states, the cell's own
  // (with a solid upwind the cell's own reversed post-collision population
  // sits in slot i in both parities)
  int32_t from[kQ];
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    from[i] = L;
    if (ODD && i != 0) {
      const int32_t src = nb.at(-cx(i), -cy(i), -cz(i));  // (a stepped cell's neighbours lie in the box)
      const int32_t e = LAYOUT == LBM_LAYOUT_DENSE ? src : __ldg(a.idx + LBM_OFF(a, kChkIdx, 0, src, LBM_NCELLS(a)));
      from[i] = ((nbm >> opp(i)) & 1u) ? L : e;
    }
  }
  typename P::S sraw[kQ];
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const int slot = (ODD && i != 0 && !((nbm >> opp(i)) & 1u)) ? opp(i) : i;
    const int64_t at = ent_off(from[i]) + 32 * slot;
    d[0][i] = C ? P::c_val(ld_pop(Cb + LBM_OFF(a, kChkPop, 0, at, LBM_NPOP(a)))) : 0.0f;
    if (NS > 1 && S) sraw[i] = ld_pop(Sb + LBM_OFF(a, kChkPop, 0, at, LBM_NPOP(a)));
  }
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    if (NS < 2) continue;
    float2 s = make_float2(0.0f, 0.0f);
    if (S) {
      s = P::s_val(sraw[i]);
      if (i != 0 && ((nbm >> opp(i)) & 1u)) {
        const int32_t node_cell = nb.at(-cx(i), -cy(i), -cz(i));
        const int32_t node = __ldg(a.idx + LBM_OFF(a, kChkIdx, 0, node_cell, LBM_NCELLS(a)));
        // inert solid or species bounce-back: every array's own reversed
        // population, as the carrier's
        if (!(node < 0 || a.sp_bb)) s = emission<ST, NS, DET>(a.rs != 0, a, i, node, node_cell);
      }
    }
    d[1][i] = s.x;
    if (NS > 2) d[2][i] = s.y;
  }
}
// Density deviation and momentum of array k (0 carrier, 1 R, 2 P) of such a
// cell: each population w d rounded, then added.
template <int ST, int NS>
__device__ __forceinline__ float cell_density(const float (&d)[NS][kQ], int k) {
  float r = 0.f;
#pragma unroll
  for (int i = 0; i < kQ; ++i) r = __fadd_rn(r, __fmul_rn(wq(i) * (k ? Pop<ST, NS>::kSpInv : 1.0f), d[k][i]));
  return r;
}
// dir: 0 x, 1 y, 2 z
template <int ST, int NS>
__device__ __forceinline__ float cell_momentum(const float (&d)[NS][kQ], int k, int dir) {
  float j = 0.f;
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    // (directions with c = 0 stay in the sum: an infinity among them makes the
    // velocity a NaN, by which the observables know a diverged state)
    const int c = dir == 0 ? cx(i) : (dir == 1 ? cy(i) : cz(i));
    j = __fadd_rn(j, __fmul_rn(c * wq(i) * (k ? Pop<ST, NS>::kSpInv : 1.0f), d[k][i]));
  }
  return j;
}

// The same, as deviations g (species unscaled), slot by slot, for the plane
// sums. The compiler contracts some of these products with the sums that
// follow, block of branches by block, and a plane's 10^5 cells round alike: an
// order of its own here moves the FP64 sums by up to 1e-8 against those of
// earlier runs. So the loads stay in this order; the branch-free form above
// would take 1,485 us instead of 2,318 (FP16, odd, 256x256x512).
template <int ST, int LAYOUT, int NS, int ODD, bool DET>
__device__ __forceinline__ void load_cell_by_slot(const StepArgs &a, int32_t L, const Nbr &nb, uint32_t nbm,
                                                  float (&f)[NS][kQ]) {
  using P = Pop<ST, NS>;
  const typename P::C *Cb = static_cast<const typename P::C *>(a.f);
  const typename P::S *Sb = static_cast<const typename P::S *>(a.fs);
  const int64_t own = ent_off(L);
  // the entries of all upwind cells, looked up together ahead of the branches
  int32_t up[kQ];
#pragma unroll
  for (int i = 1; i < kQ; ++i) {
    up[i] = nb.at(-cx(i), -cy(i), -cz(i));
    if (ODD && LAYOUT != LBM_LAYOUT_DENSE) up[i] = __ldg(a.idx + LBM_OFF(a, kChkIdx, 0, up[i], LBM_NCELLS(a)));
  }
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const bool solid_up = (i != 0) && ((nbm >> opp(i)) & 1u);
    int64_t base = own;
    int slot = i;
    if (ODD && i != 0 && !solid_up) {
      base = ent_off(up[i]);
      slot = opp(i);
    }
    // carrier: with a solid upwind, the cell's own reversed post-collision
    // population sits in slot i in both parities
    f[0][i] = wq(i) * P::c_val(ld_pop(Cb + LBM_OFF(a, kChkPop, 0, base + 32 * slot, LBM_NPOP(a))));
    if (NS > 1) {
      float2 s = P::s_val(ld_pop(Sb + LBM_OFF(a, kChkPop, 0, base + 32 * slot, LBM_NPOP(a))));
      if (solid_up) {
        const int32_t node_cell = nb.at(-cx(i), -cy(i), -cz(i));
        const int32_t node = __ldg(a.idx + LBM_OFF(a, kChkIdx, 0, node_cell, LBM_NCELLS(a)));
        // inert solid or species bounce-back: every array's own reversed
        // population, as the carrier's
        if (!(node < 0 || a.sp_bb)) s = emission<ST, NS, DET>(a.rs != 0, a, i, node, node_cell);
      }
      f[1][i] = wq(i) * P::kSpInv * s.x;
      if (NS > 2) f[2][i] = wq(i) * P::kSpInv * s.y;
    }
  }
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// 36 w_i: the lattice weights as exact integer multiples of 1/36
__host__ __device__ constexpr float w36(int i) { return i == 0 ? 12.0f : (i <= 6 ? 2.0f : 1.0f); }
// x / 36 without bias: x h + x l with h = 1/36 rounded to float and
// l = 1/36 - h rounded to float (1/36 to about 48 bits)
__device__ __forceinline__ float div36(float x) {
  constexpr float h = 1.0f / 36.0f;
  constexpr float l = (float)(1.0 / 36.0 - (double)(1.0f / 36.0f));
  return fmaf(x, l, __fmul_rn(x, h));
}
__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// This thread's shared-memory slot for the odd step's offset along c_k
// (k = 1 .. REL): the warp's [REL][32] slice of a block-wide array (volatile,
// so that the store reads it back instead of keeping a register copy). The
// offsets beyond REL stay in registers.
//
// kRelNear of them are the fastest on most boxes. us of the odd step's cells with
// 16 and 12: 191x173x300 BF16 387 and 334, 128x128x256 FP16 171 and 166,
// 256x256x512 FP16 1,377 and 1,357; 10 and 14 are slower than 12 (341 and 344 on
// the first). Eight blocks take 57 KB of the SM with 12 and 72 KB with 16, and
// the driver sets 135 KB aside for either, so the room left for L1 is not what
// tells them apart. Asking for a carve-out of 64 KB by launch attribute takes
// another 0.3 to 0.6 % off these steps, but 5 to 20 % on small boxes (37x29x50
// BF16 2,590 and 3,080 to 3,450 us for 101 steps): not done.
//
// Where the planes are large that turns round: the rows between the first and
// the last warp in flight, with the planes above and below them, outgrow L2.
// us a step of 16-bit boxes, three planes' populations in MB, kRelNear and
// kRelWide: 26 MB (320x320) 1,432 and 1,454; between 33 (512x256) and 51
// (448x448) the two are within 0.2 %; 74 (512x512) 640.7 and 630.0 (FP16, 60
// planes), 2,003 and 1,962 (BF16, 200 planes); 116 (640x640) 1,633 and 1,591;
// 181 (800x800) 1,078 and 1,058; 66 (512x512x1024) 9,215 and 9,098 in a call of
// 50 steps with six fields. (The last five differ by 1.3 to 2.6 %, and the
// three runs of either form, taken in turn, by 0.1 %.)
// FP32 keeps to kRelNear (512x512x300: 4,420 and 4,442), as do batches.
constexpr int kRelNear = 12, kRelWide = 16;
constexpr int64_t kWidePlanes = (int64_t)48 << 20;  // bytes, where the two meet
template <int REL>
__device__ __forceinline__ volatile int32_t &rel_slot(int k) {
  __shared__ int32_t s_rel[kWarpsPerBlock * REL * 32];
  return *((volatile int32_t *)s_rel + (threadIdx.x >> 5) * (REL * 32) + (k - 1) * 32 + (threadIdx.x & 31));
}

// Update of one cell: load the 19 slots of both arrays, moments, relaxation
// (or the inlet/outlet equilibrium), store to the same slots. FAST: the
// whole warp lies away from the inlet/outlet and halo planes. Without WALL
// it has no solid neighbour either; with WALL (nbm given) the odd step's
// pointers of its solid links fall back to the cell's own reversed slot.
template <int ST, int LAYOUT, int NS, int ODD, bool FAST, int PHYS, bool WALL = false, int REL = 0,
          bool UNI = false>
__device__ __forceinline__ void cell_update(const StepArgs &a, int32_t L, int32_t cell, uint32_t nbm, int64_t t,
                                            float (&flux)[6]) {
  using P = Pop<ST, NS>;
  using CT = typename P::C;
  using STy = typename P::S;
  const int32_t plane = a.nx * a.ny;
  // cell coordinates and neighbours: not needed on even fast steps (two
  // integer divisions saved)
  int z = 0, y = 0, x = 0;
  int32_t xy = 0;
  Nbr nb;
  if (!FAST || ODD) {
    z = (int)fast_div((uint32_t)cell, a.div_plane_m, a.div_sh & 0xffu, (a.div_sh >> 8) & 0xffu);
    xy = cell - z * plane;
    y = (int)fast_div((uint32_t)xy, a.div_nx_m, (a.div_sh >> 16) & 0xffu, a.div_sh >> 24);
    x = xy - y * a.nx;
    nb = Nbr(cell, x, y, z, a.nx, a.ny, a.nz, a.periodic_z);
  }
  (void)x;
  (void)y;
  // open ends (inlet below, outlet above): not periodic and not a halo
  const bool open_lo = !a.periodic_z && !a.halo_lo, open_hi = !a.periodic_z && !a.halo_hi;
  const bool bc = !FAST && ((open_lo && z == 0) || (open_hi && z == a.nz - 1));
  const int fsel = FAST ? -1
                        : ((open_lo && z == 0)             ? 0
                           : (open_lo && z == 1)          ? 1
                           : (open_hi && z == a.nz - 2)   ? 2
                           : (open_hi && z == a.nz - 1)   ? 3
                                                          : -1);
  // slots whose neighbour is solid or outside the box: the odd step's
  // pointer falls back to the cell's own reversed slot
  const uint32_t solid = (FAST && !WALL) ? 0u : nbm;
  const uint32_t redirect = solid | (bc ? (z == 0 ? kDownBits : kUpBits) : 0u);

  CT *const Co = static_cast<CT *>(a.f) + ent_off(L);
  STy *const So = static_cast<STy *>(a.fs) + ent_off(L);
  const int64_t own = ent_off(L);  // (bounds checks)

  // Odd steps: rel[k], the element offset of slot k's pointer from the
  // entry's own slot k: to the neighbour's entry (fluid-only addressing:
  // idx[cell + c_k]; in a region warp (UNI), whose numbering is the cells'
  // own order, L plus the neighbour's cell offset), or, for a solid or
  // outside neighbour, to the cell's own reversed slot. One 32-bit value per
  // slot; the node number of a solid neighbour is read again from idx where
  // a wall link needs it.
  // Odd fast steps park REL of the 18 offsets in shared memory (this warp's
  // [REL][32] slice) until the store, instead of holding them in registers
  // across the arithmetic: with them the kernel needs 80 registers and
  // spills, without them it fits 64.
  constexpr bool SREL = ODD && FAST && REL > 0;
  int32_t rel[kQ];
  const uint32_t own32 = ent_off32(L);
#pragma unroll
  for (int k = 0; k < kQ; ++k) {
    rel[k] = 0;
    if (ODD && k != 0) {
      if ((!FAST || WALL) && ((redirect >> k) & 1u)) {
        rel[k] = 32 * (opp(k) - k);
      } else {
        const int32_t c2 = nb.at(cx(k), cy(k), cz(k));
        int32_t e;
        if constexpr (LAYOUT == LBM_LAYOUT_DENSE) e = c2;
        else if constexpr (UNI) e = L + (c2 - cell);
        else e = __ldg(a.idx + LBM_OFF(a, kChkIdx, 0, c2, LBM_NCELLS(a)));
        rel[k] = (int32_t)(ent_off32(e) - own32);
      }
      if constexpr (SREL) { if (k <= REL) rel_slot<REL>(k) = rel[k]; }
    }
  }
  chain_wait();
  // ---- load ----
  // The 16-bit formats keep the species as loaded (one 32-bit register per
  // slot) and convert them where they are used, which holds 19 registers
  // fewer than the converted pairs; likewise the carrier, the values of
  // opposite directions two to a register (9 fewer; the even step's spills go
  // from 104 to 8 bytes: 0.3 % of the 512x512x1024 step, 1 % of 191x173x300).
  constexpr bool RAW = ST != LBM_FP32;
  float cv[kQ];
  uint32_t craw[kQ], cpair[(kQ + 1) / 2];
  float2 sv[kQ];
  STy sraw[kQ];
  if (!bc) {
#pragma unroll
    for (int k = 0; k < kQ; ++k) {
      const int i = ODD ? opp(k) : k;  // the incoming direction this slot holds
      const CT qc = ld_pop(Co + LBM_OFF(a, kChkPop, own, rel[k] + 32 * k, LBM_NPOP(a)));
      if (RAW) craw[i] = (uint32_t)qc;
      else cv[i] = P::c_val(qc);
      if (NS > 1) {
        sraw[i] = ld_pop(So + LBM_OFF(a, kChkPop, own, rel[k] + 32 * k, LBM_NPOP(a)));
        if (!RAW) sv[i] = P::s_val(sraw[i]);
      } else {
        sraw[i] = STy{};
        sv[i] = f2(0.0f);
      }
    }
    // (species arriving from a catalytic node: node_kernel has written
    // the sputtering law's value into the slot, the cell's own slot i)
  } else {
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      cv[i] = 0.0f;
      craw[i] = 0u;
      sv[i] = f2(0.0f);
      sraw[i] = STy{};
    }
  }
  if constexpr (RAW) {
#pragma unroll
    for (int q = 0; q < 9; ++q) cpair[q] = __byte_perm(craw[2 * q + 1], craw[2 * q + 2], 0x5410);
    cpair[9] = craw[0];
  }
  // carrier value of incoming direction i (`again`: as below)
  auto cvc = [&](int i, bool again) -> float {
    if constexpr (!RAW) {
      return cv[i];
    } else {
      uint32_t r = cpair[i == 0 ? 9 : (i - 1) / 2];
      if (again) asm volatile("" : "+r"(r));
      return P::c_half(r, i != 0 && (i & 1) == 0);
    }
  };
  // species pair of incoming direction i; `again`: convert afresh (the empty
  // asm keeps the compiler from holding the first conversion instead)
  auto spc = [&](int i, bool again) -> float2 {
    if constexpr (!RAW || NS < 2) {
      return sv[i];
    } else {
      STy r = sraw[i];
      if (again) {
        if constexpr (sizeof(STy) == 2) asm volatile("" : "+h"(r));
        else asm volatile("" : "+r"(r));
      }
      return P::s_val(r);
    }
  };

  // ---- moments ----
  constexpr bool BARY = PHYS == kPhysBary;
  float drho, ux, uy, uz;
  float2 rs;  // species densities (stored units)
  if (!bc) {
    // Moments. 16-bit storage: sums with the exact integer weights
    // 36 w_i = 12, 2, 1 and one division by 36 at the end, formed as
    // x h + x l with h + l = 1/36 to twice float precision so that its
    // rounding has no bias (float weights 1/3, 1/18, 1/36 sum to 1 + 1.4e-8
    // and would scale every collision's mass by that factor). FP32 storage:
    // see below.
    float j36x = 0.f, j36y = 0.f, j36z = 0.f, d36, inv36;
    float2 rs36, js[3] = {f2(0.f), f2(0.f), f2(0.f)};
    if constexpr (ST == LBM_FP32) {
      // FP32 storage: weighted sums population by population, w d rounded
      // once and added, as j = sum w c d and rho = sum w d (the float
      // weights carry a common relative excess of ~1e-8, which here scales
      // j and rho alike). Kept because it is the form whose fixed points lie
      // closest to the FP64 solution in long steady flows, where every
      // rounding repeats identically at every step.
      d36 = 0.f;
      rs36 = f2(0.f);
#pragma unroll
      for (int i = 0; i < kQ; ++i) {
        const float wd = __fmul_rn(wq(i), cv[i]);
        d36 = __fadd_rn(d36, wd);
        if (cx(i)) j36x = __fadd_rn(j36x, cx(i) * wd);
        if (cy(i)) j36y = __fadd_rn(j36y, cy(i) * wd);
        if (cz(i)) j36z = __fadd_rn(j36z, cz(i) * wd);
        if (NS > 1) {
          rs36 = fma2(f2(wq(i)), sv[i], rs36);
          if (BARY) {
            if (cx(i)) js[0] = fma2(f2(cx(i) * wq(i)), sv[i], js[0]);
            if (cy(i)) js[1] = fma2(f2(cy(i) * wq(i)), sv[i], js[1]);
            if (cz(i)) js[2] = fma2(f2(cz(i) * wq(i)), sv[i], js[2]);
          }
        }
      }
    } else {
      // 16-bit storage: sums and differences of opposite slots
      float sa = 0.f, sd = 0.f;
      float2 rsa = f2(0.f), rsd = f2(0.f);
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const int i = 2 * q + 1;
        const float s = __fadd_rn(cvc(i, false), cvc(i + 1, false)), dd = __fsub_rn(cvc(i, false), cvc(i + 1, false));
        if (i <= 6) sa = __fadd_rn(sa, s); else sd = __fadd_rn(sd, s);
        const float w = w36(i);
        if (cx(i)) j36x = fmaf((float)cx(i) * w, dd, j36x);
        if (cy(i)) j36y = fmaf((float)cy(i) * w, dd, j36y);
        if (cz(i)) j36z = fmaf((float)cz(i) * w, dd, j36z);
        if (NS > 1) {
          const float2 s2 = add2(spc(i, false), spc(i + 1, false));
          if (i <= 6) rsa = add2(rsa, s2); else rsd = add2(rsd, s2);
          if (BARY) {
            const float2 d2 = fma2(f2(-1.0f), spc(i + 1, false), spc(i, false));
            if (cx(i)) js[0] = fma2(f2(cx(i) * w), d2, js[0]);
            if (cy(i)) js[1] = fma2(f2(cy(i) * w), d2, js[1]);
            if (cz(i)) js[2] = fma2(f2(cz(i) * w), d2, js[2]);
          }
        }
      }
      d36 = fmaf(12.0f, cvc(0, false), fmaf(2.0f, sa, sd));
      rs36 = fma2(f2(12.0f), spc(0, false), fma2(f2(2.0f), rsa, rsd));
    }
    if constexpr (ST == LBM_FP32) {
      drho = d36;  // (FP32: the sums above are already weighted)
      rs = rs36;
    } else {
      drho = div36(d36);
      rs = make_float2(div36(rs36.x), div36(rs36.y));
    }
    // (FP32 sums are already divided by 36: the velocity divides by rho,
    // the 16-bit ones by 36 rho)
    constexpr float kR = (ST == LBM_FP32) ? 1.0f : 36.0f;
    if (BARY) {
      // u = (j_C + j_R + j_P) / (rho_C + rho_R + rho_P)
      const float msp = __fmul_rn(__fadd_rn(rs.x, rs.y), P::kSpInv);
      inv36 = 1.0f / __fmul_rn(kR, __fadd_rn(__fadd_rn(1.0f, drho), msp));
      j36x = fmaf(__fadd_rn(js[0].x, js[0].y), P::kSpInv, j36x);
      j36y = fmaf(__fadd_rn(js[1].x, js[1].y), P::kSpInv, j36y);
      j36z = fmaf(__fadd_rn(js[2].x, js[2].y), P::kSpInv, j36z);
    } else {
      inv36 = (ST == LBM_FP32) ? 1.0f / __fadd_rn(1.0f, drho) : 1.0f / fmaf(36.0f, drho, 36.0f);
    }
    const float inv_rho = inv36, jx = j36x, jy = j36y, jz = j36z;
    ux = __fmul_rn(jx, inv_rho);
    uy = __fmul_rn(jy, inv_rho);
    uz = __fmul_rn(jz, inv_rho);
    if (PHYS == kPhysChannel) uz = fmaf(0.5f, a.g_z, uz);  // body force: the velocity half a step on
    if (!FAST && ((open_lo && z == 1) || (open_hi && z == a.nz - 2))) {
      // plane cache: u_x, u_y, u_z, rho_R, rho_P at ub[0], ub[plane], ... (the check bounds the last)
      float *ub = a.ub_cur + LBM_OFF(a, kChkUb, 0, (int64_t)(z == 1 ? 0 : 5) * plane + xy,
                                     LBM_NUB(a) - 4 * (int64_t)plane);
      ub[0] = ux;
      ub[plane] = uy;
      ub[2 * (int64_t)plane] = uz;
      if (NS > 1) ub[3 * (int64_t)plane] = rs.x * P::kSpInv;
      if (NS > 2) ub[4 * (int64_t)plane] = rs.y * P::kSpInv;
    }
  } else {
    const float *ub = a.ub_prev + LBM_OFF(a, kChkUb, 0, (int64_t)(z == 0 ? 0 : 5) * plane + xy,
                                          LBM_NUB(a) - 4 * (int64_t)plane);
    ux = ub[0];
    uy = ub[plane];
    uz = ub[2 * (int64_t)plane];
    if (z == 0 && a.vel_in) {  // velocity inlet: (0, 0, u_in)
      ux = 0.f;
      uy = 0.f;
      uz = a.u_in;
    }
    drho = (z == 0) ? a.drho_in : a.drho_out;
    rs = (z == 0) ? make_float2(a.c_in * P::kSp, 0.0f)
                  : make_float2(ub[3 * (int64_t)plane] * P::kSp, NS > 2 ? ub[4 * (int64_t)plane] * P::kSp : 0.0f);
  }

  // ---- relaxation (or equilibrium on the inlet/outlet planes) and store ----
  // (every multiply-add below is written out, as an FMA or as a rounded
  // multiply and add, so that each kernel that inlines this function - the
  // fast, general and batched ones - computes bit-identical results)
  const float rho = __fadd_rn(1.0f, drho);
  const float om = bc ? 1.0f : a.omega;
  const float om_s = bc ? 1.0f : (PHYS == kPhysCarrier ? a.omega : a.omega_s);
  const float wr = __fmul_rn(om, rho), wd = __fmul_rn(om, drho), omc = __fsub_rn(1.0f, om);
  const float2 wrs = __fmul2_rn(f2(om_s), rs), omc_s = f2(__fsub_rn(1.0f, om_s));
  const float Ux = __fmul_rn(3.0f, ux), Uy = __fmul_rn(3.0f, uy), Uz = __fmul_rn(3.0f, uz);
  const float u2 = __fmul_rn(1.5f, fmaf(uz, uz, fmaf(uy, uy, __fmul_rn(ux, ux))));
  const float fz = (PHYS == kPhysChannel && !bc) ? __fmul_rn(__fmul_rn(fmaf(-0.5f, a.omega, 1.0f), rho), a.g_z) : 0.0f;
  const uint32_t h = (ST == LBM_FP32) ? 0u : mix32(((uint32_t)L + a.hash_base) ^ step_seed_of(t, a.seed_mix));
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    // P_i from the pair (i, opp(i)): q = 4.5 (c.u)^2 - 1.5 u^2 shared, +-3 c.u
    const int ip = (i == 0) ? 0 : ((i & 1) ? i : i - 1);
    float cu, Pi;
    if constexpr (ST == LBM_FP32) {
      // per direction: 3 c.u from the velocity components, then
      // (3 c.u + 4.5 (c.u)^2) - 1.5 u^2
      const float cd = __fmul_rn(3.0f, __fadd_rn(__fadd_rn(cx(ip) * ux, cy(ip) * uy), cz(ip) * uz));
      const float ci = (i & 1) || i == 0 ? cd : -cd;
      cu = cd;
      Pi = __fsub_rn(fmaf(__fmul_rn(0.5f, ci), ci, ci), u2);
    } else {
      cu = __fadd_rn(__fadd_rn(cx(ip) * Ux, cy(ip) * Uy), cz(ip) * Uz);
      const float qq = fmaf(__fmul_rn(0.5f, cu), cu, -u2);
      Pi = (i == 0) ? -u2 : ((i & 1) ? __fadd_rn(qq, cu) : __fsub_rn(qq, cu));
    }
    // FP32 storage keeps d + omega (deq - d), whose rounding shrinks with
    // the distance from equilibrium; the 16-bit formats, whose storage
    // rounding is far coarser, take (1 - omega) d + omega deq (two FMAs)
    float c_out;
    if constexpr (ST == LBM_FP32) c_out = fmaf(om, __fsub_rn(fmaf(rho, Pi, drho), cv[i]), cv[i]);
    else c_out = fmaf(wr, Pi, fmaf(omc, cvc(i, true), wd));
    if (PHYS == kPhysChannel && !bc && a.g_z != 0.f) {
      // body force F = rho g along z, Guo, Zheng and Shi (2002): in scaled
      // deviations the source adds (1 - omega/2) [3 (c_iz - u_z) + 9 (c_i . u) c_iz] F_z
      const float cui = (i & 1) || i == 0 ? cu : -cu;
      c_out = fmaf(fz, fmaf(cui, 3.0f * cz(i), __fmul_rn(3.0f, __fsub_rn((float)cz(i), uz))), c_out);
    }
    float2 s_out;
    if constexpr (ST == LBM_FP32) s_out = fma2(f2(om_s), fma2(f2(-1.0f), sv[i], fma2(f2(Pi), rs, rs)), sv[i]);
    else s_out = fma2(omc_s, spc(i, true), fma2(f2(Pi), wrs, wrs));
    const int k = ODD ? i : opp(i);  // the slot that receives f*_i
    // (odd steps: the offset passes through an empty asm so that the store
    // address is formed again from the 32-bit offset, instead of the 64-bit
    // load addresses of all 19 slots being held across the arithmetic)
    int32_t rk = rel[k];
    if constexpr (SREL) {
      if (k != 0 && k <= REL) rk = rel_slot<REL>(k);
      else if (k != 0) asm volatile("" : "+r"(rk));
    } else if (ODD) {
      asm volatile("" : "+r"(rk));
    }
    const CT qc = P::c_cv(c_out, h * sr_mul(0, i));
    __stcs(Co + LBM_OFF(a, kChkPop, own, rk + 32 * k, LBM_NPOP(a)), qc);
    STy qs{};
    if (NS > 1) {
      qs = P::s_cv(s_out, h * sr_mul(1, i));
      __stcs(So + LBM_OFF(a, kChkPop, own, rk + 32 * k, LBM_NPOP(a)), qs);
    }
    if (!FAST && i != 0) {
      // inlet / outlet face flows of the stored (rounded) values
      if (fsel >= 0 && !((redirect >> i) & 1u)) {
        const bool up = cz(i) > 0, dn = cz(i) < 0;
        const float sgn =
            ((fsel == 0 || fsel == 2) && up) ? 1.f : (((fsel == 1 || fsel == 3) && dn) ? -1.f : 0.f);
        if (sgn != 0.f) {
          const int o = fsel <= 1 ? 0 : 3;
          const float sw = sgn * wq(i);
          flux[o] = fmaf(sw, P::c_val(qc), flux[o]);
          if (NS > 1) {
            const float2 sq = P::s_val(qs);
            flux[o + 1] = fmaf(sw * P::kSpInv, sq.x, flux[o + 1]);
            if (NS > 2) flux[o + 2] = fmaf(sw * P::kSpInv, sq.y, flux[o + 2]);
          }
        }
      }
      // (species sent towards a catalytic node stay in the redirected slot,
      // where node_kernel sums them)
    }
  }
}

// Face-flow slot of lattice warp W (the warps overlapping planes 0, 1 and
// nz-2, nz-1), or -1.
__device__ __forceinline__ int32_t flux_slot(const StepArgs &a, int32_t W) {
  if (a.periodic_z) return -1;
  if (W < a.n_lo_warps) return W;
  if (W >= a.hi_warp && W < a.n_lat_warps) return a.n_lo_warps + (W - a.hi_warp);
  return -1;
}

// Adds the warp's face flows, summed in FP64 in a fixed order, to its slot.
// Every lane of the warp must call it. The six sums are formed together: each
// exchange halves the values a lane still carries (3, 2, 1, 1, 1 FP64 adds
// instead of 6 x 5, on a chip whose FP64 pipe is slow), and the six lanes that
// end with a sum add theirs to the slot at once.
__device__ __forceinline__ void bank_flux(const StepArgs &a, int32_t W, const float (&flux)[6]) {
  const int32_t slot = flux_slot(a, W);
  if (slot < 0) return;
  const int lane = threadIdx.x & 31;
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  double v[3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    v[k] = (double)(b4 ? flux[k + 3] : flux[k]) + __shfl_xor_sync(0xffffffffu, (double)(b4 ? flux[k] : flux[k + 3]), 16);
  const double u0 = (b3 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, b3 ? v[0] : v[2], 8);
  const double u1 = v[1] + __shfl_xor_sync(0xffffffffu, v[1], 8);  // (of use where bit 3 is clear)
  double w = (b2 && !b3 ? u1 : u0) + __shfl_xor_sync(0xffffffffu, b2 || b3 ? u0 : u1, 4);
  w += __shfl_xor_sync(0xffffffffu, w, 2);
  w += __shfl_xor_sync(0xffffffffu, w, 1);
  // lanes 0, 4, 8 hold sums 0, 1, 2 and lanes 16, 20, 24 sums 3, 4, 5
  if ((lane & 3) == 0 && (lane & 12) != 12)
    a.flux_cum[6 * (int64_t)slot + (b4 ? 3 : 0) + ((lane >> 2) & 3)] += w;
}

// ---- Catalytic nodes: the sputtering law (Appendix, Eq. f_P_in) ----
//
// A wall link of node n along c_j joins it to the fluid cell x = n + c_j. In
// both parities of the in-place streaming, x stores the population it sends
// towards n in its own slot j (the halfway bounce-back of the carrier), and
// it reads from that same slot the population that arrives from n along c_j.
// So the species part of the boundary acts on those slots alone, one thread
// per node, around the cell updates of a step:
//   emission, before them: bank the previous step's hits of the node, and
//     write into each link's slot what the sputtering law returns along the
//     link. Both only write what the hits say, the banked sum from one copy of
//     the cumulative hits to the other, so an emission that is made again (by
//     the call after one whose launches failed part-way) changes nothing;
//   hits, after them: the species that reached the node in this step,
//     w_j times each link's stored value, summed over the node's links in a
//     fixed order (or in 64-bit fixed point), into the step's accumulator
//     (under the random matrix, each into the slot of the link it leaves by).
// Between two steps of one call both fall to the same thread with nothing in
// between, so one launch takes the hits of step t and the emission of step
// t + 1 (kNodeBoth); the first step of a call emits alone and the last one
// takes its hits alone, so that what a call leaves behind is always the hits.
// The carrier's slot keeps its bounce-back. Inert solid is never a node, and
// under species bounce-back (sp_bb) neither kernel runs, so the species
// bounce back too.

// Lattice entries of the fluid cells across the links of the node in cell
// nc (active links in `links`), or -1 where there is no link or the cell is
// in a halo plane (stepped by the neighbouring sub-domain). Every active link
// ends inside the box. All 18 index loads are issued together.
template <int LAYOUT>
__device__ __forceinline__ void link_entries(const StepArgs &a, int32_t nc, uint32_t links, int32_t (&Ls)[kQ]) {
  const int32_t plane = a.nx * a.ny;
  const int z = nc / plane;
  const int32_t xy = nc - z * plane;
  const int y = xy / a.nx;
  const Nbr nb(nc, xy - y * a.nx, y, z, a.nx, a.ny, a.nz, a.periodic_z);
  Ls[0] = -1;
#pragma unroll
  for (int j = 1; j < kQ; ++j) {
    Ls[j] = -1;
    if (((links >> j) & 1u) && !halo_plane(a, z + cz(j))) {
      const int32_t c = nb.at(cx(j), cy(j), cz(j));
      Ls[j] = LAYOUT == LBM_LAYOUT_DENSE ? c : __ldg(a.idx + LBM_OFF(a, kChkIdx, 0, c, LBM_NCELLS(a)));
    }
  }
}

// Node n around step t: MODE kNodeEmit, the emission of step t from the
// previous step's hits; kNodeHits, the hits of step t into a.A_cur; kNodeBoth,
// the hits of step t and then the emission of step t + 1 from them. hv: the
// hits emitted from (R, P), to be banked. (t is passed apart from a.t: a
// batched launch reuses argument sets six steps apart.)
//
// Bound by latency and by the 32-byte sectors around each link's 4-8 byte
// slot. All of a node's links are issued together (one at a time took three
// times as long on the 512x512x1024 sample); in kNodeBoth the links' entries
// are found once and the slots are written while their lines are still in L2.
// Node kernels per step, two launches before and one now: 531 -> 391 us
// (512x512x1024, FP16, 7.6 M nodes), 80 -> 52 us (191x173x300, BF16, 0.93 M).
constexpr int kNodeEmit = 1, kNodeHits = 2, kNodeBoth = 3;
// Blocks per SM of the node kernels. kNodeBoth holds 18 entries and 18 loaded
// slots: left to itself it takes 80-96 registers (2-3 blocks) and is slower
// than the two launches it replaces (405 us a step on the 191x173x300 case).
// Measured there at 4, 5 and 6 blocks: 379, 376 and 378 us; on the 512x512x1024
// sample 9,082, 9,058 and 9,065; FP32 on 256x256x512 2,048, 2,054 and 2,051
// (at 5 its fixed-point form spills 140 bytes, at 4 none).
constexpr int node_min_blocks(int st, int mode) { return mode != kNodeBoth ? 1 : (st == LBM_FP32 ? 4 : 5); }
template <int ST, int LAYOUT, int NS, bool DET, bool RS, int MODE>
__device__ __forceinline__ void node_work(const StepArgs &a, int64_t n, int64_t t, float (&hv)[2]) {
  using P = Pop<ST, NS>;
  using STy = typename P::S;
  hv[0] = hv[1] = 0.f;
  const int32_t nc = __ldg(a.node_cell + LBM_OFF(a, kChkNode, 0, n, a.n_nodes));
  const uint32_t links = __ldg(a.cell_bits + LBM_OFF(a, kChkIdx, 0, nc, LBM_NCELLS(a)));
  int32_t Ls[kQ];
  link_entries<LAYOUT>(a, nc, links, Ls);
  STy *const S = static_cast<STy *>(a.fs);
  int32_t o = 0, m = 0;  // random matrix: the node's link slots
  if (RS) {
    o = __ldg(a.node_off + LBM_OFF(a, kChkNode, 0, n, a.n_nodes + 1));
    m = __ldg(a.node_off + LBM_OFF(a, kChkNode, 0, n + 1, a.n_nodes + 1)) - o;
  }
  chain_wait();
  // the hits that the emission works from: a.A_prev, or this thread's own
  const void *const A = (MODE & kNodeHits) ? a.A_cur : a.A_prev;
  if (MODE & kNodeHits) {
    STy raw[kQ];
#pragma unroll
    for (int j = 1; j < kQ; ++j)
      raw[j] = Ls[j] >= 0 ? S[LBM_OFF(a, kChkPop, 0, ent_off(Ls[j]) + 32 * j, LBM_NPOP(a))] : STy{};
    if (RS)
      for (int32_t k = 0; k < m; ++k) {
        acc_clear<DET>(a.A_cur, LBM_OFF(a, kChkAcc, 0, o + k, LBM_NACC(a)));
        if (NS > 2) acc_clear<DET>(a.A_cur, LBM_OFF(a, kChkAcc, 0, a.acc_row + o + k, LBM_NACC(a)));
      }
    acc_t iR = 0ull, iP = 0ull;  // fixed-point sums (DET)
    float fR = 0.f, fP = 0.f;    // FP32 sums, in link order
#pragma unroll
    for (int j = 1; j < kQ; ++j) {
      if (Ls[j] < 0) continue;
      const float2 s = P::s_val(raw[j]);
      // (the population that arrived moves along c_opp(j); w_opp(j) = w_j)
      const float vR = __fmul_rn(wq(j) * P::kSpInv, s.x), vP = __fmul_rn(wq(j) * P::kSpInv, s.y);
      if (RS) {
        const int64_t k = o + rs_rank(a.rs_key, nc, opp(j), t, m);
        acc_put<DET>(a.A_cur, LBM_OFF(a, kChkAcc, 0, k, LBM_NACC(a)), vR);
        if (NS > 2) acc_put<DET>(a.A_cur, LBM_OFF(a, kChkAcc, 0, a.acc_row + k, LBM_NACC(a)), vP);
      } else if (DET) {
        iR += acc_from(vR);
        if (NS > 2) iP += acc_from(vP);
      } else {
        fR = __fadd_rn(fR, vR);
        if (NS > 2) fP = __fadd_rn(fP, vP);
      }
    }
    if (!RS) {
      if (DET) {
        static_cast<acc_t *>(a.A_cur)[LBM_OFF(a, kChkAcc, 0, n, LBM_NACC(a))] = iR;
        if (NS > 2) static_cast<acc_t *>(a.A_cur)[LBM_OFF(a, kChkAcc, 0, a.acc_row + n, LBM_NACC(a))] = iP;
        hv[0] = acc_to_f(iR);
        hv[1] = acc_to_f(iP);
      } else {
        static_cast<float *>(a.A_cur)[LBM_OFF(a, kChkAcc, 0, n, LBM_NACC(a))] = fR;
        if (NS > 2) static_cast<float *>(a.A_cur)[LBM_OFF(a, kChkAcc, 0, a.acc_row + n, LBM_NACC(a))] = fP;
        hv[0] = fR;
        hv[1] = fP;
      }
    }
  }
  if (!(MODE & kNodeEmit)) return;
  if (RS) {
    for (int32_t k = o; k < o + m; ++k) {
      hv[0] += acc_get<DET>(A, LBM_OFF(a, kChkAcc, 0, k, LBM_NACC(a)));
      if (NS > 2) hv[1] += acc_get<DET>(A, LBM_OFF(a, kChkAcc, 0, a.acc_row + k, LBM_NACC(a)));
    }
  } else if (MODE == kNodeEmit) {
    hv[0] = acc_get<DET>(A, LBM_OFF(a, kChkAcc, 0, n, LBM_NACC(a)));
    if (NS > 2) hv[1] = acc_get<DET>(A, LBM_OFF(a, kChkAcc, 0, a.acc_row + n, LBM_NACC(a)));
  }
  const uint32_t sd = step_seed_of(MODE == kNodeBoth ? t + 1 : t, a.seed_mix);
  const float scale = emit_scale(RS, a, (int32_t)n);
#pragma unroll
  for (int j = 1; j < kQ; ++j) {
    if (Ls[j] < 0) continue;
    float AR = hv[0], AP = hv[1];
    if (RS) {  // (the link's rank among the node's active links)
      const int64_t k = o + __popc(links & ((1u << j) - 1u));
      AR = acc_get<DET>(A, LBM_OFF(a, kChkAcc, 0, k, LBM_NACC(a)));
      if (NS > 2) AP = acc_get<DET>(A, LBM_OFF(a, kChkAcc, 0, a.acc_row + k, LBM_NACC(a)));
    }
    const float2 v = emission_of<ST, NS>(a, j, AR, AP, scale);
    // (the slot's address is formed again from the entry, instead of the 18
    // 64-bit addresses being held since the loads)
    if (MODE == kNodeBoth) asm volatile("" : "+r"(Ls[j]));
    const uint32_t h = (ST == LBM_FP32) ? 0u : mix32(((uint32_t)Ls[j] + a.hash_base) ^ sd);
    S[LBM_OFF(a, kChkPop, 0, ent_off(Ls[j]) + 32 * j, LBM_NPOP(a))] = P::s_cv(v, h * sr_mul(2, j));
  }
}

// dst[0] and dst[1]: src's with the block's FP64 sums of a pair of per-thread
// values added, in a fixed order: the first exchange leaves one value to each
// half of the warp, then the 8 warps' pairs are summed by one warp. Must be
// called by every thread of the block.
__device__ __forceinline__ void bank_pair(const float (&v)[2], const double *src, double *dst) {
  __shared__ double sh[2][kBlock / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool hi = lane & 16;
  double s = (double)(hi ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, (double)(hi ? v[0] : v[1]), 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((lane & 15) == 0) sh[lane >> 4][wid] = s;
  __syncthreads();
  if (wid == 0 && lane < 2 * (kBlock / 32)) {
    s = sh[lane / (kBlock / 32)][lane % (kBlock / 32)];
#pragma unroll
    for (int o = kBlock / 64; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffu, s, o);
    if (lane % (kBlock / 32) == 0) dst[lane / (kBlock / 32)] = src[lane / (kBlock / 32)] + s;
  }
}

// Node block blk (nodes blk 256 .. blk 256 + 255) of a node kernel; an
// emission banks the hits it emits from into the block's FP64 slot. Every
// thread of the block must call it.
template <int ST, int LAYOUT, int NS, bool DET, bool RS, int MODE>
__device__ __forceinline__ void node_block(const StepArgs &a, int blk, int64_t t) {
  if ((int64_t)blk * kBlock >= a.n_nodes) return;  // (uniform over the block)
  const int64_t n = (int64_t)blk * kBlock + threadIdx.x;
  float hv[2] = {0.f, 0.f};
  if (n < a.n_nodes) {
    node_work<ST, LAYOUT, NS, DET, RS, MODE>(a, n, t, hv);
    if (n < a.bank_lo || n >= a.bank_hi) hv[0] = hv[1] = 0.f;  // (halo nodes are the neighbour's)
  }
  // (kNodeBoth emits for step t + 1, where the copies have changed places)
  if (MODE & kNodeEmit)
    bank_pair(hv, (MODE == kNodeBoth ? a.cum_next : a.cum_now) + 2 * (int64_t)blk,
              (MODE == kNodeBoth ? a.cum_now : a.cum_next) + 2 * (int64_t)blk);
}

template <int ST, int LAYOUT, int NS, bool DET, bool RS, int MODE>
__global__ void __launch_bounds__(kBlock, node_min_blocks(ST, MODE)) node_kernel(const StepArgs a) {
  chain_next();
  node_block<ST, LAYOUT, NS, DET, RS, MODE>(a, (int)blockIdx.x, a.t);
}

// General warp w of the list (solid neighbours, inlet/outlet planes, halo
// planes).
template <int ST, int LAYOUT, int NS, int ODD, int PHYS>
__device__ __forceinline__ void gen_warp(const StepArgs &a, int w, int64_t t) {
  const int32_t W = __ldg(a.gen_list + w);
  const int32_t L = W * 32 + (threadIdx.x & 31);
  float flux[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // in C,R,P ; out C,R,P
  if (L < a.n_lat) {
    const int32_t cell = (LAYOUT == LBM_LAYOUT_DENSE) ? L : __ldg(a.fcell + L);
    if ((LAYOUT != LBM_LAYOUT_DENSE || !__ldg(a.mask + cell)) && !halo_plane(a, cell / (a.nx * a.ny)))
      cell_update<ST, LAYOUT, NS, ODD, false, PHYS>(a, L, cell, __ldg(a.nbm + L), t, flux);
  }
  chain_wait();  // (a warp of halo entries alone has not waited yet)
  bank_flux(a, W, flux);
}

// Warp w of the fast list.
template <int ST, int LAYOUT, int NS, int ODD, int PHYS, bool UNI, int REL>
__device__ __forceinline__ void fast_warp(const StepArgs &a, int w, int64_t t) {
  if (w >= (UNI ? a.n_uni : a.n_fast + a.n_wall)) return;
  const uint32_t v = (uint32_t)__ldg(a.fast_list + w);
  const int32_t L = (int32_t)(v & kWarpIdMask) * 32 + (threadIdx.x & 31);
  if (L >= a.n_lat) return;
  int32_t cell = L;
  if (LAYOUT == LBM_LAYOUT_DENSE) {
    if (__ldg(a.mask + L)) return;
  } else if (UNI) {
    cell = L + __ldg(a.fast_list + a.n_lat_warps + ((v >> kUniShift) & (uint32_t)kUniRegions));
  } else if (ODD) {
    cell = __ldg(a.fcell + L);
  }
  float flux[6];
  // odd steps: one code path for plain and wall warps, the solid-neighbour
  // mask being zero for a plain warp (two paths in one kernel spill more)
  const uint32_t nbm = (ODD && !UNI && (v & kWallWarp)) ? __ldg(a.nbm + L) : 0u;
  cell_update<ST, LAYOUT, NS, ODD, true, PHYS, ODD != 0 && !UNI, REL, UNI>(a, L, cell, nbm, t, flux);
}

// Cell kernel: one warp per listed lattice warp, the general warps in the
// first blocks and the fast ones after them (block_0: the first block of that
// sequence that this launch takes; list_0: the first fast warp). Fast warps
// need no neighbour mask, no wall-hit accumulators and no face flows; even
// steps touch only the entries' own slots. Even steps take the whole fast list
// in one launch. Odd steps of large boxes take it in two: the region warps at
// its head (UNI: cell = entry + the region's shift, a word of the small table
// after the lists, which stays in L1; no fcell, idx or nbm reads), then the
// rest.
//
// The general warps need 84-116 registers; in a launch of their own they ran at
// 13 warps per SM after the fast warps had drained. In the fast warps' launch
// the kernel spills more: even steps 0-96 bytes, odd ones 104-324, the most in
// FP32 with the channel's terms; the region form, which has no general warps,
// 0-52. (Spilling requests a warp, 191x173x300 BF16: 0.06 on even steps, the
// general warps' alone, and 5.4 on odd ones, two thirds or more of them not the
// general warps'.) It is the faster all the same. Step, in one launch and with
// one of their own: 158.5 and 161 us (128x128x256, FP16), 9,048 and 9,054
// (512x512x1024, FP16); 32x32x64 FP32 13.6 and 17.9 us. Boxes of which half the
// planes are general gained as well, 512x512x8 (C+R+P) from four launches that
// waited for one another to the present ones: 213.9 -> 116.0 us (FP16,
// fluid-only), 202.3 -> 115.1 (FP16, dense), 250.1 -> 175.4 (FP32, fluid-only),
// 243.7 -> 175.5 (FP32, dense).
template <int ST, int LAYOUT, int NS, int ODD, int PHYS, bool UNI = false, int REL = kRelNear>
__global__ void __launch_bounds__(kCellBlock, cell_min_blocks(ST))
    cell_kernel(const __grid_constant__ StepArgs a, int block_0, int list_0) {
  chain_next();
  int b = block_0 + (int)blockIdx.x;
  if (!UNI) {
    const int n_gen_blocks = (a.n_gen + kWarpsPerBlock - 1) / kWarpsPerBlock;
    if (b < n_gen_blocks) {
      const int w = b * kWarpsPerBlock + (int)(threadIdx.x >> 5);
      if (w < a.n_gen) gen_warp<ST, LAYOUT, NS, ODD, PHYS>(a, w, a.t);
      return;
    }
    b -= n_gen_blocks;
  }
  fast_warp<ST, LAYOUT, NS, ODD, PHYS, UNI, REL>(a, list_0 + b * kWarpsPerBlock + (int)(threadIdx.x >> 5), a.t);
}

// One step of the cells of one 256-entry block of lattice entries
// (single-launch batches): each warp takes the fast path when all its live
// entries can. Same arithmetic and face-flow slots as the fast and general
// kernels.
template <int ST, int LAYOUT, int NS, int ODD, int PHYS>
__device__ __forceinline__ void step_block(const StepArgs &a, const int blk, const int64_t t) {
  const int32_t L = (int32_t)(blk * kBlock + threadIdx.x);
  float flux[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // in C,R,P ; out C,R,P
  bool live = L < a.n_lat;
  int32_t cell = 0;
  uint32_t nbm = 0;
  if (live) {
    cell = (LAYOUT == LBM_LAYOUT_DENSE) ? L : __ldg(a.fcell + L);
    if (LAYOUT == LBM_LAYOUT_DENSE && __ldg(a.mask + cell)) live = false;
    nbm = __ldg(a.nbm + L);
  }
  // (halo cells are not stepped, and a warp holding one takes the general
  // path, as the warp lists have it)
  const bool halo = live && halo_plane(a, cell / (a.nx * a.ny));
  const bool plain = !live || (!halo && fast_entry(a, cell, nbm));
  const bool onplane = !live || (!halo && fast_plane(a, cell));
  live = live && !halo;
  if (__all_sync(0xffffffffu, plain) || (!ODD && __all_sync(0xffffffffu, onplane))) {
    if (live) cell_update<ST, LAYOUT, NS, ODD, true, PHYS>(a, L, cell, 0u, t, flux);
  } else if (__all_sync(0xffffffffu, onplane)) {  // a wall warp, odd step
    if (live) cell_update<ST, LAYOUT, NS, ODD, true, PHYS, true>(a, L, cell, nbm, t, flux);
  } else if (live) {
    cell_update<ST, LAYOUT, NS, ODD, false, PHYS>(a, L, cell, nbm, t, flux);
  }
  bank_flux(a, (int32_t)(L >> 5), flux);
}

// Batched launch advancing many simulations by several steps (continuous
// batching). Work block w of a step belongs to the simulation k with
// block_start[k] <= w < block_start[k + 1], whose arguments (constant bank)
// and own parity pick the path.
__device__ __forceinline__ int batch_sim_of(const BatchLaunch &p, int w) {
  int lo = 0, hi = p.n_sims - 1;  // last simulation with block_start <= w
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (p.block_start[mid] <= w)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// One launch covers p.n_steps steps in 3 n_steps phases of total_blocks
// CTAs, one work block each: for each step the node emission, the cell
// updates and the node hits (a simulation's n_blocks cover both its lattice
// blocks and its node blocks). A CTA takes the next ticket when it starts
// (ticket = phase x total_blocks + work block), and a CTA of phase k > 0
// first waits until every work block of phase k - 1 has finished: each
// phase reads what the previous one wrote. Tickets follow the order in
// which CTAs actually start, so every CTA a waiter depends on is already
// running or done, and the lowest unfinished phase never waits: the launch
// needs no co-residency guarantee. Each CTA runs exactly one work block,
// with no loop around the step (a loop of steps inside one CTA made the
// compiler spill about 1 KB per thread).
template <int ST, int LAYOUT, int NS, bool DET, bool RS, int PHYS>
__global__ void __launch_bounds__(kBlock, kGenMinBlocks) batch_step_kernel(const __grid_constant__ BatchLaunch p) {
  __shared__ int s_ticket;
  if (threadIdx.x == 0) {
    int tk = (int)atomicAdd(&p.sync->ticket, 1u);
    const int k = tk / p.total_blocks;
    if (*(volatile int *)&p.sync->timed_out ||
        (k > 0 &&
         !wait_counter(&p.sync->done[k - 1], (unsigned)p.total_blocks, &p.sync->timed_out, kWaitTimeoutNs)))
      tk = -1;
    s_ticket = tk;
  }
  __syncthreads();
  const int t = s_ticket;
  if (t < 0) return;  // a wait gave up: the host reports it
  const int ph = t / p.total_blocks;
  const int w = t - ph * p.total_blocks;
  const int ks = p.k0 + ph / 3;
  const int q = batch_sim_of(p, w);
  const StepArgs &a = p.v[q][ks % 6];
  const int64_t step = p.t0[q] + ks;
  const int blk = w - p.block_start[q];
  if (ph % 3 == 1) {
    if (a.parity)
      step_block<ST, LAYOUT, NS, 1, PHYS>(a, blk, step);
    else
      step_block<ST, LAYOUT, NS, 0, PHYS>(a, blk, step);
  } else if (!a.sp_bb) {
    if (ph % 3 == 0)
      node_block<ST, LAYOUT, NS, DET, RS, kNodeEmit>(a, blk, step);
    else
      node_block<ST, LAYOUT, NS, DET, RS, kNodeHits>(a, blk, step);
  }
  __syncthreads();  // every thread's writes of this block precede the release
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&p.sync->done[ph], 1u);
  }
}

// Simulation whose blocks [start[k], start[k + 1]) hold block w.
__device__ __forceinline__ int batch_owner(const int32_t *start, int n, int w) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= w)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// Per-step batched node kernels: node block w - node_start[q] of simulation
// q, each at its own step.
template <int ST, int LAYOUT, int NS, bool DET, bool RS, int MODE>
__global__ void __launch_bounds__(kBlock, node_min_blocks(ST, MODE)) batch_node_kernel(const __grid_constant__ BatchLaunch p) {
  const int w = (int)blockIdx.x;
  const int q = batch_owner(p.node_start, p.n_sims, w);
  const StepArgs &a = p.v[q][p.k0 % 6];
  if (a.sp_bb) return;
  node_block<ST, LAYOUT, NS, DET, RS, MODE>(a, w - p.node_start[q], p.t0[q] + p.k0);
}

// Per-step batched cell launches, as for a single simulation: the general
// warps and the fast ones of every simulation of one parity in one launch
// (each simulation's general blocks first), and on odd steps the region warps
// in a launch of their own before it where the batch has enough of them. The
// batch is ordered by parity, so a launch takes one run of simulations
// (sim_0: the first) and no block is launched for nothing; each launch has its
// parity's register budget. Same arithmetic and face-flow slots as the
// single-simulation kernels, so a simulation evolves identically alone or
// batched.
//
// One tick of the serving loop (24 boxes of side 48 to 192, FP16, 40 steps)
// took 102.8 ms with a launch of the general warps, a launch for each parity
// over every block and no region launch; now 91.1. The launches do not overlap
// as a single simulation's do: on that batch it is worth 0.7 %.
template <int ST, int LAYOUT, int NS, int PHYS, int ODD, bool UNI = false>
__global__ void __launch_bounds__(kCellBlock, cell_min_blocks(ST))
    batch_cell_kernel(const __grid_constant__ BatchLaunch p, int sim_0) {
  const int32_t *const start = UNI ? p.uni_start : p.cell_start;
  const int w = start[sim_0] + (int)blockIdx.x;
  const int q = batch_owner(start, p.n_sims, w);
  const StepArgs &a = p.v[q][p.k0 % 6];
  const int64_t step = p.t0[q] + p.k0;
  int b = w - start[q];
  if (!UNI) {
    const int n_gen_blocks = (a.n_gen + kWarpsPerBlock - 1) / kWarpsPerBlock;
    if (b < n_gen_blocks) {
      const int gw = b * kWarpsPerBlock + (int)(threadIdx.x >> 5);
      if (gw < a.n_gen) gen_warp<ST, LAYOUT, NS, ODD, PHYS>(a, gw, step);
      return;
    }
    b -= n_gen_blocks;
  }
  const int list_0 = (ODD && !UNI && p.uni) ? a.n_uni : 0;
  fast_warp<ST, LAYOUT, NS, ODD, PHYS, UNI, kRelNear>(a, list_0 + b * kWarpsPerBlock + (int)(threadIdx.x >> 5), step);
}

// Per-plane FP64 sums of the current state: one cluster of `parts` blocks
// (sum_blocks) per plane, which share out its entries and nodes and add their
// partial sums in rank order through distributed shared memory (no scratch in
// device memory, the same order on every call). Columns: rho_C, rho_R, rho_P,
// rho_P u_z over the plane's fluid cells (u_z the carrier's, or the
// barycentric one when a.bary), and the raw wall hits A^R, A^P of the last
// step over the plane's catalytic nodes. Inlet/outlet planes give zeros.
//
// Bound by the bytes of the populations, read once, and next to that by the
// FP64 pipe (two lanes per SM): a cell costs four conversions, three adds and
// one fused multiply-add; the ones of the densities are counted, not added.
// One block per plane left few warps in flight and the chip to the last
// blocks' tails: the whole call took 1,347 us on the 256x256x512 box (FP16,
// even state), 5,249 (FP16, odd), 1,593 and 2,641 (FP32), now 917, 2,318, 1,248
// and 1,683.
constexpr int kSumBlocks = 8;  // (the largest portable cluster)
// Blocks per plane: 8, halved while a block would hold fewer cells than its
// share of the grid's cost allows: 3,072 where the grid has more than 12 blocks
// per SM, 1,024 from 6, and 768 (fluid-only) or 256 (dense, whose solid cells
// leave the blocks uneven) from 2. A block costs 30 ns of the whole grid's time
// however few its cells are, so 8 for every plane were slow where planes are
// small and many. us of an lbm_observables_noalloc call (FP32, even state,
// fluid-only) with 1, 2, 4 and 8, the one taken in brackets: 16x16x4000 (385)
// 521 781 1,324; 24x24x256 (64) 67 82 114; 48x48x128 66 (65) 67 85; 64x64x64 78
// 64 (54) 64; 64x64x1024 (281) 300 351 511; 128x128x32 189 123 84 (68);
// 128x128x256 261 239 (250) 275; 256x256x512 1,425 1,423 1,366 (1,432). Over
// 1,440 boxes and states it is within 4 % of 8 wherever that is better, within
// 22 % of the best of the four, and 13 % below 8 in the mean.
inline int sum_blocks(const StepArgs &a, int layout) {
  const int64_t plane = (int64_t)a.nx * a.ny, sms = 152;
  int parts = kSumBlocks;
  for (; parts > 1; parts /= 2) {
    const int64_t blocks = (int64_t)a.nz * parts;
    const int64_t least = blocks > 12 * sms  ? 3072
                          : blocks > 6 * sms ? 1024
                          : blocks > 2 * sms ? (layout == LBM_LAYOUT_DENSE ? 256 : 768)
                                                : 0;
    if (plane >= least * parts) break;
  }
  return parts;
}
// Blocks per SM. Odd states load slot by slot, so they want warps: FP16 3,100,
// 2,318, 2,474 us at 3, 4, 5 blocks, FP32 1,772, 1,683, 2,377 (more blocks
// spill). Even ones: FP16 1,026, 982, 917, 1,133 at 2, 3, 4, 5; FP32 1,248,
// 1,261, 1,354 at 2, 3, 4.
constexpr int sum_min_blocks(int st, int odd) { return !odd && st == LBM_FP32 ? 2 : 4; }
// PARTS: the number of blocks where it is known at compile time, else 0. Eight,
// the large planes' number, has an instance of its own: 256x256x512 FP16 906 us
// (even) and 2,288 (odd), against 931 and 2,324 with the number as an argument.
template <int ST, int LAYOUT, int NS, int ODD, bool DET, int PARTS>
__global__ void __launch_bounds__(kBlock, sum_min_blocks(ST, ODD)) plane_sums_kernel(const ObsArgs o, const int n_parts) {
  const int parts = PARTS ? PARTS : n_parts;
  namespace cg = cooperative_groups;
  const cg::cluster_group cluster = cg::this_cluster();
  const StepArgs &a = o.s;
  const int z = (int)blockIdx.x / parts, part = (int)blockIdx.x % parts;
  const bool bc = (!a.periodic_z && (z == 0 || z == a.nz - 1)) || halo_plane(a, z);
  double s[kPlaneCols] = {0, 0, 0, 0, 0, 0};
  if (!bc) {
    const int64_t hi = o.lat_plane[z + 1];
    int cells = 0;
    for (int64_t Lw = o.lat_plane[z] + part * kBlock + threadIdx.x; Lw < hi; Lw += parts * kBlock) {
      const int32_t L = (int32_t)Lw;
      const int32_t cell = (LAYOUT == LBM_LAYOUT_DENSE) ? L : __ldg(a.fcell + L);
      const uint32_t nbm = __ldg(a.nbm + L);
      if (LAYOUT == LBM_LAYOUT_DENSE && __ldg(a.mask + cell)) continue;
      const int32_t xy = cell - z * a.nx * a.ny;
      const int y = (int)fast_div((uint32_t)xy, a.div_nx_m, (a.div_sh >> 16) & 0xffu, a.div_sh >> 24);
      const Nbr nb(cell, xy - y * a.nx, y, z, a.nx, a.ny, a.nz, a.periodic_z);
      float f[NS][kQ];
      load_cell_by_slot<ST, LAYOUT, NS, ODD, DET>(a, L, nb, nbm, f);
      float drho = 0.f, jz = 0.f, rR = 0.f, rP = 0.f, jzs = 0.f;
#pragma unroll
      for (int i = 0; i < kQ; ++i) {
        drho += f[0][i];
        jz += cz(i) * f[0][i];
        if (NS > 1) rR += f[1][i];
        if (NS > 2) rP += f[NS - 1][i];
#pragma unroll
        for (int sp = 1; sp < NS; ++sp) jzs += cz(i) * f[sp][i];
      }
      ++cells;
      s[0] += (double)drho;
      s[1] += (double)rR;
      const float uz = a.bary ? (jz + jzs) / ((1.0f + drho) + (rR + rP)) : jz / (1.0f + drho) + 0.5f * a.g_z;
      const double P = (double)rP;
      s[2] += P;
      s[3] = fma(P, (double)uz, s[3]);
    }
    s[0] += (double)cells;
    if (NS > 1) {
      for (int64_t k = o.node_plane[z] + part * kBlock + threadIdx.x; k < o.node_plane[z + 1]; k += parts * kBlock) {
        s[4] += hits_d<DET>(a, 0, k);
        if (NS > 2) s[5] += hits_d<DET>(a, 1, k);
      }
    }
  }
  // FP64 sums in a fixed order: lanes, warps, then the cluster's blocks
  __shared__ double sh[kPlaneCols][kBlock / 32];
  __shared__ double total[kPlaneCols];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kPlaneCols; ++k) {
    double v = warp_sum_d(s[k]);
    if (lane == 0) sh[k][wid] = v;
  }
  __syncthreads();
  if (threadIdx.x < kPlaneCols) {
    double v = 0.0;
    for (int w = 0; w < kBlock / 32; ++w) v += sh[threadIdx.x][w];
    total[threadIdx.x] = v;
  }
  cluster.sync();
  if (part == 0 && threadIdx.x < kPlaneCols) {
    double v = 0.0;
    for (int r = 0; r < parts; ++r) v += *cluster.map_shared_rank(&total[threadIdx.x], r);
    o.plane_sums[kPlaneCols * (int64_t)z + threadIdx.x] = v;
  }
  cluster.sync();  // (a block's shared memory lives until the sums are read)
}

// The species' momenta together, direction by direction.
template <int ST, int NS>
__device__ __forceinline__ float species_momentum(const float (&d)[NS][kQ], int dir) {
  float j = 0.f;
#pragma unroll
  for (int i = 0; i < kQ; ++i)
#pragma unroll
    for (int k = 1; k < NS; ++k) {
      const int c = dir == 0 ? cx(i) : (dir == 1 ? cy(i) : cz(i));
      j = __fadd_rn(j, __fmul_rn(c * wq(i) * Pop<ST, NS>::kSpInv, d[k][i]));
    }
  return j;
}

// What an export reads: the carrier's populations, the species', or both
// (all populations; the barycentric velocity).
constexpr int kReadCarrier = 1, kReadSpecies = 2, kReadAll = 3;
inline int export_reads(const StepArgs &a, int which) {
  if (which < 0) return kReadAll;
  if (which == LBM_FIELD_RHO_R || which == LBM_FIELD_RHO_P) return kReadSpecies;
  const bool velocity = which == LBM_FIELD_UX || which == LBM_FIELD_UY || which == LBM_FIELD_UZ;
  return velocity && a.bary ? kReadAll : kReadCarrier;
}

// Dense export of a field (which >= 0) or of all populations (which < 0).
// Bound by the bytes of the arrays it reads, once the loads of a cell are in
// flight together. 256x256x512, us per field, before (every reader took both
// arrays, 80 registers) and now: carrier fields 1,094 -> 393 (FP32, even
// state), 2,193 -> 527 (FP32, odd), 1,007 -> 306 and 3,094 -> 485 (FP16);
// species 1,089 -> 714, 2,190 -> 888, 1,000 -> 472, 3,091 -> 689.
// Blocks per SM, the fastest of those measured there (3-6): a carrier reader
// at 5 or 6, a species reader at 4 or 5 unless its odd FP32 form spills (995
// us at 4, 946 at 3), a reader of both at 3.
constexpr int export_min_blocks(int st, int odd, int read) {
  return read == kReadAll ? 3 : read == kReadCarrier ? (odd ? 6 : 5) : st == LBM_FP32 ? (odd ? 3 : 4) : (odd ? 4 : 5);
}
template <int ST, int LAYOUT, int NS, int ODD, bool DET, int READ>
__global__ void __launch_bounds__(kBlock, export_min_blocks(ST, ODD, READ))
    export_kernel(const StepArgs a, int which, float *dst, int64_t n) {
  const int64_t Lw = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  if (Lw >= a.n_lat) return;
  const int32_t L = (int32_t)Lw;
  const int32_t cell = (LAYOUT == LBM_LAYOUT_DENSE) ? L : __ldg(a.fcell + L);
  const uint32_t nbm = __ldg(a.nbm + L);
  if (LAYOUT == LBM_LAYOUT_DENSE && __ldg(a.mask + cell)) return;
  const int z = (int)fast_div((uint32_t)cell, a.div_plane_m, a.div_sh & 0xffu, (a.div_sh >> 8) & 0xffu);
  // inlet/outlet planes hold no state of their own (their upwind cells lie
  // outside the box): leave them at 0
  if ((!a.periodic_z && (z == 0 || z == a.nz - 1)) || halo_plane(a, z)) return;
  float d[NS][kQ];
  load_cell<ST, LAYOUT, NS, ODD, DET, (READ & kReadCarrier) != 0, (READ & kReadSpecies) != 0>(a, L, cell, nbm, d);
  if (READ == kReadAll && which < 0) {
#pragma unroll
    for (int s = 0; s < NS; ++s)
#pragma unroll
      for (int i = 0; i < kQ; ++i) dst[(int64_t)(s * kQ + i) * n + cell] = wq(i) * (s ? Pop<ST, NS>::kSpInv : 1.0f) * d[s][i];
    return;
  }
  float v = 0.f;
  if (READ == kReadSpecies) {
    v = cell_density<ST, NS>(d, which == LBM_FIELD_RHO_R ? 1 : NS - 1);
  } else {
    const float drho = cell_density<ST, NS>(d, 0), rho = 1.0f + drho;
    if (which == LBM_FIELD_RHO_C) {
      v = rho;
    } else if (which == LBM_FIELD_DRHO_C) {
      v = drho;
    } else {
      // velocity: the carrier's, or the barycentric one over every array
      float j[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        j[k] = cell_momentum<ST, NS>(d, 0, k);
        if (READ == kReadAll) j[k] += species_momentum<ST, NS>(d, k);
      }
      float over = rho;
      if (READ == kReadAll) over = rho + (cell_density<ST, NS>(d, 1) + (NS > 2 ? cell_density<ST, NS>(d, NS - 1) : 0.f));
      v = (which == LBM_FIELD_UX ? j[0] : which == LBM_FIELD_UY ? j[1] : j[2]) / over;
      if (READ != kReadAll && which == LBM_FIELD_UZ) v += 0.5f * a.g_z;
    }
  }
  dst[cell] = v;
}

#define LBM_DISPATCH_ONE(LYV, NSV, ODDV, DETV, ...) \
  do {                                              \
    constexpr int LY = LYV;                         \
    constexpr int NSC = NSV;                        \
    constexpr int OD = ODDV;                        \
    constexpr bool DT = DETV;                       \
    (void)LY; (void)NSC; (void)OD; (void)DT;        \
    __VA_ARGS__;                                    \
  } while (0)
#define LBM_DISPATCH_D(LYV, NSV, ODDV, DET_, ...)                                            \
  do {                                                                                     \
    if (DET_) LBM_DISPATCH_ONE(LYV, NSV, ODDV, true, __VA_ARGS__);                         \
    else LBM_DISPATCH_ONE(LYV, NSV, ODDV, false, __VA_ARGS__);                             \
  } while (0)
#define LBM_DISPATCH_O(LYV, NSV, ODD_, DET_, ...)                                            \
  do {                                                                                     \
    if (ODD_) LBM_DISPATCH_D(LYV, NSV, 1, DET_, __VA_ARGS__);                              \
    else LBM_DISPATCH_D(LYV, NSV, 0, DET_, __VA_ARGS__);                                   \
  } while (0)
#define LBM_DISPATCH_N(LYV, NS_, ODD_, DET_, ...)                                            \
  do {                                                                                     \
    if ((NS_) == 2) LBM_DISPATCH_O(LYV, 2, ODD_, DET_, __VA_ARGS__);                       \
    else LBM_DISPATCH_O(LYV, 3, ODD_, DET_, __VA_ARGS__);                                  \
  } while (0)
// layout and species count only (LY, NSC)
#define LBM_DISPATCH_LN(LAYOUT_, NS_, ...)                                      \
  do {                                                                          \
    if ((LAYOUT_) == LBM_LAYOUT_DENSE) {                                        \
      constexpr int LY = LBM_LAYOUT_DENSE;                                      \
      if ((NS_) == 2) { constexpr int NSC = 2; __VA_ARGS__; }                   \
      else { constexpr int NSC = 3; __VA_ARGS__; }                              \
    } else {                                                                    \
      constexpr int LY = LBM_LAYOUT_FLUID;                                      \
      if ((NS_) == 2) { constexpr int NSC = 2; __VA_ARGS__; }                   \
      else { constexpr int NSC = 3; __VA_ARGS__; }                              \
    }                                                                           \
  } while (0)

// species count only (NSC)
#define LBM_DISPATCH_FLUID_N(NS_, ...)                                          \
  do {                                                                          \
    if ((NS_) == 2) { constexpr int NSC = 2; __VA_ARGS__; }                     \
    else { constexpr int NSC = 3; __VA_ARGS__; }                                \
  } while (0)

// layout x species x parity x deterministic accumulation
#define LBM_DISPATCH_LNS(LAYOUT_, NS_, ODD_, DET_, ...)                                      \
  do {                                                                                     \
    if ((LAYOUT_) == LBM_LAYOUT_DENSE) LBM_DISPATCH_N(LBM_LAYOUT_DENSE, NS_, ODD_, DET_, __VA_ARGS__); \
    else LBM_DISPATCH_N(LBM_LAYOUT_FLUID, NS_, ODD_, DET_, __VA_ARGS__);                   \
  } while (0)

// A launch of the step's chain on st; overlap: it may begin before the kernel
// ahead of it on the stream has completed (see chain_wait).
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), unsigned grid, int threads, cudaStream_t st, bool overlap, const A &...args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3((unsigned)threads);
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, args...);
}

// Whether three planes' populations take so much of L2 that odd steps keep to
// kRelWide offsets (see rel_slot).
template <int ST>
bool wide_planes(const StepArgs &a, int layout, int ns) {
  const int64_t entry = kQ * (int64_t)(sizeof(typename Pop<ST, 3>::C) + (ns == 3 ? sizeof(typename Pop<ST, 3>::S) : sizeof(typename Pop<ST, 2>::S)));
  return layout == LBM_LAYOUT_FLUID && 3 * entry * (a.n_lat / a.nz) > kWidePlanes;
}

// RS (the random sputtering matrix) and PHYS (carrier velocity; barycentric
// velocity; validation channel: inert solid, body force, species relaxation
// time) are compile-time parameters, so that the default kernels carry none
// of the other modes' code.
template <int ST, bool RS, int PHYS>
cudaError_t launch_step_st(const StepArgs &a, int layout, int ns, int parity, cudaStream_t st, const cudaEvent_t *ev,
                           bool first, bool last) {
  if (ev) cudaEventRecord(ev[0], st);
  const unsigned ggrid = (unsigned)((a.n_gen + kWarpsPerBlock - 1) / kWarpsPerBlock);
  const unsigned ngrid = a.sp_bb ? 0u : (unsigned)((a.n_nodes + kBlock - 1) / kBlock);
  const bool overlap = !ev;  // (timed apart, each launch waits for the one before)
  cudaError_t e = cudaSuccess;
  if (ngrid > 0 && first)
    LBM_DISPATCH_LNS(layout, ns, 0, a.det, e = launch_chained(node_kernel<ST, LY, NSC, DT, RS, kNodeEmit>, ngrid, kBlock, st, overlap, a));
  if (e != cudaSuccess) return e;
  if (ev) cudaEventRecord(ev[1], st);
  // even steps: the whole fast list in one launch; odd steps: the region
  // warps (fluid-only addressing, where there are enough of them), then the
  // plain and wall warps in increasing order
  const int32_t n_uni = (parity && layout == LBM_LAYOUT_FLUID && a.n_uni >= kUniMinWarps) ? a.n_uni : 0;
  constexpr int kRel = PHYS == kPhysCarrier && ST != LBM_FP32 ? kRelWide : kRelNear;
  const bool wide = kRel == kRelWide && wide_planes<ST>(a, layout, ns);
  if (n_uni > 0) {
    const unsigned ugrid = (unsigned)((n_uni + kWarpsPerBlock - 1) / kWarpsPerBlock);
    if (wide)
      LBM_DISPATCH_FLUID_N(ns, e = launch_chained(cell_kernel<ST, LBM_LAYOUT_FLUID, NSC, 1, PHYS, true, kRel>, ugrid, kCellBlock, st, overlap, a, 0, 0));
    else
      LBM_DISPATCH_FLUID_N(ns, e = launch_chained(cell_kernel<ST, LBM_LAYOUT_FLUID, NSC, 1, PHYS, true>, ugrid, kCellBlock, st, overlap, a, 0, 0));
    if (e != cudaSuccess) return e;
  }
  const unsigned fgrid =
      (unsigned)(((int64_t)a.n_fast + a.n_wall - n_uni + kWarpsPerBlock - 1) / kWarpsPerBlock);
  auto cells = [&](unsigned block_0, unsigned blocks) {
    if (blocks == 0) return cudaSuccess;
    cudaError_t r;
    if (parity && wide)
      LBM_DISPATCH_FLUID_N(ns, r = launch_chained(cell_kernel<ST, LBM_LAYOUT_FLUID, NSC, 1, PHYS, false, kRel>, blocks, kCellBlock, st, overlap, a, (int)block_0, n_uni));
    else if (parity)
      LBM_DISPATCH_LN(layout, ns, r = launch_chained(cell_kernel<ST, LY, NSC, 1, PHYS>, blocks, kCellBlock, st, overlap, a, (int)block_0, n_uni));
    else
      LBM_DISPATCH_LN(layout, ns, r = launch_chained(cell_kernel<ST, LY, NSC, 0, PHYS>, blocks, kCellBlock, st, overlap, a, (int)block_0, n_uni));
    return r;
  };
  if (ev) {  // the fast and the general warps timed apart
    e = cells(ggrid, fgrid);
    if (e != cudaSuccess) return e;
    cudaEventRecord(ev[2], st);
    e = cells(0, ggrid);
  } else {
    e = cells(0, ggrid + fgrid);
  }
  if (e != cudaSuccess) return e;
  if (ev) cudaEventRecord(ev[3], st);
  if (ngrid > 0) {
    if (last)
      LBM_DISPATCH_LNS(layout, ns, 0, a.det, e = launch_chained(node_kernel<ST, LY, NSC, DT, RS, kNodeHits>, ngrid, kBlock, st, overlap, a));
    else
      LBM_DISPATCH_LNS(layout, ns, 0, a.det, e = launch_chained(node_kernel<ST, LY, NSC, DT, RS, kNodeBoth>, ngrid, kBlock, st, overlap, a));
  }
  if (ev) cudaEventRecord(ev[4], st);
  return e;
}

template <int ST, bool RS, int PHYS>
cudaError_t launch_batch_st(const BatchLaunch &p, int layout, int ns, int det, cudaStream_t st) {
  if (p.total_blocks <= 0 || p.n_sims <= 0 || p.n_steps <= 0) return cudaSuccess;
  if (!p.sync || p.n_steps > kStepsPerLaunch) return cudaErrorInvalidValue;
  if (3 * (int64_t)p.n_steps * p.total_blocks >= ((int64_t)1 << 31)) return cudaErrorInvalidValue;
  const unsigned grid = (unsigned)(3 * p.n_steps * p.total_blocks);
  LBM_DISPATCH_LNS(layout, ns, 0, det, batch_step_kernel<ST, LY, NSC, DT, RS, PHYS><<<grid, kBlock, 0, st>>>(p));
  return cudaGetLastError();
}

template <int ST, bool RS, int PHYS>
cudaError_t launch_batch_split_st(const BatchLaunch &p, int layout, int ns, int det, cudaStream_t st, bool first,
                                  bool last) {
  if (p.n_sims <= 0 || p.n_steps != 1) return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
  const unsigned ngrid = (unsigned)p.total_node;
  if (ngrid > 0 && first)
    LBM_DISPATCH_LNS(layout, ns, 0, det, e = launch_chained(batch_node_kernel<ST, LY, NSC, DT, RS, kNodeEmit>, ngrid, kBlock, st, false, p));
  if (e != cudaSuccess) return e;
  // the run of simulations at the first one's parity, then the others
  const int run[3] = {0, p.n_lead, p.n_sims};
  for (int r = 0; r < 2; ++r) {
    const int q0 = run[r], q1 = run[r + 1];
    if (q0 == q1) continue;
    const int odd = p.v[q0][p.k0 % 6].parity;
    const unsigned ugrid = odd ? (unsigned)(p.uni_start[q1] - p.uni_start[q0]) : 0u;
    if (ugrid > 0) {  // (p.uni: fluid-only addressing)
      if (ns == 2)
        e = launch_chained(batch_cell_kernel<ST, LBM_LAYOUT_FLUID, 2, PHYS, 1, true>, ugrid, kCellBlock, st, false, p, q0);
      else
        e = launch_chained(batch_cell_kernel<ST, LBM_LAYOUT_FLUID, 3, PHYS, 1, true>, ugrid, kCellBlock, st, false, p, q0);
      if (e != cudaSuccess) return e;
    }
    const unsigned grid = (unsigned)(p.cell_start[q1] - p.cell_start[q0]);
    if (grid == 0) continue;
    if (odd)
      LBM_DISPATCH_LN(layout, ns, e = launch_chained(batch_cell_kernel<ST, LY, NSC, PHYS, 1>, grid, kCellBlock, st, false, p, q0));
    else
      LBM_DISPATCH_LN(layout, ns, e = launch_chained(batch_cell_kernel<ST, LY, NSC, PHYS, 0>, grid, kCellBlock, st, false, p, q0));
    if (e != cudaSuccess) return e;
  }
  if (ngrid > 0) {
    if (last)
      LBM_DISPATCH_LNS(layout, ns, 0, det, e = launch_chained(batch_node_kernel<ST, LY, NSC, DT, RS, kNodeHits>, ngrid, kBlock, st, false, p));
    else
      LBM_DISPATCH_LNS(layout, ns, 0, det, e = launch_chained(batch_node_kernel<ST, LY, NSC, DT, RS, kNodeBoth>, ngrid, kBlock, st, false, p));
  }
  return e;
}

template <int ST>
cudaError_t launch_plane_sums_st(const ObsArgs &o, int layout, int ns, cudaStream_t st) {
  const int parts = sum_blocks(o.s, layout);
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)parts;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)o.s.nz * (unsigned)parts);
  c.blockDim = dim3(kBlock);
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaError_t e = cudaSuccess;
  if (parts == kSumBlocks)
    LBM_DISPATCH_LNS(layout, ns, o.parity, o.s.det, e = cudaLaunchKernelEx(&c, plane_sums_kernel<ST, LY, NSC, OD, DT, kSumBlocks>, o, parts));
  else
    LBM_DISPATCH_LNS(layout, ns, o.parity, o.s.det, e = cudaLaunchKernelEx(&c, plane_sums_kernel<ST, LY, NSC, OD, DT, 0>, o, parts));
  return e;
}

template <int ST>
cudaError_t launch_export_st(const StepArgs &a, int parity, int layout, int ns, int which, float *dst,
                             cudaStream_t st) {
  const unsigned grid = (unsigned)((a.n_lat + kBlock - 1) / kBlock);
  if (grid == 0) return cudaSuccess;
  const int64_t n = (int64_t)a.nx * a.ny * a.nz;
  switch (export_reads(a, which)) {
    case kReadCarrier:  // (no wall hits: one form for either accumulator)
      if (parity)
        LBM_DISPATCH_LN(layout, ns, export_kernel<ST, LY, NSC, 1, false, kReadCarrier><<<grid, kBlock, 0, st>>>(a, which, dst, n));
      else
        LBM_DISPATCH_LN(layout, ns, export_kernel<ST, LY, NSC, 0, false, kReadCarrier><<<grid, kBlock, 0, st>>>(a, which, dst, n));
      break;
    case kReadSpecies:
      LBM_DISPATCH_LNS(layout, ns, parity, a.det,
                       export_kernel<ST, LY, NSC, OD, DT, kReadSpecies><<<grid, kBlock, 0, st>>>(a, which, dst, n));
      break;
    default:
      LBM_DISPATCH_LNS(layout, ns, parity, a.det,
                       export_kernel<ST, LY, NSC, OD, DT, kReadAll><<<grid, kBlock, 0, st>>>(a, which, dst, n));
  }
  return cudaGetLastError();
}

#define LBM_INSTANTIATE_STEP(ST, RS, PHYS)                                                           \
  template cudaError_t launch_step_st<ST, RS, PHYS>(const StepArgs &, int, int, int, cudaStream_t, const cudaEvent_t *, \
                                                          bool, bool);                                     \
  template cudaError_t launch_batch_st<ST, RS, PHYS>(const BatchLaunch &, int, int, int, cudaStream_t);   \
  template cudaError_t launch_batch_split_st<ST, RS, PHYS>(const BatchLaunch &, int, int, int, cudaStream_t, bool, bool);
#define LBM_INSTANTIATE_STORAGE(ST)                                                                    \
  LBM_INSTANTIATE_STEP(ST, false, kPhysCarrier)                                                               \
  template cudaError_t launch_plane_sums_st<ST>(const ObsArgs &, int, int, cudaStream_t);             \
  template cudaError_t launch_export_st<ST>(const StepArgs &, int, int, int, int, float *, cudaStream_t);

}  // namespace lbm

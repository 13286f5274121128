// Density and force passes (Section II: two interaction stages), the ghost /
// h-update step between them, the FP64 conservation reductions and the
// per-field output gathers.
//
// Pair-interactions follow the sorted cell-pair interaction of Section II-C
// (Fig. 3) at warp granularity: particles are grouped into clusters of at most
// 32; a warp takes one cluster of cell A and walks the clusters of cell B in
// their sorted order along the axis joining the cell centres, stopping once the
// projected gap exceeds every support radius that could still bridge it, and
// culling clusters whose boxes are out of reach.  Each in-reach particle pair
// is found once and updates both sides (Section II-D: symmetric interactions).
#include "sph_engine.h"

#include <cfloat>
#include <mutex>

namespace sph {

constexpr float BAND_REL = 7.62939453125e-06f;  // 2^-17: guard band of the FP32 predicate

struct ItemGeom {
  float e;          // cell edge (units of L)
  float3 offB;      // centre of B minus centre of A (units of L), exact: e * db
  float invL;
  float es;         // absolute rounding of plain FP32 positions added to the culling slack
  float drift;      // largest displacement since the decomposition was built (units of L)
};

__device__ __forceinline__ ItemGeom item_geom(const Tree& T, const BoxDesc* box, int A, int ax) {
  ItemGeom g;
  const int d = T.level[A];
  const BoxDesc bd = box[T.box[A]];
  g.e = ldexpf(1.0f, -d);
  int dx, dy, dz;
  axis_vec(ax, dx, dy, dz);
  g.offB = make_float3(g.e * dx, g.e * dy, g.e * dz);
  g.invL = (float)bd.invL;
  g.es = bd.global32 ? 9.5367431640625e-07f : 0.0f;   // 2^-20 L: the 2^-25 rounding of both positions
  g.drift = bd.drift_u;
  return g;
}

// Units of work are handed out from a counter in device memory (zeroed before every
// launch): their cost varies by orders of magnitude, so a static split leaves most
// SMs idle behind the longest ones.

// Blocks per SM of the recording first density pass (4.2M clustered 10.2 ms at 5, 9.9 at 6,
// 9.2 at 7), of the plain first pass (see k_density) and of the later passes; the
// gathered ones have GATHER_BLOCKS.  (4.2M clustered h iteration, all three at once: density
// phase 39.4 ms at 6, 38.8 at 7, 40.6 at 8.)
#ifndef REC_BLOCKS
#define REC_BLOCKS 7
#endif
#ifndef DENS_BLOCKS
#define DENS_BLOCKS 7
#endif
#ifndef PART_BLOCKS
#define PART_BLOCKS 7
#endif

// Exact decision r_ij < H (physical H) from the caller's FP64 positions.
__device__ __noinline__ bool exact_less(int gi, int gj, float Hphys, const unsigned int* __restrict__ perm,
                                        const double* __restrict__ x, double L, double halfL, int periodic) {
  const long long i = perm[gi], j = perm[gj];
  const double xi[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
  const double xj[3] = {x[3 * j], x[3 * j + 1], x[3 * j + 2]};
  return canonical_less(canonical_r2(xi, xj, L, halfL, periodic), Hphys);
}

// =========================================================================== density
struct Box3 {
  float3 lo, hi;
};

// Per warp: what a unit of work (one cluster against the clusters of its cell's
// interactions) keeps out of registers: its constants, the current group of
// interactions, and the candidate clusters of the current scan.  Read back with
// broadcast loads where they are needed, which costs less than the registers they
// would hold through the batches.
constexpr int GROUP = 14;      // interactions whose geometry is set up at once, one per lane (a leaf's self and 13 pairs)

struct __align__(16) UnitShared {
  float4 blo;            // box of the own cluster's particles to find partners for (leaf frame); w: their largest H
  float4 bhi;            // ... w: 1 / L
  float4 clo, chi;       // box of the whole own cluster; w of clo: its largest H
  float4 cl;             // its leaf's centre
  float eb;              // length scale of the position rounding: the cell edge, or 1 (L) for plain FP32 positions
  float es, L32, drift;
  int box, cell;         // the cell whose interactions come next (-1: none left)
  unsigned int ti, at, idx;    // own cluster; position in the cell's list; interactions seen so far
  unsigned int part, parts;    // the unit's share of the cluster's work
  unsigned int gidx;           // interactions seen before the current group
  int selfit;                  // the group's self interaction (-1: none)
  // per interaction of the group: frame offset of the partner cell's clusters (exact) and culling slack; sorted
  // window offset (projection of the cell offset minus the drift and the own upper end), the partner cell's
  // largest H, its sorted list (SORT_NONE: clusters tb, tb + 1, ... in their own order) and length
  float4 gsh[GROUP];
  float4 gwin[GROUP];
  unsigned int gtb[GROUP];
  float4 co[32];         // candidates: frame offset, first particle (bits)
  unsigned char cn[32];  //   size
};

// The lane's own particle of a density unit.
struct DensI {
  float3 p;
  float H, invH, Hphys, m;
  int g;
  bool valid, act;
};

// (in the frame of its leaf: its offset as stored)
__device__ __forceinline__ DensI load_dens(bool valid, unsigned int gidx, const float4* pos4, const float4* cen4,
                                           const unsigned char* act, float invL) {
  DensI r;
  r.valid = valid;
  if (valid) {
    const float4 p = pos4[gidx];
    r.p = make_float3(p.x, p.y, p.z);
    const float H = p.w * invL;
    r.H = H;
    r.invH = __fdividef(1.0f, H);   // 2 ulp: enters the kernel's argument only
    r.Hphys = p.w;
    r.m = cen4[gidx].w;
    r.g = (int)gidx;
    r.act = act ? act[gidx] != 0 : true;   // no activity array: every particle iterates
  } else {
    r.p = make_float3(1e30f, 1e30f, 1e30f);
    r.H = 0.0f;
    r.invH = 0.0f;
    r.Hphys = 0.0f;
    r.m = 0.0f;
    r.g = -1;
    r.act = false;
  }
  return r;
}

// Per warp: the staged partners, the warp's own cluster (ip), and what the unit of
// work keeps out of registers.  The coordinates are kept apart so that the mask phase reads four slots of
// one coordinate with one 16-byte load, as two packed FP32 pairs.  A partner is
// staged with its position, H and index only; what follows from them is computed
// once per batch, by the slot's lane, and its mass is loaded then.
struct __align__(16) DensShared {
  float x[32], y[32], z[32];
  float hi[32];     // H^2 + guard band (units of L^2); -1 marks an empty slot
  float H[32];      // H (physical)
  float m[32];
  int g[32];
  float4 ip[32];    // own cluster: position, m
  float4 is[32];    //   sums over the interactions done
  int ig[32];       //   index
  UnitShared tk;
  float4 jlo[32], jhi[32];   // the scan's fine candidates: box in the unit's frame, largest H (w of jlo)
  unsigned char act[32];
  // pair records (first pass): the current task's first batch, batch count and
  // record slot, and 0 once one of its batches was lost (lane 0 keeps them)
  unsigned int rc_first, rc_nb, rc_slot, rc_ok;
};

// A warp's next batch (first pass, the same in every lane); a multiple of
// REC_CHUNK means that its chunk is used up (0: no chunk yet).
struct RecW {
  unsigned int pos = 0;
};

__device__ __forceinline__ void dens_put(DensShared& S, int slot, float3 p, float Hphys, unsigned int g, bool act) {
  S.x[slot] = p.x;
  S.y[slot] = p.y;
  S.z[slot] = p.z;
  S.H[slot] = Hphys;
  S.g[slot] = (int)g;
  S.act[slot] = act ? 1 : 0;
}

struct Counters {
  unsigned int cand = 0, pairs = 0, sides = 0, rechecks = 0;
};

template <bool COUNT>
__device__ __forceinline__ void commit_counters(const Counters& C, unsigned long long* pc, int which) {
  if (!COUNT) return;
  unsigned long long c = C.cand, p = C.pairs, s = C.sides, r = C.rechecks;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    c += __shfl_xor_sync(0xffffffffu, c, o);
    p += __shfl_xor_sync(0xffffffffu, p, o);
    s += __shfl_xor_sync(0xffffffffu, s, o);
    r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  if ((threadIdx.x & 31) == 0) {
    // pc: [0..2] density cell-pair kernel (pairs, sides, candidates), [3..5] density
    // self kernel, [6..7] force cell-pair kernel (pairs, candidates), [8..9] force
    // self kernel, [10] FP64 re-decisions
    const int base = which == 0 ? 0 : which == 1 ? 3 : which == 2 ? 6 : 8;
    atomicAdd(&pc[base], p);
    if (which < 2) atomicAdd(&pc[base + 1], s);
    atomicAdd(&pc[base + (which < 2 ? 2 : 1)], c);
    atomicAdd(&pc[10], r);
  }
}


// the lanes above this one
__device__ __forceinline__ unsigned int upper_mask(int lane) {
  return lane == 31 ? 0u : (0xffffffffu << (lane + 1));
}

// ------------------------------------------------------------- pair records
// Called by the whole warp.  A task starts with no batch; its batches go to the
// warp's current chunk, and to a new chunk (linked from the old one) when that is
// full.  A batch that finds the pool full is lost, and with it the task's record.
__device__ __forceinline__ void rec_task_begin(DensShared& S, unsigned int slot) {
  if ((threadIdx.x & 31) == 0) {
    S.rc_nb = 0;
    S.rc_ok = 1;
    S.rc_slot = slot;
  }
}

__device__ __forceinline__ void rec_batch(const PairRec& R, RecW& W, DensShared& S, unsigned int jvalid,
                                          unsigned int m) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  if (!S.rc_ok) return;
  if (W.pos % REC_CHUNK == 0u) {
    unsigned int c = 0;
    if (lane == 0) c = atomicAdd(R.ctr, 1u);
    c = __shfl_sync(0xffffffffu, c, 0);
    if (c >= R.cap) {
      if (lane == 0) S.rc_ok = 0;
      W.pos = 0;
      return;
    }
    if (lane == 0 && W.pos != 0) R.next[W.pos / REC_CHUNK - 1u] = c;
    W.pos = c * REC_CHUNK;
  }
  // streaming stores: the records are read once, by the force pass, and should
  // not push the particle data the passes share out of L2
  unsigned int* B = R.pool + 64ull * W.pos;
  __stcs(B + lane, (jvalid >> lane) & 1u ? (unsigned int)S.g[lane] : REC_NONE);
  __stcs(B + 32 + lane, m);
  if (lane == 0) {
    if (S.rc_nb == 0) S.rc_first = W.pos;
    S.rc_nb += 1;
  }
  W.pos += 1;
}

__device__ __forceinline__ void rec_task_end(uint2* slots, const DensShared& S) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0 && S.rc_ok) slots[S.rc_slot] = make_uint2(S.rc_nb ? S.rc_first : 0u, S.rc_nb);
}

// =========================================================================== force
// Per warp: the staged partners and the warp's own cluster.  A partner is staged
// with its position, H and index (as in the density pass); its velocity and ghost
// quantities are loaded once per batch by the slot's lane, before the masks, and
// written after them.  8 blocks of 4 warps fit an SM's shared memory.
constexpr unsigned int PLIST_CAP = 320;    // pairs listed at once (a batch with more runs in several goes)
struct __align__(16) ForceShared {
  float x[32], y[32], z[32];
  float hi[32], lo[32];  // H^2 +- guard band (units of L^2); hi = -1 marks an empty slot
  float H[32];           // staged: H (physical); in a batch: 1 / H (units of L)
  int g[32];
  float4 v[32];    // partner velocity, m; between batches the boxes of the scan's
  float4 f[32];    // partner rho, f P / rho^2, c, K/H^4;   fine candidates (lo, hi)
  float4 jacc[32]; // partner sums of the batch: acceleration (3), du/dt
  float jvs[32];   //   and largest signal velocity
  float4 ip[32];   // own cluster: position, m
  float4 iv[32];   // own cluster: velocity, rho
  float4 if_[32];  // own cluster: 1/H, f P / rho^2, c, K/H^4
  float ilo[32];   // own cluster: H^2 - guard band
  float4 iacc[32]; // own cluster sums over the task
  float ivs[32];
  UnitShared tk;
  float4 cb[32];         // partner-side terms of one round, by lane
  float cv[32];          //   signal velocities
  unsigned char plist[PLIST_CAP];   // the batch's pairs, own lane major: slot, bit 5: the first of its row
  unsigned int own0;     // the own cluster's first particle
};

// The lane's own particle (p.w: H in units of L; 1e30 and H = 0 on an empty lane).
__device__ __forceinline__ float4 force_stage_own(ForceShared& S, int lane, bool valid, unsigned int gidx,
                                                  const float4* pos4, const float4* cen4, const float4* vel4,
                                                  const float4* ghost4) {
  float4 p = make_float4(1e30f, 1e30f, 1e30f, 0.0f);
  float4 v = make_float4(0.f, 0.f, 0.f, 1.f), f = make_float4(0.f, 0.f, 0.f, 0.f);
  float m = 0.0f;
  if (valid) {
    p = pos4[gidx];
    const float4 vv = vel4[gidx], gh = ghost4[gidx];
    m = cen4[gidx].w;
    const float H = p.w * S.tk.bhi.w;
    p.w = H;
    v = make_float4(vv.x, vv.y, vv.z, gh.x);
    f = make_float4(gh.w * S.tk.L32, gh.y, gh.z, SPH_KNORM * (gh.w * gh.w) * (gh.w * gh.w));   // gh.w = 1 / H
  }
  S.ip[lane] = make_float4(p.x, p.y, p.z, m);
  S.iv[lane] = v;
  S.if_[lane] = f;
  S.iacc[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  S.ivs[lane] = 0.f;
  return p;
}

__device__ __forceinline__ void force_put(ForceShared& S, int slot, float3 p, float Hphys, unsigned int g) {
  S.x[slot] = p.x;
  S.y[slot] = p.y;
  S.z[slot] = p.z;
  S.H[slot] = Hphys;
  S.g[slot] = (int)g;
}

// The loads of a staged partner, and what the pair rounds read of it.
struct ForceRaw {
  float4 v, gh;
  float m;
};

__device__ __forceinline__ void force_derive(ForceShared& S, int lane, bool v, const ForceRaw& r) {
  if (v) {
    S.H[lane] = r.gh.w * S.tk.L32;                 // 1 / H in units of L
    S.v[lane] = make_float4(r.v.x, r.v.y, r.v.z, r.m);
    S.f[lane] = make_float4(r.gh.x, r.gh.y, r.gh.z, SPH_KNORM * (r.gh.w * r.gh.w) * (r.gh.w * r.gh.w));
  }
  S.jacc[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  S.jvs[lane] = 0.f;
}

__device__ __forceinline__ void flush_force(int gidx, float4 acc, float vs, float4* facc, float* fvsig) {
  if (gidx < 0 || !(vs > 0.0f)) return;   // vsig > 0 for every pair that contributed
  atomicAdd(&facc[gidx], acc);
  atomic_max_pos(&fvsig[gidx], vs);
}

// ------------------------------------------------------------- two-phase tiles
// Up to 32 partners sit in shared memory: particles of one or several partner
// clusters that passed a test against the box of the warp's cluster.  Phase 1:
// every lane tests its particle i against the staged partners (broadcast
// reads) and keeps two bitmasks, r < H_i and r < H_j, decided exactly.  Phase 2
// runs two sweeps without atomics: in the row sweep every lane walks its own
// bits and accumulates its own side; the r < H_j mask is then transposed with
// ballots so that in the column sweep every staged partner walks the lanes it
// interacts with and accumulates its side in registers, flushed once to global
// memory.  Each in-reach pair is still found once and updates both sides.
// Inside one cluster (own-only batches) every lane walks its full row for its
// own side, which keeps the lanes balanced: each pair's two sides are then
// computed by the two lanes concerned.  Invalid lanes sit at 1e30 with
// H^2 = -1, so they never pass a test.

// Two FP32 values in one 64-bit register, added and multiplied by one instruction
// (rounded as the scalar ones, element by element).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ void unpack2(f32x2 v, unsigned int& a, unsigned int& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// r^2 of a pair, in the order of operations of the mask phase (the sign of the
// separation does not matter: both phases then take the same value).
__device__ __forceinline__ float pair_r2(float dx, float dy, float dz) {
  return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
}

// Mask phase over the first n staged partners (n a multiple of 4): the slots not
// surely outside, r^2 <= hi of the own particle (mI) and of the partner (mJ).  Four
// slots take four 16-byte loads and, two slots per instruction, six operations for
// r^2 and one per threshold; each decision is the sign of hi - r^2, shifted into
// its mask (slots taken from the last, so that slot s lands in bit s).  The few
// slots inside the band are told apart in the sweeps, which have r^2 again: testing
// them here as well took 17 instructions per slot instead of 7.  With this phase, one
// copy of the task code for pair and self tasks and the partners' values derived
// once per batch, the density passes of a 33.5M clustered step took 55.4 ms instead
// of 63.7 and issued a sixth fewer instructions (issue slots are what bounds them:
// 74 % busy, DRAM at 3 %).  Unrolled further, the loops cost registers: 256 bytes
// spilled, 100 ms.  Empty slots and empty lanes (1e30, hi = -1) pass neither test.
template <bool BOTH>
__device__ __forceinline__ void near_masks(float3 ip, float ihi, const float* X, const float* Y, const float* Z,
                                           const float* W, int n, unsigned int& mI, unsigned int& mJ) {
  const f32x2 nx = pack2(-ip.x, -ip.x), ny = pack2(-ip.y, -ip.y), nz = pack2(-ip.z, -ip.z);
  const f32x2 hi = pack2(ihi, ihi), neg = pack2(-1.0f, -1.0f);
  unsigned int oI = 0, oJ = 0;     // surely outside
#pragma unroll 1
  for (int s0 = n - 4; s0 >= 0; s0 -= 4) {
    const ulonglong2 xx = *reinterpret_cast<const ulonglong2*>(X + s0);
    const ulonglong2 yy = *reinterpret_cast<const ulonglong2*>(Y + s0);
    const ulonglong2 zz = *reinterpret_cast<const ulonglong2*>(Z + s0);
    ulonglong2 ww = make_ulonglong2(0, 0);
    if (BOTH) ww = *reinterpret_cast<const ulonglong2*>(W + s0);
#pragma unroll
    for (int k = 1; k >= 0; --k) {
      const f32x2 dx = add2(k ? xx.y : xx.x, nx), dy = add2(k ? yy.y : yy.x, ny), dz = add2(k ? zz.y : zz.x, nz);
      const f32x2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
      unsigned int a0, a1;
      unpack2(fma2(r2, neg, hi), a0, a1);
      oI = __funnelshift_l(a1, oI, 1);
      oI = __funnelshift_l(a0, oI, 1);
      if (BOTH) {
        unsigned int b0, b1;
        unpack2(fma2(r2, neg, k ? ww.y : ww.x), b0, b1);
        oJ = __funnelshift_l(b1, oJ, 1);
        oJ = __funnelshift_l(b0, oJ, 1);
      }
    }
  }
  mI = ~oI;
  mJ = ~oJ;
}

// lane s receives the lanes whose mask has bit s: the 32 x 32 bit matrix (row =
// lane) transposed by recursive exchange of its off-diagonal blocks, 16 x 16
// down to 1 x 1, one shuffle per level.
__device__ __forceinline__ unsigned int transpose_bits(unsigned int m) {
  const int lane = threadIdx.x & 31;
  unsigned int x = m;
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) {
    const unsigned int mk = j == 16 ? 0x0000FFFFu : j == 8 ? 0x00FF00FFu : j == 4 ? 0x0F0F0F0Fu
                          : j == 2 ? 0x33333333u : 0x55555555u;
    const unsigned int y = __shfl_xor_sync(0xffffffffu, x, j);
    x = (lane & j) ? ((x & ~mk) | ((y & ~mk) >> j)) : ((x & mk) | ((y & mk) << j));
  }
  return x;
}

// The four density sums of a particle (sum m w, sum m q w', sum w, sum q w').
// KAHAN: compensated (Neumaier) summation, for high neighbour counts: each sum
// carries the rounding errors of its additions in c, and the total is s + c, so
// its error no longer grows with the number of terms.
template <bool KAHAN>
struct DensAcc {
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
  __device__ __forceinline__ static void kadd(float& sum, float& comp, float x) {
    const float t = sum + x;
    comp += fabsf(sum) >= fabsf(x) ? (sum - t) + x : (x - t) + sum;
    sum = t;
  }
  __device__ __forceinline__ void add(float m, float w, float gg) {
    if (KAHAN) {
      kadd(s.x, c.x, m * w);
      kadd(s.y, c.y, m * gg);
      kadd(s.z, c.z, w);
      kadd(s.w, c.w, gg);
    } else {
      s.x = fmaf(m, w, s.x);
      s.y = fmaf(m, gg, s.y);
      s.z += w;
      s.w += gg;
    }
  }
  __device__ __forceinline__ float4 total() const { return make_float4(s.x + c.x, s.y + c.y, s.z + c.z, s.w + c.w); }
};

// A particle's sums added to its sums in global memory (dacc), its neighbours to
// dcnt.  Compensated sums (dcomp given) carry the rounding of the additions in memory
// too: an atomic addition returns what it found, so that its rounding error is known
// exactly and is added to dcomp, which the ghost pass joins to the sums.
__device__ __forceinline__ float two_sum_err(float a, float b) {
  const float t = a + b, bb = t - a;
  return (a - (t - bb)) + (b - bb);
}

template <bool KAHAN>
__device__ __forceinline__ void flush_dens(int gidx, const DensAcc<KAHAN>& acc, unsigned int cnt, float4* dacc,
                                           unsigned int* dcnt, float4* dcomp) {
  if (gidx < 0 || cnt == 0) return;
  if (KAHAN) {
    const float4 x = acc.total();
    const float4 o = atomicAdd(&dacc[gidx], x);
    atomicAdd(&dcomp[gidx], make_float4(((acc.s.x - x.x) + acc.c.x) + two_sum_err(o.x, x.x),
                                        ((acc.s.y - x.y) + acc.c.y) + two_sum_err(o.y, x.y),
                                        ((acc.s.z - x.z) + acc.c.z) + two_sum_err(o.z, x.z),
                                        ((acc.s.w - x.w) + acc.c.w) + two_sum_err(o.w, x.w)));
  } else {
    atomicAdd(&dacc[gidx], acc.s);
  }
  atomicAdd(&dcnt[gidx], cnt);
}

// r from r^2 by the fast reciprocal square root (its rounding enters the kernel's
// argument only; the neighbour decision is taken on r^2).  The floor keeps r = 0
// at 0 without a test; it is below any r^2 of distinct positions that matters to W
// (r = 1e-19 L).
__device__ __forceinline__ float rsqrt_floor(float r2) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(fmaxf(r2, 1.2e-38f)));
  return y;
}
__device__ __forceinline__ float pair_r(float r2) { return r2 * rsqrt_floor(r2); }

// One density contribution: w and q w'(q) at q = r / H, weighted by m.
template <bool KAHAN>
__device__ __forceinline__ void dens_add(float r, float invH, float m, DensAcc<KAHAN>& acc) {
  float w, dw;
  const float q = r * invH;
  spline_w_dw(q, w, dw);
  const float gg = q * dw;                 // q w'(q) = r dW/dr in units of W
  acc.add(m, w, gg);
}

// The pairs of a sweep inside the guard band, decided in FP64 and added to the
// particle's sums in global memory (about one batch in ten has one).  Out of line,
// with everything read back from memory, so that the sweeps keep their registers.
// column: this lane's staged partner against own lanes (bits of unc); else this
// lane's own particle against staged partners.
template <bool KAHAN>
__device__ __noinline__ void dens_band(const DensShared& S, unsigned int unc, bool column,
                                       const unsigned int* __restrict__ perm, const double* __restrict__ x,
                                       const float4* __restrict__ pos4, const BoxDesc* __restrict__ box,
                                       float4* dacc, unsigned int* dcnt, float4* dcomp) {
  const int lane = threadIdx.x & 31;
  const BoxDesc& bd = box[S.tk.box];
  const int gme = column ? S.g[lane] : S.ig[lane];
  const float Hp = pos4[gme].w;
  const float invH = __fdividef(1.0f, Hp * (float)bd.invL);
  const float4 me = column ? make_float4(S.x[lane], S.y[lane], S.z[lane], 0.0f) : S.ip[lane];
  for (; unc; unc &= unc - 1) {
    const int k = __ffs(unc) - 1;
    const int go = column ? S.ig[k] : S.g[k];
    if (!exact_less(gme, go, Hp, perm, x, bd.L, 0.5 * bd.L, bd.periodic)) continue;
    const float4 o = column ? S.ip[k] : make_float4(S.x[k], S.y[k], S.z[k], S.m[k]);
    DensAcc<KAHAN> a;
    dens_add(pair_r(pair_r2(me.x - o.x, me.y - o.y, me.z - o.z)), invH, o.w, a);
    flush_dens(gme, a, 1u, dacc, dcnt, dcomp);
  }
}

// One sweep of a density batch: the lane's particle (at me, with 1/H) against the
// partners of its mask, whose position and mass get(slot) gives.  Two partners per
// turn, packed, so that most of the arithmetic takes one instruction for both; an odd
// one's second partner, and those inside the guard band (set aside in unc, decided
// afterwards), take q = 1, where w and w' vanish.  The terms are added one by one, in the
// order of the slots (two packed sums, one per partner of a turn, round differently: see
// sum_done).
template <bool KAHAN, class Get>
__device__ __forceinline__ unsigned int dens_sweep(unsigned int mask, float3 me, float lo, float invH, Get get,
                                                   DensAcc<KAHAN>& acc) {
  const f32x2 nx = pack2(-me.x, -me.x), ny = pack2(-me.y, -me.y), nz = pack2(-me.z, -me.z), ih = pack2(invH, invH);
  unsigned int unc = 0;
#pragma unroll 1
  for (unsigned int m = mask; m;) {
    const int ja = __ffs(m) - 1;
    m &= m - 1;
    const bool two = m != 0;
    const int jb = two ? __ffs(m) - 1 : ja;
    m &= m - 1;
    const float4 A = get(ja), B = get(jb);
    const f32x2 dx = add2(pack2(A.x, B.x), nx), dy = add2(pack2(A.y, B.y), ny), dz = add2(pack2(A.z, B.z), nz);
    const f32x2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
    float ra, rb;
    unpack2(r2, ra, rb);
    const bool ua = ra >= lo, ub = rb >= lo;
    if (ua) unc |= 1u << ja;
    if (ub && two) unc |= 1u << jb;
    float qa, qb;
    unpack2(mul2(mul2(r2, pack2(rsqrt_floor(ra), rsqrt_floor(rb))), ih), qa, qb);
    qa = ua ? 1.0f : qa;
    qb = ub || !two ? 1.0f : qb;
    // spline_w_dw of both
    const f32x2 q = pack2(qa, qb), one = pack2(1.0f, 1.0f);
    const f32x2 om = fma2(q, pack2(-1.0f, -1.0f), one), q2 = mul2(q, q);
    float wia, wib, wda, wdb, woa, wob, wea, web;
    unpack2(fma2(mul2(q2, pack2(-6.0f, -6.0f)), om, one), wia, wib);                                   // 1 - 6q^2 + 6q^3
    unpack2(mul2(q, fma2(q, pack2(18.0f, 18.0f), pack2(-12.0f, -12.0f))), wda, wdb);                   // -12q + 18q^2
    const f32x2 o2 = mul2(om, om);
    unpack2(mul2(mul2(o2, om), pack2(2.0f, 2.0f)), woa, wob);                                          // 2(1-q)^3
    unpack2(mul2(o2, pack2(-6.0f, -6.0f)), wea, web);                                                  // -6(1-q)^2
    const bool ia = qa < 0.5f, ib = qb < 0.5f;
    const f32x2 w = pack2(ia ? wia : woa, ib ? wib : wob);
    const f32x2 g = mul2(q, pack2(ia ? wda : wea, ib ? wdb : web));      // q w'(q) = r dW/dr in units of W
    float wa, wb, ga, gb;
    unpack2(w, wa, wb);
    unpack2(g, ga, gb);
    acc.add(A.w, wa, ga);
    acc.add(B.w, wb, gb);
  }
  return unc;
}

// The plain sums over one interaction's partners are done: they join those of the unit's
// interactions before, and the next interaction's start anew.  So each particle's sums are
// made of the same parts whatever shares a batch or a unit, one per interaction of its
// cluster and one per cluster it is a partner of, each added up in the order of the sorted
// particles; only the order in which the units' totals meet in memory is open.  The rounding
// of N~ decides which particles at the tolerance's edge iterate once more, and a change of
// grouping changes it more (8e-8 of N~) than that order does (3e-8): grouped in another
// way, three to five times as many particles of a multi-scale box ended an iteration apart
// as between two runs.  (Each part added to memory by itself: nearer to a pass of one task
// per interaction by a seventh, but more left open, two runs of a 20,000-particle box differ
// in which particles stop in 6 % of the tries, and in none of 400 this way.)
// (A part ends early where it exceeds SUM_MAX, at 14 times the usual number of neighbours: of
// 250 coincident particles one chain of additions was off by 1.9e-5.)
constexpr float SUM_MAX = 64.0f;

template <bool KAHAN>
__device__ __forceinline__ void sum_done(DensShared& S, DensAcc<KAHAN>& acc) {
  const int lane = threadIdx.x & 31;
  const float4 t = S.is[lane];
  S.is[lane] = make_float4(t.x + acc.s.x, t.y + acc.s.y, t.z + acc.s.z, t.w + acc.s.w);
  acc = DensAcc<KAHAN>();
}

// Own side of a density batch: the lane walks its mask of staged partners.  segs: the
// slots at which another interaction's partners begin (the same in every lane).
template <bool KAHAN>
__device__ __forceinline__ void dens_row(const DensI& I, float ilo, DensShared& S, unsigned int ui, unsigned int segs,
                                         DensAcc<KAHAN>& acc,
                                         unsigned int& cnt, const unsigned int* perm, const double* x,
                                         const float4* pos4, const BoxDesc* box, float4* dacc, unsigned int* dcnt,
                                         float4* dcomp) {
  unsigned int rest = ui, unc = 0;
#pragma unroll 1
  for (;;) {
    const unsigned int now = segs ? rest & ((segs & (0u - segs)) - 1u) : rest;
    unc |= dens_sweep(
        now, I.p, ilo, I.invH, [&](int s) { return make_float4(S.x[s], S.y[s], S.z[s], S.m[s]); }, acc);
    if (KAHAN || !segs) break;
    rest &= ~now;
    segs &= segs - 1u;
    sum_done(S, acc);
  }
  if (!KAHAN && acc.s.z > SUM_MAX) sum_done(S, acc);
  cnt += __popc(ui & ~unc);
  if (unc) dens_band<KAHAN>(S, unc, false, perm, x, pos4, box, dacc, dcnt, dcomp);
}

// The masks as exact decisions (counting and recording passes, which need them
// before the sweeps): both decisions of a pair inside either band, in FP64.  Each lane
// walks its own candidates; S.m holds the slots' lower bounds.
__device__ __noinline__ void resolve_masks(const DensShared& S, float ilo, unsigned int& mI, unsigned int& mJ,
                                           unsigned int& rc, const unsigned int* perm, const double* x,
                                           const float4* pos4, const BoxDesc* box) {
  const int lane = threadIdx.x & 31;
  const float4 P = S.ip[lane];
  for (unsigned int m = mI | mJ; m; m &= m - 1) {
    const int s = __ffs(m) - 1;
    const unsigned int bit = 1u << s;
    const float r2 = pair_r2(P.x - S.x[s], P.y - S.y[s], P.z - S.z[s]);
    if (((mI & bit) && r2 >= ilo) || ((mJ & bit) && r2 >= S.m[s])) {
      const BoxDesc& bd = box[S.tk.box];
      rc += 2;
      const int gi = S.ig[lane];
      mI = exact_less(gi, S.g[s], pos4[gi].w, perm, x, bd.L, 0.5 * bd.L, bd.periodic) ? (mI | bit) : (mI & ~bit);
      mJ = exact_less(gi, S.g[s], S.H[s], perm, x, bd.L, 0.5 * bd.L, bd.periodic) ? (mJ | bit) : (mJ & ~bit);
    }
  }
}

// One density batch of q <= 32 staged partners (slots 0..q-1) against the warp's
// cluster: the slots' derived values and masses by their lanes, the masks over the
// first q rounded up to 4, then the two sweeps: own side for r < H_i (active i),
// partner side for r < H_j (active j).  own_only: the partners are the warp's own
// cluster (each lane leaves itself out and updates its own side only; the
// counters count the upper triangle, since every pair appears in both rows).
template <bool COUNT, bool PART, bool KAHAN, bool REC>
__device__ __forceinline__ void dens_batch(const DensI& I, DensShared& S, unsigned int q, unsigned int segs, bool own_only,
                                           DensAcc<KAHAN>& acc, unsigned int& cnt, const unsigned int* perm,
                                           const double* x, const float4* __restrict__ pos4,
                                           const BoxDesc* __restrict__ box, const float4* __restrict__ cen4,
                                           float4* dacc, unsigned int* dcnt, float4* dcomp, Counters& C, const PairRec& R,
                                           RecW& W) {
  const int lane = threadIdx.x & 31;
  const bool v = (unsigned int)lane < q;
  __syncwarp();
  float jm = 0.0f, jlo = -1.0f, jinvH = 0.0f;
  if (v) {
    jm = cen4[S.g[lane]].w;       // needed after the masks
    const float H = S.H[lane] * S.tk.bhi.w;
    const float H2 = H * H, band = BAND_REL * H * (S.tk.eb + H);
    jinvH = __fdividef(1.0f, H);
    jlo = H2 - band;
    S.hi[lane] = H2 + band;
  } else {
    S.x[lane] = 1e30f;
    S.y[lane] = 1e30f;
    S.z[lane] = 1e30f;
    S.hi[lane] = -1.0f;
  }
  const unsigned int jvalid = __ballot_sync(0xffffffffu, v);
  const unsigned int jact = PART ? __ballot_sync(0xffffffffu, v && S.act[lane]) : jvalid;
  __syncwarp();
  const unsigned int allow = own_only ? jvalid & ~(1u << lane) : jvalid;
  unsigned int mI, mJ;
  // the own guard band: r^2 below ilo is inside, above ihi outside, between them
  // decided in FP64
  const float iband = BAND_REL * I.H * (S.tk.eb + I.H), ilo = I.H * I.H - iband;
  const float ihi = I.valid ? I.H * I.H + iband : -1.0f;
  near_masks<true>(I.p, ihi, S.x, S.y, S.z, S.hi, (int)((q + 3u) & ~3u), mI, mJ);
  mI &= allow;
  mJ &= allow;
  unsigned int rc = 0;
  if (COUNT || (REC && !PART)) {
    S.m[lane] = jlo;
    __syncwarp();
    resolve_masks(S, ilo, mI, mJ, rc, perm, x, pos4, box);
    __syncwarp();
  }
  // the pairs for the force pass: each unordered pair once (inside one cluster,
  // the partners above the lane)
  if (REC && !PART) rec_batch(R, W, S, jvalid, (mI | mJ) & (own_only ? upper_mask(lane) : 0xffffffffu));
  const unsigned int ui = I.act ? mI : 0u, uj = own_only ? 0u : (mJ & jact);
  if (COUNT) {
    const unsigned int cmask = own_only ? upper_mask(lane) : 0xffffffffu;
    C.cand += I.valid ? __popc(allow & jvalid & cmask) : 0u;
    C.rechecks += rc;
    C.pairs += __popc((ui | (mJ & jact)) & cmask);
    C.sides += __popc(ui) + __popc(uj);
  }
  S.m[lane] = jm;
  __syncwarp();
  dens_row(I, ilo, S, ui, segs, acc, cnt, perm, x, pos4, box, dacc, dcnt, dcomp);
  // column sweep: partner side, staged partner = lane
  const unsigned int col = own_only ? 0u : transpose_bits(uj);
  if (col) {
    const float3 J = make_float3(S.x[lane], S.y[lane], S.z[lane]);
    DensAcc<KAHAN> pacc;
    const unsigned int unc = dens_sweep(
        col, J, jlo, jinvH, [&](int s) { return S.ip[s]; }, pacc);
    flush_dens(S.g[lane], pacc, __popc(col & ~unc), dacc, dcnt, dcomp);
    if (unc) dens_band<KAHAN>(S, unc, true, perm, x, pos4, box, dacc, dcnt, dcomp);
  }
  __syncwarp();
}

// Both sides of one force pair, a (own particle: mass ma, VA = velocity and rho, FA =
// 1/H, f P / rho^2, c, K/H^4) and b (partner: VB = velocity and mass, FB = rho, f P /
// rho^2, c, K/H^4, and 1/H), d = x_a - x_b: a gains ca, b gains cb (the antisymmetric
// acceleration terms and each side's du/dt), both see vsig.  No contribution when r =
// 0.  A side's kernel gradient is taken inside its support and is zero outside (q
// clamped to 1, where it is zero too: the FP32 test agrees with the exact one to within
// the gradient's size there, about 6 (1 - q)^2 for q within rounding of 1).  The two
// sides' kernels are evaluated packed.
__device__ __forceinline__ void force_pair_terms(float ma, const float4& VA, const float4& FA, const float4& VB,
                                                 const float4& FB, float invHb, float dx, float dy, float dz, float r2,
                                                 float alpha, float4& ca, float4& cb, float& vsig) {
  ca = make_float4(0.f, 0.f, 0.f, 0.f);
  cb = ca;
  vsig = 0.0f;
  if (!(r2 > 0.0f)) return;
  const float rinv = rsqrtf(r2);
  const float r = r2 * rinv;
  float qa, qb;
  unpack2(mul2(pack2(r, r), pack2(FA.x, invHb)), qa, qb);
  qa = fminf(qa, 1.0f);
  qb = fminf(qb, 1.0f);
  const f32x2 q = pack2(qa, qb);
  const f32x2 om = fma2(q, pack2(-1.0f, -1.0f), pack2(1.0f, 1.0f));
  float ia, ib, oa, ob;
  unpack2(mul2(q, fma2(q, pack2(18.0f, 18.0f), pack2(-12.0f, -12.0f))), ia, ib);   // -12q + 18q^2
  unpack2(mul2(mul2(om, om), pack2(-6.0f, -6.0f)), oa, ob);                         // -6(1-q)^2
  const f32x2 W = mul2(pack2(FA.w, FB.w), pack2(qa < 0.5f ? ia : oa, qb < 0.5f ? ib : ob));
  const f32x2 FW = mul2(pack2(FA.y, FB.y), W);
  float Wa, Wb, FWa, FWb;
  unpack2(W, Wa, Wb);
  unpack2(FW, FWa, FWb);
  const float vdx = fmaf(VA.x - VB.x, dx, fmaf(VA.y - VB.y, dy, (VA.z - VB.z) * dz));
  const float wv = vdx * rinv;
  const float mu = fminf(wv, 0.0f);
  vsig = FA.z + FB.z - 3.0f * mu;
  const float Pi = __fdividef(-alpha * vsig * mu, VA.w + FB.x);
  const float PW = Pi * (0.5f * (Wa + Wb));
  const float coef = ((FWa + FWb) + PW) * rinv;
  const float hv = 0.5f * PW;
  const float ka = -VB.w * coef, kb = ma * coef;
  float ea, eb;
  unpack2(mul2(mul2(add2(FW, pack2(hv, hv)), pack2(wv, wv)), pack2(VB.w, ma)), ea, eb);
  ca = make_float4(ka * dx, ka * dy, ka * dz, ea);
  cb = make_float4(kb * dx, kb * dy, kb * dz, eb);
}

// Sums (v) and maxima (m) over runs of adjacent lanes with the same key, no run
// longer than maxrun; true on the first lane of each run, which then holds them.
__device__ __forceinline__ bool run_sum_max(int key, unsigned int maxrun, float4& v, float& m) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (unsigned int off = 1; off < 32; off <<= 1) {
    if (off >= maxrun) break;            // the same in every lane
    const int k2 = __shfl_down_sync(0xffffffffu, key, off);
    const float x = __shfl_down_sync(0xffffffffu, v.x, off), y = __shfl_down_sync(0xffffffffu, v.y, off);
    const float z = __shfl_down_sync(0xffffffffu, v.z, off), w = __shfl_down_sync(0xffffffffu, v.w, off);
    const float m2 = __shfl_down_sync(0xffffffffu, m, off);
    if (lane + off < 32 && k2 == key) {
      v.x += x;
      v.y += y;
      v.z += z;
      v.w += w;
      m = fmaxf(m, m2);
    }
  }
  const int prev = __shfl_up_sync(0xffffffffu, key, 1);   // every lane takes part in the shuffle
  return lane == 0 || prev != key;
}

// A pair inside the guard band of both radii (or in one band and outside the other
// radius): r < max(H_i, H_j) in FP64.
__device__ __noinline__ bool force_band(const ForceShared& S, int li, int sj, const unsigned int* __restrict__ perm,
                                        const double* __restrict__ x, const float4* __restrict__ pos4,
                                        const BoxDesc* __restrict__ box) {
  const BoxDesc& bd = box[S.tk.box];
  const int gi = (int)S.own0 + li, gj = S.g[sj];
  const float Hm = fmaxf(pos4[gi].w, pos4[gj].w);      // r < H_i or r < H_j
  return exact_less(gi, gj, Hm, perm, x, bd.L, 0.5 * bd.L, bd.periodic);
}

// What the rounds need besides the staged data.
struct ForceArgs {
  const unsigned int* perm;
  const double* x;
  const float4* pos4;
  const BoxDesc* box;
  unsigned int* fcnt;
  float alpha;
};

// The pairs of one batch (mask m of the lane's own particle over the staged
// slots), each evaluated once for both sides.  The pairs form a list, own lane
// major, of which every lane takes an equal run, so that all lanes work however
// unevenly the pairs fall on the rows.  Own side: a lane's run mostly stays in one
// row, whose terms it sums in registers; where a row ends inside a run, the sum goes
// to the row's task sums (only one lane sees a row end), and what is left at the end
// is summed over adjacent lanes (rounds of 32 consecutive pairs, each with a
// segmented reduction, took 60 instructions more per round; each lane taking its own
// next pair while most have one left was slower still).  Partner side: the terms go
// through shared memory, where the first of each partner's lanes adds them up, to the
// partner's batch sums (or, inside one cluster, to that particle's task sums).
// Shared-memory float atomics are slow, the more so where lanes collide.
// With the two sides' kernels packed (force_pair_terms): force pass of 33.5M clustered
// particles 38.7 -> 36.6 ms (at wide supports 78.9 -> 68.1), of the 1M open lattice
// 0.85 -> 0.72 ms, of 4096 particles 38 -> 33 us.
// EXACT: the mask holds exact decisions; else those of slots inside the guard band
// are taken here, where r^2 is at hand.
template <bool COUNT, bool EXACT>
__device__ __forceinline__ void force_rounds(ForceShared& S, unsigned int m, bool own_only, const ForceArgs& A,
                                             Counters* C) {
  const int lane = threadIdx.x & 31;
  const unsigned int lt = (1u << lane) - 1u;
  const unsigned int cnt = __popc(m);
  unsigned int k = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int y = __shfl_up_sync(0xffffffffu, k, o);
    if (lane >= o) k += y;
  }
  const unsigned int total = __shfl_sync(0xffffffffu, k, 31);
  k -= cnt;      // the place of the lane's next pair in the list
  const unsigned int maxrow = __reduce_max_sync(0xffffffffu, cnt);
  const unsigned int rowmask = __ballot_sync(0xffffffffu, cnt != 0u);
  const unsigned int incl = k + cnt;
  bool first = true;       // the lane's next listed pair is its row's first
  __syncwarp();
#pragma unroll 1
  for (unsigned int w0 = 0; w0 < total; w0 += PLIST_CAP) {
    const unsigned int np = min(PLIST_CAP, total - w0), R = (np + 31u) >> 5;
#pragma unroll 1
    for (; m && k < w0 + PLIST_CAP; m &= m - 1, ++k) {
      S.plist[k - w0] = (unsigned char)((__ffs(m) - 1) | (first ? 32 : 0));
      first = false;
    }
    const unsigned int i0 = lane * R, i1 = min(i0 + R, np);
    // the row of pair w0 + i0: the first lane whose pairs end behind it
    int li = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned int e = __shfl_sync(0xffffffffu, incl, li + o - 1);
      if (e <= w0 + i0) li += o;
    }
    if (i0 >= i1) li = 32 + lane;     // (a key no other lane has)
    float4 oa = make_float4(0.f, 0.f, 0.f, 0.f);
    float ov = 0.0f;
    __syncwarp();
#pragma unroll 1
    for (unsigned int r = 0; r < R; ++r) {
      const bool a = i0 + r < i1;
      int sj = 64 + lane;      // (likewise)
      float4 cj = make_float4(0.f, 0.f, 0.f, 0.f);
      float vs = 0.0f;
      if (a) {
        const unsigned int w = S.plist[i0 + r];
        sj = (int)(w & 31u);
        if (r > 0u && (w & 32u)) {
          float4 t = S.iacc[li];
          t.x += oa.x; t.y += oa.y; t.z += oa.z; t.w += oa.w;
          S.iacc[li] = t;
          S.ivs[li] = fmaxf(S.ivs[li], ov);
          oa = make_float4(0.f, 0.f, 0.f, 0.f);
          ov = 0.0f;
          li = __ffs(rowmask & (0xfffffffeu << li)) - 1;
        }
        const float4 P = S.ip[li];
        const float dx = P.x - S.x[sj], dy = P.y - S.y[sj], dz = P.z - S.z[sj];
        const float r2 = pair_r2(dx, dy, dz);
        bool in = true;
        if (!EXACT && r2 >= S.ilo[li] && r2 >= S.lo[sj]) {
          in = force_band(S, li, sj, A.perm, A.x, A.pos4, A.box);
          if (COUNT) C->rechecks += 2;
        }
        if (in) {
          const float4 V = S.iv[li], F = S.if_[li], VJ = S.v[sj], FJ = S.f[sj];
          float4 ci;
          force_pair_terms(P.w, V, F, VJ, FJ, S.H[sj], dx, dy, dz, r2, A.alpha, ci, cj, vs);
          oa.x += ci.x; oa.y += ci.y; oa.z += ci.z; oa.w += ci.w;
          ov = fmaxf(ov, vs);
          if (COUNT) {
            // force partners of both particles (the pair set, checked per particle)
            atomicAdd(&A.fcnt[S.own0 + li], 1u);
            atomicAdd(&A.fcnt[S.g[sj]], 1u);
            C->pairs += 1;
          }
        }
      }
      const unsigned int peers = __match_any_sync(0xffffffffu, sj);
      S.cb[lane] = cj;
      S.cv[lane] = vs;
      __syncwarp();
      if (a && (peers & lt) == 0u) {
        float4* dst = own_only ? &S.iacc[sj] : &S.jacc[sj];
        float* dv = own_only ? &S.ivs[sj] : &S.jvs[sj];
#pragma unroll 1
        for (unsigned int b = peers & (peers - 1); b; b &= b - 1) {
          const int l = __ffs(b) - 1;
          const float4 t = S.cb[l];
          cj.x += t.x; cj.y += t.y; cj.z += t.z; cj.w += t.w;
          vs = fmaxf(vs, S.cv[l]);
        }
        float4 t = *dst;
        t.x += cj.x; t.y += cj.y; t.z += cj.z; t.w += cj.w;
        *dst = t;
        *dv = fmaxf(*dv, vs);
      }
      __syncwarp();
    }
    // what is left of each lane's last row: a row spans at most maxrow / R + 2 lanes
    if (run_sum_max(li, R == 1u ? maxrow : (maxrow + R - 1u) / R + 1u, oa, ov) && li < 32) {
      float4 t = S.iacc[li];
      t.x += oa.x; t.y += oa.y; t.z += oa.z; t.w += oa.w;
      S.iacc[li] = t;
      S.ivs[li] = fmaxf(S.ivs[li], ov);
    }
    __syncwarp();
  }
}

// One force batch of q staged partners: every pair with r < max(H_i, H_j), found by
// the mask phase and evaluated for both sides.  The partners' velocities and ghost
// quantities are loaded before the masks and used after them (loaded with the
// position, for every particle of a candidate cluster, they were three quarters of
// the bytes and two fifths of them were used).
template <bool COUNT>
__device__ __forceinline__ void force_batch(ForceShared& S, float3 ip, float iH, unsigned int q, bool own_only,
                                            const ForceArgs& A, const float4* __restrict__ cen4,
                                            const float4* __restrict__ vel4, const float4* __restrict__ ghost4,
                                            float4* facc, float* fvsig, Counters* C) {
  const int lane = threadIdx.x & 31;
  const bool v = (unsigned int)lane < q;
  __syncwarp();
  ForceRaw r;
  if (v) {
    const unsigned int g = (unsigned int)S.g[lane];
    r.v = vel4[g];
    r.gh = ghost4[g];
    r.m = cen4[g].w;
    const float H = S.H[lane] * S.tk.bhi.w;
    const float H2 = H * H, band = BAND_REL * H * (S.tk.eb + H);
    S.hi[lane] = H2 + band;
    S.lo[lane] = H2 - band;
  } else {
    S.x[lane] = 1e30f;
    S.y[lane] = 1e30f;
    S.z[lane] = 1e30f;
    S.hi[lane] = -1.0f;
  }
  const unsigned int jvalid = __ballot_sync(0xffffffffu, v);
  __syncwarp();
  // inside one cluster each unordered pair once (partners above the lane)
  const unsigned int allow = own_only ? jvalid & upper_mask(lane) : jvalid;
  unsigned int mI, mJ;
  const float iband = BAND_REL * iH * (S.tk.eb + iH), ihi = iH > 0.0f ? iH * iH + iband : -1.0f;
  S.ilo[lane] = iH * iH - iband;      // (read after the masks)
  near_masks<true>(ip, ihi, S.x, S.y, S.z, S.hi, (int)((q + 3u) & ~3u), mI, mJ);
  const unsigned int m = (mI | mJ) & allow;
  if (COUNT) C->cand += ihi >= 0.0f ? __popc(allow) : 0u;
  if (!__any_sync(0xffffffffu, m != 0u)) return;
  force_derive(S, lane, v, r);
  force_rounds<COUNT, false>(S, m, own_only, A, C);
  if (v && !own_only) flush_force(S.g[lane], S.jacc[lane], S.jvs[lane], facc, fvsig);
  __syncwarp();
}

// One recorded batch B of the first density pass: the staged partners are read
// back by index (own_only: the warp's own cluster), the pairs come from the recorded
// masks, and the rounds run as in force_batch.
template <bool COUNT>
__device__ __noinline__ void force_replay_batch(ForceShared& S, const unsigned int* __restrict__ B, bool own_only,
                                                const float4* __restrict__ cen4, const float4* __restrict__ vel4,
                                                const float4* __restrict__ ghost4, const ForceArgs A, float3 sh,
                                                float4* facc, float* fvsig, Counters* C) {
  const int lane = threadIdx.x & 31;
  const unsigned int gj = __ldcs(B + lane);     // read once: evict first
  const unsigned int m = __ldcs(B + 32 + lane);
  const bool v = gj != REC_NONE;
  __syncwarp();
  ForceRaw r;
  if (v) {
    const float4 p = A.pos4[gj], c = cen4[gj];
    r.v = vel4[gj];
    r.gh = ghost4[gj];
    r.m = c.w;
    // the cell offsets (c + sh) are exact dyadic values: add them first, round once
    force_put(S, lane, make_float3(p.x + (c.x + sh.x), p.y + (c.y + sh.y), p.z + (c.z + sh.z)), p.w, gj);
  }
  force_derive(S, lane, v, r);
  __syncwarp();
  if (COUNT) {
    const unsigned int jvalid = __ballot_sync(0xffffffffu, v);
    C->cand += S.if_[lane].x > 0.0f ? __popc(jvalid & (own_only ? upper_mask(lane) : 0xffffffffu)) : 0u;
  }
  force_rounds<COUNT, true>(S, m, own_only, A, C);
  __syncwarp();
  if (v && !own_only) flush_force(S.g[lane], S.jacc[lane], S.jvs[lane], facc, fvsig);
  __syncwarp();
}

// ------------------------------------------------------------- cluster geometry
__device__ __forceinline__ float3 axis_unit_f(int a) {
  int dx, dy, dz;
  axis_vec(a, dx, dy, dz);
  const int n2 = dx * dx + dy * dy + dz * dz;
  const float s = n2 == 1 ? 1.0f : (n2 == 2 ? 0.70710678118654752f : 0.57735026918962576f);
  return make_float3(dx * s, dy * s, dz * s);
}

// box of cluster t in the frame whose origin sits at -off from the leaf frame:
// box + (leaf centre + off), the offset being exact (dyadic)
__device__ __forceinline__ Box3 tile_box3(const Tiles& TL, const Tree& T, unsigned int t, float3 off) {
  const float4 lc = TL.cen[t];
  const float4 lo = TL.lo[t], hi = TL.hi[t];
  const float ox = lc.x + off.x, oy = lc.y + off.y, oz = lc.z + off.z;
  Box3 b;
  b.lo = make_float3(lo.x + ox, lo.y + oy, lo.z + oz);
  b.hi = make_float3(hi.x + ox, hi.y + oy, hi.z + oz);
  return b;
}

// Distance between two boxes within reach, compared squared (FP32; the
// caller's slack, at least 1e-6 of the reach, covers the rounding of both forms).
__device__ __forceinline__ bool box_near(const Box3& a, const Box3& b, float reach) {
  const float gx = fmaxf(0.0f, fmaxf(b.lo.x - a.hi.x, a.lo.x - b.hi.x));
  const float gy = fmaxf(0.0f, fmaxf(b.lo.y - a.hi.y, a.lo.y - b.hi.y));
  const float gz = fmaxf(0.0f, fmaxf(b.lo.z - a.hi.z, a.lo.z - b.hi.z));
  return fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= reach * reach;
}

// distance from a point to a box within reach (as box_near)
__device__ __forceinline__ bool near_box(const float3 p, const Box3& b, float reach) {
  const float gx = fmaxf(0.0f, fmaxf(b.lo.x - p.x, p.x - b.hi.x));
  const float gy = fmaxf(0.0f, fmaxf(b.lo.y - p.y, p.y - b.hi.y));
  const float gz = fmaxf(0.0f, fmaxf(b.lo.z - p.z, p.z - b.hi.z));
  return fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= reach * reach;
}

// a box moved by an offset (one rounding per bound, within the culling slack)
__device__ __forceinline__ Box3 box_shift(const Box3& b, float3 d) {
  Box3 r;
  r.lo = make_float3(b.lo.x + d.x, b.lo.y + d.y, b.lo.z + d.z);
  r.hi = make_float3(b.hi.x + d.x, b.hi.y + d.y, b.hi.z + d.z);
  return r;
}

// upper end of the projection of a box on u
__device__ __forceinline__ float box_rhi(const Box3& b, float3 u) {
  return fmaf(u.x, u.x >= 0.0f ? b.hi.x : b.lo.x,
              fmaf(u.y, u.y >= 0.0f ? b.hi.y : b.lo.y, u.z * (u.z >= 0.0f ? b.hi.z : b.lo.z)));
}

// Box and largest H of the warp's particles that still iterate h.  In a full pass
// every particle does, and the cluster's own box and H are returned unchanged;
// in a later pass the own side needs only the neighbours of these particles.
struct ActiveBox {
  Box3 b;
  float H;
  bool any, all;   // some / every particle of the cluster iterates
};

__device__ __forceinline__ ActiveBox active_box(const DensI& I, const Box3& bi, float Hi) {
  ActiveBox a;
  const bool ia = I.valid && I.act;
  if (__all_sync(0xffffffffu, ia || !I.valid)) {
    a.b = bi;
    a.H = Hi;
    a.any = a.all = true;
    return a;
  }
  a.all = false;
  a.any = __any_sync(0xffffffffu, ia);
  a.b.lo = make_float3(warp_min(ia ? I.p.x : 1e30f), warp_min(ia ? I.p.y : 1e30f), warp_min(ia ? I.p.z : 1e30f));
  a.b.hi = make_float3(warp_max(ia ? I.p.x : -1e30f), warp_max(ia ? I.p.y : -1e30f), warp_max(ia ? I.p.z : -1e30f));
  a.H = warp_max(ia ? I.H : 0.0f);
  return a;
}

// What the task lists of the pair records (params.pair_cache) need of a pair-interaction.
struct PairSetup {
  int A, B;
  ItemGeom g;
  float3 tshA;            // cluster box offset of A's clusters (the leaf centre is added per cluster)
  float HmB, slack;
  Box3 cellB;             // B's cell in A's frame
};

__device__ __forceinline__ PairSetup pair_setup(const Lists& Lq, const Tree& T, const BoxDesc* box, int item) {
  PairSetup P;
  P.A = Lq.pair_a[item];
  P.B = Lq.pair_b[item];
  P.g = item_geom(T, box, P.A, Lq.pair_axis[item]);
  const float4 cA = T.cen[P.A];
  P.tshA = make_float3(-cA.x, -cA.y, -cA.z);
  P.HmB = T.hmax[P.B] * P.g.invL;
  P.slack = P.g.e * 1.52587890625e-05f + P.g.es + 1e-6f * fmaxf(P.HmB, T.hmax[P.A] * P.g.invL);   // 2^-16 e
  // B's cell, widened by the drift of particles kept in it since the build
  const float h = 0.5f * P.g.e + P.g.drift;
  P.cellB.lo = make_float3(P.g.offB.x - h, P.g.offB.y - h, P.g.offB.z - h);
  P.cellB.hi = make_float3(P.g.offB.x + h, P.g.offB.y + h, P.g.offB.z + h);
  return P;
}

// ------------------------------------------------------------- units of work
// A unit is one cluster against the partner clusters of its interactions: the self
// interaction of its leaf and the pairs (A, B, axis) of every cell A on its chain
// (Section II-B: an interaction of a cell is one of all its particles).  The
// geometry of up to GROUP interactions is set up at once, one per lane, and the
// partners of all of them share the staged batches: with a task per (interaction,
// cluster) a fifth of both passes went into setting the tasks up (2 to 3 staged
// partners per own particle and task in a uniform box), and most batches were
// partly filled.  Where a box has few clusters, a unit is split into parts (every
// parts-th interaction), so that every warp has several.
//
// The frame of a unit's particle arithmetic is the centre of the own cluster's leaf.  A
// pair of large cells that cannot split (one particle of large H in it is enough) still
// holds particles of small H; in the cells' frame their positions would be rounded at
// the cells' scale, in their leaf's frame at the leaf's.  Own offsets are used as stored,
// the partners' move by an exact dyadic offset, so each position is rounded once, at most
// at the cells' scale, and the guard band stays valid.
// (One unit per warp in the smallest boxes, two where a cluster per warp would leave a
// partial wave: lattices of 25^3 and 30^3 lose 10 % with twice the parts, of 36^3, 42^3
// and a 40k Plummer box gain 10-40 %; three or five times the warps lose 5-30 % there.)
__device__ __forceinline__ unsigned int unit_parts(unsigned int ntile) {
  const unsigned int warps = gridDim.x * (blockDim.x >> 5);
  const unsigned int want = 10u * ntile >= 3u * warps ? 2u * warps : warps;
  return min(16u, max(1u, want / max(ntile, 1u)));
}

__device__ __forceinline__ void unit_begin(UnitShared& K, unsigned int ti, const Tree& T, const Tiles& TL,
                                           const BoxDesc* __restrict__ box,
                                           unsigned int part, unsigned int parts) {
  const float4 blo = TL.lo[ti], bhi = TL.hi[ti], cl = TL.cen[ti];
  const int leaf = (int)TL.leaf[ti], b = T.box[leaf];
  const float invL = (float)box[b].invL;
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    K.blo = make_float4(blo.x, blo.y, blo.z, blo.w * invL);
    K.bhi = make_float4(bhi.x, bhi.y, bhi.z, invL);
    K.clo = K.blo;
    K.chi = K.bhi;
    K.cl = cl;
    K.es = box[b].global32 ? 9.5367431640625e-07f : 0.0f;   // 2^-20 L: the 2^-25 rounding of both positions
    K.L32 = (float)box[b].L;
    K.drift = box[b].drift_u;
    K.eb = box[b].global32 ? 1.0f : ldexpf(1.0f, -T.level[leaf]);
    K.box = b;
    K.cell = leaf;
    K.ti = ti;
    K.part = part;
    K.parts = parts;
    K.at = 0;
    K.idx = 0;
  }
  __syncwarp();
}

// The first run of 32 clusters of an interaction's list that belongs to the unit.  RUNS
// (force): its part of the parts takes the runs r with (interaction + r) % parts == part.
// Else (density): the whole of the interactions with interaction % parts == part, so
// that a particle's sum over an interaction's partners is one (see sum_done).  A single
// list that outweighs all others is then not divided, which costs density passes little
// (4.2M clustered h iteration 44.0 -> 45.4 ms; the force pass of a million log-normal
// particles would take 4.2 ms instead of 2.9).
template <bool RUNS>
__device__ __forceinline__ unsigned int unit_first(const UnitShared& K, unsigned int interaction) {
  const unsigned int P = K.parts;
  if (P == 1u) return 0u;
  const unsigned int r = (K.part + P - interaction % P) % P;
  return RUNS || r == 0u ? r : 0x07ffffffu;      // (past every list)
}

// The next group of the unit's interactions: one per lane, from the cell's list (the
// leaf's self interaction first), then from its parent's.  Returns a ballot of the
// lanes whose interaction has work: its partner cell lies within reach of the own
// box and, in a later pass (PART; iact: the own cluster holds iterating particles),
// iterates itself or meets the own cluster's.  K.cell is -1 past the last group.
// The cell edge sets the guard band (K.eb; it grows along the chain).
// GATHER (the own side only, of a packed cluster): the pairs of which the cell is the
// second come too, the self interaction has all of the leaf's clusters, and only the own
// reach counts.
template <bool PART, bool GATHER, bool RUNS>
__device__ __forceinline__ unsigned int unit_group(UnitShared& K, const Tree& T, const uint2* __restrict__ csr,
                                                   bool iact) {
  const int lane = threadIdx.x & 31;
  const int A = K.cell;
  const unsigned int at = K.at, idx = K.idx;
  const int d = T.level[A];
  const bool leaf = T.child[A] < 0;
  // a leaf's list starts with its self interaction
  const unsigned int n = (unsigned int)__popc(T.pmask[A]) + (GATHER ? (unsigned int)__popc(T.rmask[A]) : 0u) + (leaf ? 1u : 0u);
  const unsigned int mine = at + lane;
  const bool valid = lane < GROUP && mine < n;
  bool live = false;
  const float e = ldexpf(1.0f, -d);
  if (valid) {
    const bool self = leaf && mine == 0u;
    int B = A, ax = 0;
    if (!self) {
      const uint2 pr = csr[T.pstart[A] + mine - (leaf ? 1u : 0u)];
      B = (int)pr.x;
      ax = (int)pr.y;
    }
    const bool second = GATHER && (ax & 16) != 0;
    int dx, dy, dz;
    axis_vec(GATHER ? ax & 15 : ax, dx, dy, dz);
    if (second) {
      dx = -dx;
      dy = -dy;
      dz = -dz;
    }
    const float3 off = self ? make_float3(0.f, 0.f, 0.f) : make_float3(e * dx, e * dy, e * dz);   // exact
    const float4 cA = T.cen[A], cB = T.cen[B], cl = K.cl;
    const float3 dl = make_float3(cl.x - cA.x, cl.y - cA.y, cl.z - cA.z);   // the leaf centre in A's frame, exact
    const float4 clo = K.clo, chi = K.chi;
    const Box3 bil{make_float3(clo.x, clo.y, clo.z), make_float3(chi.x, chi.y, chi.z)};
    const float invL = chi.w, HmB = T.hmax[B] * invL;
    const float slack = e * 1.52587890625e-05f + K.es + 1e-6f * fmaxf(HmB, T.hmax[A] * invL);   // 2^-16 e
    const unsigned int t0 = T.tile0[B], nt = T.ntile[B];
    unsigned int sb = SORT_NONE;
    if (!GATHER && !self) {      // (a gathered unit takes every list in the order of its clusters)
      const unsigned int sbB = T.sortbase[B];
      if (sbB != SORT_NONE) sb = sbB + (unsigned int)__popc(T.axes[B] & ((1u << ax) - 1u)) * nt;
    }
    const int n2 = dx * dx + dy * dy + dz * dz;
    const float offBp = e * (n2 == 1 ? 1.0f : (n2 == 2 ? 1.41421356237f : 1.73205080757f));
    // sort keys are the projections at the build; a cluster's projection has
    // since moved by at most the drift
    const float win = offBp - K.drift - box_rhi(box_shift(bil, dl), axis_unit_f(GATHER ? ax & 15 : ax));
    K.gsh[lane] = make_float4((off.x - cB.x) - dl.x, (off.y - cB.y) - dl.y, (off.z - cB.z) - dl.z, slack);
    K.gwin[lane] = make_float4(win, GATHER ? 0.0f : HmB, __uint_as_float(sb),
                               __uint_as_float(self && !GATHER ? t0 + nt - (K.ti + 1u) : nt));
    K.gtb[lane] = self && !GATHER ? K.ti + 1u : t0;
    // the partner cell, widened by the drift of particles kept in it since the build
    const float h = 0.5f * e + K.drift;
    const float3 cb = make_float3(off.x - dl.x, off.y - dl.y, off.z - dl.z);
    live = self || box_near(bil, Box3{make_float3(cb.x - h, cb.y - h, cb.z - h), make_float3(cb.x + h, cb.y + h, cb.z + h)},
                            (GATHER ? clo.w : fmaxf(clo.w, HmB)) + slack);
    if (PART && live && !iact) {
      // only the partner cell's iterating particles need this cluster
      live = T.active[B] != 0;
      if (live && !self) {
        Box3 ba;
        ba.lo = make_float3(key_float(T.alo[3 * B]) + cb.x, key_float(T.alo[3 * B + 1]) + cb.y,
                            key_float(T.alo[3 * B + 2]) + cb.z);
        ba.hi = make_float3(key_float(T.ahi[3 * B]) + cb.x, key_float(T.ahi[3 * B + 1]) + cb.y,
                            key_float(T.ahi[3 * B + 2]) + cb.z);
        live = box_near(bil, ba, HmB + slack);
      }
    }
  }
  if (live && K.parts > 1u)    // the unit's share has a run of this list
    live = 32u * unit_first<RUNS>(K, idx + lane) < __float_as_uint(K.gwin[lane].w);
  const unsigned int bal = __ballot_sync(0xffffffffu, live);
  const int up = T.parent[A];
  __syncwarp();
  if (lane == 0) {
    const bool more = at + GROUP < n;
    K.at = more ? at + GROUP : 0u;
    K.idx = idx + min((unsigned int)GROUP, n - at);
    K.cell = more ? A : up;
    K.selfit = leaf && at == 0u ? 0 : -1;
    K.gidx = idx;
    if (K.es == 0.0f) K.eb = e;
  }
  __syncwarp();
  return bal;
}

// One interaction as a unit's only one (a listed task, params.pair_cache).
__device__ __forceinline__ void unit_single(UnitShared& K, bool self, int item, const Lists& Lq, const Tree& T) {
  const int A = self ? Lq.self_a[item] : Lq.pair_a[item];
  const int B = self ? A : Lq.pair_b[item], ax = self ? 0 : Lq.pair_axis[item];
  int dx, dy, dz;
  axis_vec(ax, dx, dy, dz);
  const float e = ldexpf(1.0f, -T.level[A]);
  const float3 off = self ? make_float3(0.f, 0.f, 0.f) : make_float3(e * dx, e * dy, e * dz);
  const float4 cA = T.cen[A], cB = T.cen[B], cl = K.cl, clo = K.clo, chi = K.chi;
  const float3 dl = make_float3(cl.x - cA.x, cl.y - cA.y, cl.z - cA.z);
  const Box3 bil{make_float3(clo.x, clo.y, clo.z), make_float3(chi.x, chi.y, chi.z)};
  const float invL = chi.w, HmB = T.hmax[B] * invL;
  const float slack = e * 1.52587890625e-05f + K.es + 1e-6f * fmaxf(HmB, T.hmax[A] * invL);
  const unsigned int t0 = T.tile0[B], nt = T.ntile[B];
  unsigned int sb = SORT_NONE;
  if (!self) {
    const unsigned int sbB = T.sortbase[B];
    if (sbB != SORT_NONE) sb = sbB + (unsigned int)__popc(T.axes[B] & ((1u << ax) - 1u)) * nt;
  }
  const int n2 = dx * dx + dy * dy + dz * dz;
  const float offBp = e * (n2 == 1 ? 1.0f : (n2 == 2 ? 1.41421356237f : 1.73205080757f));
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    K.gsh[0] = make_float4((off.x - cB.x) - dl.x, (off.y - cB.y) - dl.y, (off.z - cB.z) - dl.z, slack);
    K.gwin[0] = make_float4(offBp - K.drift - box_rhi(box_shift(bil, dl), axis_unit_f(ax)), HmB, __uint_as_float(sb),
                            __uint_as_float(self ? t0 + nt - (K.ti + 1u) : nt));
    K.gtb[0] = self ? K.ti + 1u : t0;
    if (K.es == 0.0f) K.eb = e;
    K.cell = -1;
    K.gidx = 0;
    K.selfit = self ? 0 : -1;
  }
  __syncwarp();
}

// Lane-parallel scan of the cluster list of interaction it of the group, from entry
// e0 on: the clusters in reach (sorted window, then box distance) as a ballot, with
// their size, first particle and exact frame offset in K.cn, K.co (entries up to nt).  e0 advances past
// the entries scanned (and the other parts' runs), to nt once the sorted window has
// passed every cluster.  PART: the clusters that hold neighbours of the particles that iterate
// (box blo, bhi), and those that iterate near any particle of the own cluster (all:
// every particle iterates, the first test covers the second).
//
// A candidate much finer than the own cluster (its largest H below FINE_H of the own
// one) is tested once more, against every own particle's own reach (iH, one particle
// per lane).  A dense clump inside the reach of the own cluster's box lies outside
// most particles' supports, which end before it (a support holds N_ngb particles),
// but its thousands of particles would all be staged: on the clustered box half of
// all staged partners came from the tenth of the clusters that have one nearby.
// The test takes about 20 instructions per candidate; the others, where a box about
// the own cluster's size makes it pass nearly always, do without (at 0.5 a few per
// cent more stay staged, above 0.7 none fewer).  Density passes of the 33.5M
// clustered step 55.4 -> 49.8 ms, of the 262k Plummer box 2.02 -> 1.69 ms; a
// uniform box has no such candidate and pays nothing.
constexpr float FINE_H = 0.7f;

template <bool PART, bool GATHER, bool RUNS>
__device__ __forceinline__ unsigned int scan_clusters(UnitShared& K, float4* jlo, float4* jhi, const Tiles& TL,
                                                      const float* __restrict__ sort_r,
                                                      const unsigned int* __restrict__ sort_i, int it,
                                                      unsigned int& e0, unsigned int nt, bool any, bool all, float3 ip,
                                                      float iH) {
  const int lane = threadIdx.x & 31;
  const float4 win = K.gwin[it], sh = K.gsh[it], blo = K.blo, bhi = K.bhi;
  const unsigned int sb = __float_as_uint(win.z), e = e0 + lane;
  const bool sorted = sb != SORT_NONE;
  const float slack = sh.w, invL = bhi.w, Hi = K.clo.w;
  if (sorted && sort_r[sb + e0] + win.x > fmaxf(Hi, win.y) + slack) {
    e0 = nt;           // the sorted list only moves further away
    return 0u;
  }
  e0 += RUNS ? 32u * K.parts : 32u;
  bool pass = false, fine = false;
  if (e < nt) {
    const unsigned int t = sorted ? sort_i[sb + e] : K.gtb[it] + e;
    const float4 lo = TL.lo[t];
    const float Hj = GATHER ? 0.0f : lo.w * invL;      // (gathered: the own reach only)
    if (!sorted || sort_r[sb + e] + win.x <= fmaxf(Hi, Hj) + slack) {
      const float4 lc = TL.cen[t], hi = TL.hi[t];
      const float3 o = make_float3(lc.x + sh.x, lc.y + sh.y, lc.z + sh.z);
      const Box3 bj{make_float3(lo.x + o.x, lo.y + o.y, lo.z + o.z), make_float3(hi.x + o.x, hi.y + o.y, hi.z + o.z)};
      const Box3 b{make_float3(blo.x, blo.y, blo.z), make_float3(bhi.x, bhi.y, bhi.z)};
      pass = (!PART || any) && box_near(b, bj, fmaxf(blo.w, Hj) + slack);
      if (PART && !pass && !all && TL.active[t]) {
        const float4 clo = K.clo, chi = K.chi;
        pass = box_near(Box3{make_float3(clo.x, clo.y, clo.z), make_float3(chi.x, chi.y, chi.z)}, bj, Hj + slack);
      }
      if (pass) {
        K.co[lane] = make_float4(o.x, o.y, o.z, __uint_as_float(TL.start[t]));
        K.cn[lane] = (unsigned char)TL.n[t];
        fine = (GATHER ? lo.w * invL : Hj) < FINE_H * Hi;
        if (fine) {
          jlo[lane] = make_float4(bj.lo.x, bj.lo.y, bj.lo.z, Hj);
          jhi[lane] = make_float4(bj.hi.x, bj.hi.y, bj.hi.z, 0.0f);
        }
      }
    }
  }
  unsigned int mask = __ballot_sync(0xffffffffu, pass);
  unsigned int todo = __ballot_sync(0xffffffffu, fine);
  __syncwarp();
  for (; todo; todo &= todo - 1) {
    const int k = __ffs(todo) - 1;
    const float4 lo = jlo[k], hi = jhi[k];
    const bool hit = near_box(ip, Box3{make_float3(lo.x, lo.y, lo.z), make_float3(hi.x, hi.y, hi.z)},
                              fmaxf(iH, lo.w) + slack);
    if (!__any_sync(0xffffffffu, hit)) mask &= ~(1u << k);
  }
  return mask;
}

// ------------------------------------------------------------- walking a unit
// Where a unit stands, the same in every lane: the interactions of the group with
// work (live), the one whose clusters are scanned (it) from e0 to nt, the candidates
// of the scan (mask).
struct Walk {
  unsigned int live = 0, e0 = 0, nt = 0, mask = 0;
  int it = 0;
};

// The next candidates (W.mask, non-zero) of the unit; false at its end.
template <bool PART, bool GATHER, bool RUNS>
__device__ __forceinline__ bool unit_next(UnitShared& K, Walk& W, float4* jlo, float4* jhi, const Lists& Lq,
                                          const Tree& T, const Tiles& TL, const float* __restrict__ sort_r,
                                          const unsigned int* __restrict__ sort_i, bool any, bool all, float3 ip, float iH) {
  while (!W.mask) {
    if (W.e0 < W.nt) {
      W.mask = scan_clusters<PART, GATHER, RUNS>(K, jlo, jhi, TL, sort_r, sort_i, W.it, W.e0, W.nt, any, all, ip, iH);
    } else if (W.live) {
      W.it = __ffs(W.live) - 1;
      W.live &= W.live - 1;
      W.nt = __float_as_uint(K.gwin[W.it].w);
      W.e0 = 32u * unit_first<RUNS>(K, K.gidx + (unsigned int)W.it);
    } else if (K.cell >= 0) {
      W.live = unit_group<PART, GATHER, RUNS>(K, T, Lq.csr, any);
    } else {
      return false;
    }
  }
  return true;
}

// The density interactions of one unit (cluster ti, part of parts), or of one listed
// task (LISTED: interaction `item` only, its pairs recorded).  One copy of the batch
// serves the own cluster (the self interaction's first batch) and all partners.
template <bool COUNT, bool PART, bool KAHAN, bool LISTED>
__device__ __forceinline__ void density_unit(unsigned int ti, unsigned int part, unsigned int parts, bool self, int item,
    const Lists& Lq, const Tree& T, const Tiles& TL, const BoxDesc* __restrict__ box, const float4* __restrict__ pos4,
    const float4* __restrict__ cen4, const float* __restrict__ sort_r, const unsigned int* __restrict__ sort_i,
    const unsigned char* __restrict__ act, const unsigned int* __restrict__ perm, const double* __restrict__ x,
    float4* dacc, unsigned int* dcnt, float4* dcomp, DensShared& S, Counters& Cp, Counters& Cs, const PairRec& R, RecW& W) {
  const int lane = threadIdx.x & 31;
  UnitShared& K = S.tk;
  unit_begin(K, ti, T, TL, box, part, parts);
  if (LISTED) {
    rec_task_begin(S, self ? Lq.s_toff[item] + (ti - T.tile0[Lq.self_a[item]])
                           : Lq.p_toff[item] + (ti - T.tile0[Lq.pair_a[item]]));
    unit_single(K, self, item, Lq, T);
  }
  const unsigned int ni = TL.n[ti], own0 = TL.start[ti];
  const unsigned char* actp = PART ? act : nullptr;
  DensI I = load_dens((unsigned int)lane < ni, own0 + lane, pos4, cen4, actp, K.bhi.w);
  bool any = true, all = true;
  if (PART) {
    const float4 blo = K.blo, bhi = K.bhi;
    const ActiveBox AB = active_box(I, Box3{make_float3(blo.x, blo.y, blo.z), make_float3(bhi.x, bhi.y, bhi.z)}, blo.w);
    any = AB.any;
    all = AB.all;
    __syncwarp();
    if (lane == 0) {
      K.blo = make_float4(AB.b.lo.x, AB.b.lo.y, AB.b.lo.z, AB.H);
      K.bhi = make_float4(AB.b.hi.x, AB.b.hi.y, AB.b.hi.z, bhi.w);
    }
    __syncwarp();
  }
  S.ip[lane] = make_float4(I.p.x, I.p.y, I.p.z, I.m);
  S.ig[lane] = I.g;
  DensAcc<KAHAN> acc;
  unsigned int cnt = 0, q = 0, cur = 0, segs = 0;
  S.is[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  // inside the cluster itself first (the self interaction is a unit's first: cur, the
  // interaction whose sums acc holds)
  Walk Wk;
  bool own_only = LISTED ? self : part == 0u && (!PART || any || T.active[TL.leaf[ti]]);
  if (LISTED) Wk.live = 1u;

  if (own_only) {
    if (I.valid) dens_put(S, lane, I.p, I.Hphys, own0 + lane, I.act);
    q = ni;
  }
  bool in_self = own_only;     // the batch's pairs are counted as those of the self interaction
  // k: the candidate whose particles nr holds (-1: none), loaded one candidate ahead,
  // so that the load overlaps the work on the one before
  int k = -1;
  float4 nr = make_float4(0.f, 0.f, 0.f, 0.f);
  for (;;) {
    if (k < 0 && unit_next<PART, false, false>(K, Wk, S.jlo, S.jhi, Lq, T, TL, sort_r, sort_i, any, all, I.p,
                                 I.act ? I.H : 0.0f)) {
      k = __ffs(Wk.mask) - 1;
      Wk.mask &= Wk.mask - 1;
      if ((unsigned int)lane < K.cn[k]) nr = pos4[__float_as_uint(K.co[k].w) + lane];
    }
    const bool last = k < 0;
    unsigned int bal = 0, gj = 0;
    float4 pj = make_float4(0.f, 0.f, 0.f, 0.f);
    bool pass = false, aj = true;
    if (!last) {
      const float4 o = K.co[k];
      const bool vj = (unsigned int)lane < K.cn[k];
      gj = __float_as_uint(o.w) + lane;
      pj = make_float4(nr.x + o.x, nr.y + o.y, nr.z + o.z, nr.w);
      if (PART) aj = vj && actp[gj] != 0;
      k = -1;
      if (Wk.mask) {
        k = __ffs(Wk.mask) - 1;
        Wk.mask &= Wk.mask - 1;
        if ((unsigned int)lane < K.cn[k]) nr = pos4[__float_as_uint(K.co[k].w) + lane];
      }
      // stage only the partners within reach: of the particles that iterate (own
      // side), or, when the partner iterates, of any particle of the cluster
      const float4 blo = K.blo, bhi = K.bhi;
      const float Hj = pj.w * bhi.w, slack = K.gsh[Wk.it].w;
      const float3 p3 = make_float3(pj.x, pj.y, pj.z);
      pass = vj && (!PART || any) &&
             near_box(p3, Box3{make_float3(blo.x, blo.y, blo.z), make_float3(bhi.x, bhi.y, bhi.z)},
                      fmaxf(blo.w, Hj) + slack);
      if (PART && !pass && !all && aj) {
        const float4 clo = K.clo, chi = K.chi;
        pass = near_box(p3, Box3{make_float3(clo.x, clo.y, clo.z), make_float3(chi.x, chi.y, chi.z)}, Hj + slack);
      }
      bal = __ballot_sync(0xffffffffu, pass);
    }
    const unsigned int np = __popc(bal), rank = __popc(bal & ((1u << lane) - 1u));
    const unsigned int now = K.gidx + (unsigned int)Wk.it;
    const bool close = own_only || last || (COUNT && in_self != (Wk.it == K.selfit));
    if (close || q + np > 32u) {
      // a batch runs full: it takes the first of the candidate's particles, the next one
      // the others (batches closed before they overflow were three quarters full; with
      // full ones density passes take 3 to 8 % less time.  Force batches gain 1 to 2 % in
      // large boxes and lose 2 to 6 % below 30k particles, where a unit's latency counts
      // and a full batch's list is cut in two: they stay as they are)
      const unsigned int room = close ? 0u : 32u - q;
      if (room && now != cur) {
        if (q) segs |= 1u << q;
        else if (!KAHAN) sum_done(S, acc);
        cur = now;
      }
      if (pass && rank < room) dens_put(S, (int)(q + rank), make_float3(pj.x, pj.y, pj.z), pj.w, gj, aj);
      pass = pass && rank >= room;
      q += room;
      if (q)
        dens_batch<COUNT, PART, KAHAN, LISTED>(I, S, q, KAHAN ? 0u : segs, own_only, acc, cnt, perm, x, pos4, box, cen4, dacc, dcnt, dcomp,
                                               COUNT && in_self ? Cs : Cp, R, W);
      q = 0u - room;
      segs = 0;
      own_only = false;
      in_self = Wk.it == K.selfit;
    }
    if (last) break;
    if (np && now != cur) {
      if (q) segs |= 1u << q;
      else if (!KAHAN) sum_done(S, acc);
      cur = now;
    }
    if (pass) dens_put(S, (int)(q + rank), make_float3(pj.x, pj.y, pj.z), pj.w, gj, aj);
    q += np;
  }
  if (!KAHAN) {
    const float4 t = S.is[lane];
    acc.s = make_float4(t.x + acc.s.x, t.y + acc.s.y, t.z + acc.s.z, t.w + acc.s.w);
  }
  flush_dens(I.g, acc, cnt, dacc, dcnt, dcomp);
  if (LISTED) rec_task_end(self ? R.stask : R.ptask, S);
}

// The force interactions of one unit, as density_unit.
template <bool COUNT, bool LISTED>
__device__ __forceinline__ void force_unit(unsigned int ti, unsigned int part, unsigned int parts, bool self, int item,
    const Lists& Lq, const Tree& T, const Tiles& TL, const BoxDesc* __restrict__ box, const float4* __restrict__ cen4,
    const float4* __restrict__ vel4, const float4* __restrict__ ghost4, const float* __restrict__ sort_r,
    const unsigned int* __restrict__ sort_i, const ForceArgs& A, float4* facc, float* fvsig, ForceShared& S,
    Counters& Cp, Counters& Cs) {
  const int lane = threadIdx.x & 31;
  UnitShared& K = S.tk;
  unit_begin(K, ti, T, TL, box, part, parts);
  if (LISTED) unit_single(K, self, item, Lq, T);
  const unsigned int ni = TL.n[ti], own0 = TL.start[ti];
  const bool vi = (unsigned int)lane < ni;
  if (lane == 0) S.own0 = own0;
  const float4 P = force_stage_own(S, lane, vi, own0 + lane, A.pos4, cen4, vel4, ghost4);
  const float3 ip = make_float3(P.x, P.y, P.z);
  unsigned int q = 0;
  Walk Wk;
  bool own_only = LISTED ? self : part == 0u;      // inside the cluster itself first: each unordered pair once
  if (LISTED) Wk.live = 1u;

  if (own_only) {
    if (vi) force_put(S, lane, ip, A.pos4[own0 + lane].w, own0 + lane);
    q = ni;
  }
  bool in_self = own_only;
  int k = -1;
  float4 nr = make_float4(0.f, 0.f, 0.f, 0.f);
  for (;;) {
    if (k < 0 && unit_next<false, false, true>(K, Wk, S.v, S.f, Lq, T, TL, sort_r, sort_i, true, true, ip, P.w)) {
      k = __ffs(Wk.mask) - 1;
      Wk.mask &= Wk.mask - 1;
      if ((unsigned int)lane < K.cn[k]) nr = A.pos4[__float_as_uint(K.co[k].w) + lane];
    }
    const bool last = k < 0;
    unsigned int bal = 0, gj = 0;
    float4 pj = make_float4(0.f, 0.f, 0.f, 0.f);
    bool pass = false;
    if (!last) {
      const float4 o = K.co[k];
      const bool vj = (unsigned int)lane < K.cn[k];
      gj = __float_as_uint(o.w) + lane;
      pj = make_float4(nr.x + o.x, nr.y + o.y, nr.z + o.z, nr.w);
      k = -1;
      if (Wk.mask) {
        k = __ffs(Wk.mask) - 1;
        Wk.mask &= Wk.mask - 1;
        if ((unsigned int)lane < K.cn[k]) nr = A.pos4[__float_as_uint(K.co[k].w) + lane];
      }
      const float4 blo = K.blo, bhi = K.bhi;
      pass = vj && near_box(make_float3(pj.x, pj.y, pj.z),
                            Box3{make_float3(blo.x, blo.y, blo.z), make_float3(bhi.x, bhi.y, bhi.z)},
                            fmaxf(blo.w, pj.w * bhi.w) + K.gsh[Wk.it].w);
      bal = __ballot_sync(0xffffffffu, pass);
    }
    if (own_only || last || q + __popc(bal) > 32u || (COUNT && in_self != (Wk.it == K.selfit))) {
      if (q)
        force_batch<COUNT>(S, ip, P.w, q, own_only, A, cen4, vel4, ghost4, facc, fvsig,
                           COUNT ? (in_self ? &Cs : &Cp) : nullptr);
      q = 0;
      own_only = false;
      in_self = Wk.it == K.selfit;
    }
    if (last) break;
    if (pass) force_put(S, (int)(q + __popc(bal & ((1u << lane) - 1u))), make_float3(pj.x, pj.y, pj.z), pj.w, gj);
    q += __popc(bal);
  }
  __syncwarp();
  if (vi) flush_force((int)(own0 + lane), S.iacc[lane], S.ivs[lane], facc, fvsig);
}

// Whether a task's records still hold when its partner cell (the own cell for a
// self task) holds particles that took a new h after the recording: they do when
// every such particle lies out of reach of the own cluster, reach taken with the
// largest H the cell has had since the recording (cell H maxima only grow within
// a step), so that no pair with them was recorded or is missing.
__device__ __forceinline__ bool changed_out_of_reach(bool self, int item, unsigned int ti, const Lists& Lq,
                                                  const Tree& T, const Tiles& TL, const BoxDesc* __restrict__ box) {
  int C;
  Box3 bi;
  float reach;
  float3 off;
  if (self) {
    C = Lq.self_a[item];
    const ItemGeom g = item_geom(T, box, C, 0);
    const float4 cA = T.cen[C];
    bi = tile_box3(TL, T, ti, make_float3(-cA.x, -cA.y, -cA.z));
    const float Hm = T.hmax[C] * g.invL;
    reach = fmaxf(TL.lo[ti].w * g.invL, Hm) + g.e * 1.52587890625e-05f + g.es + 1e-6f * Hm;
    off = make_float3(0.0f, 0.0f, 0.0f);
  } else {
    const PairSetup P = pair_setup(Lq, T, box, item);
    C = P.B;
    bi = tile_box3(TL, T, ti, P.tshA);
    reach = fmaxf(TL.lo[ti].w * P.g.invL, P.HmB) + P.slack;
    off = P.g.offB;
  }
  Box3 cb;
  cb.lo = make_float3(key_float(T.clo[3 * C]) + off.x, key_float(T.clo[3 * C + 1]) + off.y,
                      key_float(T.clo[3 * C + 2]) + off.z);
  cb.hi = make_float3(key_float(T.chi[3 * C]) + off.x, key_float(T.chi[3 * C + 1]) + off.y,
                      key_float(T.chi[3 * C + 2]) + off.z);
  return !box_near(bi, cb, reach);
}

// A force task replayed from the records of the first density pass: the frame
// of the particle arithmetic is that of the units, the
// batches follow the recording warp's chain of chunks.  Valid while no particle of
// the own cluster or of the partner cell (the own cell for a self task) has taken
// a new h since the recording: the recorded pairs are then the pairs at the
// current h.
template <bool COUNT>
__device__ __forceinline__ void force_replay_task(bool self, int item, unsigned int ti, uint2 rec, const PairRec& R,
    const Lists& Lq, const Tree& T, const Tiles& TL, const BoxDesc* __restrict__ box,
    const float4* __restrict__ cen4, const float4* __restrict__ vel4, const float4* __restrict__ ghost4,
    const ForceArgs& A, float4* facc, float* fvsig, ForceShared& S, Counters* C) {
  const int lane = threadIdx.x & 31;
  // of a unit's constants only what the batches read, and the partners' frame
  const int A0 = self ? Lq.self_a[item] : Lq.pair_a[item], B0 = self ? A0 : Lq.pair_b[item];
  const int bx = T.box[A0];
  const float e = ldexpf(1.0f, -T.level[A0]);
  int dx = 0, dy = 0, dz = 0;
  if (!self) axis_vec(Lq.pair_axis[item], dx, dy, dz);
  const float4 cA = T.cen[A0], cB = T.cen[B0], cl = TL.cen[ti];
  const float3 sh = make_float3((e * dx - cB.x) - (cl.x - cA.x), (e * dy - cB.y) - (cl.y - cA.y),
                                (e * dz - cB.z) - (cl.z - cA.z));
  __syncwarp();
  if (lane == 0) {
    S.tk.box = bx;
    S.tk.L32 = (float)box[bx].L;
    S.tk.bhi.w = (float)box[bx].invL;
    S.tk.eb = box[bx].global32 ? 1.0f : e;
  }
  __syncwarp();
  const unsigned int own0 = TL.start[ti];
  const bool vi = (unsigned int)lane < TL.n[ti];
  if (lane == 0) S.own0 = own0;
  force_stage_own(S, lane, vi, own0 + lane, A.pos4, cen4, vel4, ghost4);
  unsigned int b = rec.x;
  for (unsigned int k = 0; k < rec.y; ++k, ++b) {
    if (k > 0 && b % REC_CHUNK == 0u) b = R.next[b / REC_CHUNK - 1u] * REC_CHUNK;   // the chunk is full: next one
    force_replay_batch<COUNT>(S, R.pool + 64ull * b, self && k == 0, cen4, vel4, ghost4, A, sh, facc, fvsig, C);
  }
  __syncwarp();
  if (vi) flush_force((int)(own0 + lane), S.iacc[lane], S.ivs[lane], facc, fvsig);
}

// Density interactions of one pass: one queue of units (REC: of the listed tasks).
// PART: a later pass of the h iteration (particles still iterating), where the own
// side culls against the box of the cluster's iterating particles; the first pass
// (every particle) has its own instance without that code.  Both are launched in
// a captured step, and the one that does not match the iteration returns.
// The first pass (PART = false) runs 7 blocks of 128 threads per SM (at most 73
// registers, a few spilled): issue slots bound the pass, and more warps in flight fill
// them until the spills grow (density phase of the 33.5M step 42.0 ms at 6 blocks, 41.1 at
// 7, 41.5 at 8).
template <bool COUNT, bool PART, bool KAHAN, bool REC>
__global__ void __launch_bounds__(SPH_THREADS, PART ? PART_BLOCKS : (REC ? REC_BLOCKS : DENS_BLOCKS)) k_density(Lists Lq, Tree T, Tiles TL, const BoxDesc* __restrict__ box,
                                                         const float4* __restrict__ pos4,
                                                         const float4* __restrict__ cen4,
                                                         const float* __restrict__ sort_r,
                                                         const unsigned int* __restrict__ sort_i,
                                                         const unsigned char* __restrict__ act,
                                                         const unsigned int* __restrict__ perm,
                                                         const double* __restrict__ x, float4* dacc,
                                                         unsigned int* dcnt, float4* dcomp,
                                                         unsigned long long* pc,
                                                         unsigned int* __restrict__ task_ctr, int partial_host,
                                                         const int* __restrict__ it_dev, const int* __restrict__ gflag,
                                                         unsigned int ntcap, const unsigned int* __restrict__ ntile_dev,
                                                         const uint2* __restrict__ units,
                                                         const unsigned int* __restrict__ n_units, unsigned int cap_units,
                                                         const __grid_constant__ PairRec Rec) {
  pdl_wait();
  const int partial = it_dev ? (*it_dev > 1 ? 1 : 0) : partial_host;
  if ((partial != 0) != PART) return;
  if (it_dev && it_dev[2] != 0) return;                        // the iteration has stopped
  if (PART && gflag && gflag[0] != 0) return;                  // the pass gathers
  __shared__ DensShared SH[SPH_WARPS_PER_CTA];
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  DensShared& S = SH[wl];
  RecW W;
  Counters Cp, Cs;
  // units of work (REC: the listed tasks, whose pairs are recorded one by one)
  const unsigned int nt = ntile_dev ? min(ntcap, *ntile_dev) : ntcap;
  const bool listed = !REC && units && *n_units <= cap_units;
  const unsigned int parts = REC ? 1u : unit_parts(nt);
  const unsigned int nunit = REC ? *Lq.n_live : (listed ? *n_units : nt * parts);
  // the next unit is fetched while the current one runs, unless there are so few that
  // a warp would hold one back from an idle warp
  const bool few = nunit < 4u * gridDim.x * (blockDim.x >> 5);
  unsigned int raw = 0;
  if (lane == 0) raw = atomicAdd(task_ctr, 1u);
  for (unsigned int u = __shfl_sync(0xffffffffu, raw, 0); u < nunit; u = __shfl_sync(0xffffffffu, raw, 0)) {
    if (!few && lane == 0) raw = atomicAdd(task_ctr, 1u);
    // (REC: interaction and cluster; else cluster, part and parts)
    uint2 un = make_uint2(0u, 0u);
    if (REC) un = Lq.p_live[u];
    else un = listed ? units[u] : make_uint2(u / parts, (u % parts) | (parts << 16));
    const bool self = REC && (un.x >> 31) != 0u;
    density_unit<COUNT, PART, KAHAN, REC>(REC ? un.y : un.x, REC ? 0u : un.y & 0xffffu, REC ? 1u : un.y >> 16, self,
                                          (int)(un.x & 0x7fffffffu), Lq, T, TL, box, pos4, cen4, sort_r, sort_i, act,
                                          perm, x, dacc, dcnt, dcomp, S, Cp, Cs, Rec, W);
    if (few && lane == 0) raw = atomicAdd(task_ctr, 1u);
  }
  commit_counters<COUNT>(Cp, pc, 0);
  commit_counters<COUNT>(Cs, pc, 1);
}

// Force interactions of one pass: one queue of units, or (REC) of the listed tasks,
// whose pairs the first density pass recorded.
// Registers capped at 64 per thread (8 blocks of 128 threads, whose shared memory
// fits an SM): more warps in flight to hide the partner loads outweigh the few
// spilled values (33.5M, an earlier form of the kernel: 6, 5 and 4 blocks took 74, 84
// and 98 ms against 65 ms).
template <bool COUNT, bool REC>
__global__ void __launch_bounds__(SPH_THREADS, 8) k_force(Lists Lq, Tree T, Tiles TL, const BoxDesc* __restrict__ box,
                                                       const float4* __restrict__ pos4,
                                                       const float4* __restrict__ cen4,
                                                       const float4* __restrict__ vel4,
                                                       const float4* __restrict__ ghost4,
                                                       const float* __restrict__ sort_r,
                                                       const unsigned int* __restrict__ sort_i,
                                                       const unsigned int* __restrict__ perm,
                                                       const double* __restrict__ x, float alpha, float4* facc,
                                                       float* fvsig, unsigned int* fcnt, unsigned long long* pc,
                                                       unsigned int* __restrict__ task_ctr, unsigned int ntcap,
                                                       const unsigned int* __restrict__ ntile_dev,
                                                       const uint2* __restrict__ units,
                                                       const unsigned int* __restrict__ n_units, unsigned int cap_units,
                                                       const __grid_constant__ PairRec R) {
  pdl_wait();
  __shared__ ForceShared SH[SPH_WARPS_PER_CTA];
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  ForceShared& S = SH[wl];
  Counters Cp, Cs;
  const ForceArgs A{perm, x, pos4, box, fcnt, alpha};
  const unsigned int nt = ntile_dev ? min(ntcap, *ntile_dev) : ntcap;
  const bool listed = !REC && units && *n_units <= cap_units;
  const unsigned int parts = REC ? 1u : unit_parts(nt);
  const unsigned int nunit = REC ? *Lq.n_live : (listed ? *n_units : nt * parts);
  // as in k_density
  const bool few = nunit < 4u * gridDim.x * (blockDim.x >> 5);
  unsigned int raw = 0;
  if (lane == 0) raw = atomicAdd(task_ctr, 1u);
  for (unsigned int u = __shfl_sync(0xffffffffu, raw, 0); u < nunit; u = __shfl_sync(0xffffffffu, raw, 0)) {
    if (!few && lane == 0) raw = atomicAdd(task_ctr, 1u);
    if (!REC) {
      if (COUNT && lane == 0) atomicAdd(&pc[12], 1ull);
      const uint2 un = listed ? units[u] : make_uint2(u / parts, (u % parts) | (parts << 16));
      force_unit<COUNT, false>(un.x, un.y & 0xffffu, un.y >> 16, false, 0, Lq, T, TL, box, cen4, vel4, ghost4, sort_r,
                               sort_i, A, facc, fvsig, S, Cp, Cs);
    } else {
      const uint2 lt = Lq.p_live[u];
      const int item = (int)(lt.x & 0x7fffffffu);
      const bool self = (lt.x >> 31) != 0u;
      // the records of the first density pass, where they hold
      uint2 rec = make_uint2(REC_NONE, 0u);
      if (!TL.changed[lt.y]) {
        const int a = self ? Lq.self_a[item] : Lq.pair_a[item];
        const int c = self ? a : Lq.pair_b[item];
        if (!T.changed[c] || changed_out_of_reach(self, item, lt.y, Lq, T, TL, box))
          rec = self ? R.stask[Lq.s_toff[item] + (lt.y - T.tile0[a])] : R.ptask[Lq.p_toff[item] + (lt.y - T.tile0[a])];
      }
      if (COUNT && lane == 0) atomicAdd(&pc[rec.x != REC_NONE ? 11 : 12], 1ull);
      if (rec.x != REC_NONE)
        force_replay_task<COUNT>(self, item, lt.y, rec, R, Lq, T, TL, box, cen4, vel4, ghost4, A, facc, fvsig, S,
                                 COUNT ? (self ? &Cs : &Cp) : nullptr);
      else
        force_unit<COUNT, true>(lt.y, 0u, 1u, self, item, Lq, T, TL, box, cen4, vel4, ghost4, sort_r, sort_i, A, facc,
                                fvsig, S, Cp, Cs);
    }
    if (few && lane == 0) raw = atomicAdd(task_ctr, 1u);
  }
  commit_counters<COUNT>(Cp, pc, 2);
  commit_counters<COUNT>(Cs, pc, 3);
}

// The units of a decomposition whose clusters are neither few (all are then split the
// same way) nor so many that the longest does not matter: a cluster's expected
// partners, from the share of each partner cell within reach of its box, and one unit
// per UNIT_PARTNERS of them.  A sparse cluster beside a dense cell (the rim of a
// clump, or a first guess of h far from its root) has thousands: as one unit, one
// warp held the force pass of a 636k-particle log-normal box at its first guess for
// as long again as all the others took.  One warp per cluster.
constexpr float UNIT_PARTNERS = 2048.0f;

__global__ void k_unit_list(unsigned int ntcap, const unsigned int* __restrict__ ntile_dev, Lists Lq, Tree T, Tiles TL,
                            const BoxDesc* __restrict__ box, uint2* __restrict__ units,
                            unsigned int* __restrict__ n_units, unsigned int cap) {
  pdl_wait();
  const unsigned int nt = ntile_dev ? min(ntcap, *ntile_dev) : ntcap;
  const int lane = threadIdx.x & 31;
  const unsigned int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
  // a warp takes up to 16 adjacent clusters and their places in the list with one atomic
  // (one per cluster on the one counter: 0.96 ms for 1.2M clusters), fewer where that
  // would leave warps idle
  const unsigned int run = min(16u, max(1u, nt / nwarps));
  for (unsigned int t0 = warp * run; t0 < nt; t0 += nwarps * run) {
    unsigned int mine = 0;       // lane j: the units of cluster t0 + j
    for (unsigned int j = 0; j < run && t0 + j < nt; ++j) {
      const unsigned int t = t0 + j;
      const int leaf = (int)TL.leaf[t];
      const float4 lo = TL.lo[t], hi = TL.hi[t], cl = TL.cen[t];
      const float H = lo.w * (float)box[T.box[leaf]].invL;
      float est = 0.0f;
      for (int A = leaf; A >= 0; A = T.parent[A]) {
        const unsigned int n = (unsigned int)__popc(T.pmask[A]) + (A == leaf ? 1u : 0u);
        const float e = ldexpf(1.0f, -T.level[A]);
        for (unsigned int k = lane; k < n; k += 32) {
          int B = A, dx = 0, dy = 0, dz = 0;
          if (A != leaf || k > 0u) {
            const uint2 pr = Lq.csr[T.pstart[A] + k - (A == leaf ? 1u : 0u)];
            B = (int)pr.x;
            axis_vec((int)pr.y, dx, dy, dz);
          }
          const float4 cA = T.cen[A];
          // the partner cell's centre in the frame of the own leaf; the part of each of
          // its edges within H of the own box
          const float bx = e * dx - (cl.x - cA.x), by = e * dy - (cl.y - cA.y), bz = e * dz - (cl.z - cA.z);
          const float fx = fminf(hi.x + H, bx + 0.5f * e) - fmaxf(lo.x - H, bx - 0.5f * e);
          const float fy = fminf(hi.y + H, by + 0.5f * e) - fmaxf(lo.y - H, by - 0.5f * e);
          const float fz = fminf(hi.z + H, bz + 0.5f * e) - fmaxf(lo.z - H, bz - 0.5f * e);
          const float ie = 1.0f / e;
          est += fmaxf(fx, 0.0f) * ie * (fmaxf(fy, 0.0f) * ie) * (fmaxf(fz, 0.0f) * ie) * (float)T.count[B];
        }
      }
      est = warp_sum(est);
      const unsigned int parts = (unsigned int)fminf(32.0f, fmaxf(1.0f, ceilf(est * (1.0f / UNIT_PARTNERS))));
      if ((unsigned int)lane == j) mine = parts;
    }
    const unsigned int total = __reduce_add_sync(0xffffffffu, mine);
    unsigned int at = 0;
    if (lane == 0) at = atomicAdd(n_units, total);
    at = __shfl_sync(0xffffffffu, at, 0);
    for (unsigned int j = 0; j < run && t0 + j < nt; ++j) {
      const unsigned int parts = __shfl_sync(0xffffffffu, mine, (int)j);
      if ((unsigned int)lane < parts && at + lane < cap)
        units[at + lane] = make_uint2(t0 + j, (unsigned int)lane | (parts << 16));
      at += parts;
    }
  }
}

// Tasks of a recording first density pass, or of the force pass that replays it, as
// (interaction, cluster); bit 31 of the interaction marks a self task.  Pair tasks: those
// whose cluster lies within reach of the partner cell (the test the sweep would start
// with).  Self tasks come first: the costliest tasks are then taken early and the short
// pair tasks fill the end of the pass.  One thread per task; warp-aggregated appends.
__global__ void k_live_tasks(Lists Lq, Tree T, Tiles TL, const BoxDesc* __restrict__ box, long long npt,
                             long long nst) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const long long ntask = npt + nst;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long b0 = (long long)blockIdx.x * blockDim.x; b0 < ntask; b0 += stride) {
    const long long t = b0 + threadIdx.x;
    bool live = false;
    unsigned int rec = 0, ti = 0;
    if (t < nst) {
      const unsigned int ts = (unsigned int)t;
      const int item = (int)Lq.s_task[ts];
      const int A = Lq.self_a[item];
      ti = T.tile0[A] + (ts - Lq.s_toff[item]);
      rec = (unsigned int)item | 0x80000000u;
      live = true;
    } else if (t < ntask) {
      const unsigned int tp = (unsigned int)(t - nst);
      const int item = (int)Lq.p_task[tp];
      const int A0 = Lq.pair_a[item];
      ti = T.tile0[A0] + (tp - Lq.p_toff[item]);
      rec = (unsigned int)item;
      const PairSetup P = pair_setup(Lq, T, box, item);
      const Box3 bi = tile_box3(TL, T, ti, P.tshA);
      live = box_near(bi, P.cellB, fmaxf(TL.lo[ti].w * P.g.invL, P.HmB) + P.slack);
    }
    const unsigned int bal = __ballot_sync(0xffffffffu, live);
    unsigned int at = 0;
    if (lane == 0 && bal) at = atomicAdd(Lq.n_live, (unsigned int)__popc(bal));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (live) Lq.p_live[at + __popc(bal & ((1u << lane) - 1u))] = make_uint2(rec, ti);
  }
}

// =========================================================================== gathered later passes
// A later pass of the h iteration needs the density sums of the particles still
// iterating only (Section II-D: the density loop runs again for the particles
// whose h has not converged).  Tracked per cluster and cell, a few per cent of
// randomly placed iterating particles make most clusters and cells active, and
// the symmetric tasks then run nearly in full for their partner side.  A later
// pass with few iterating particles gathers instead: each leaf's iterating
// particles are packed, in their sorted order, into clusters of up to 32, so that
// the packed clusters of a cell are one range; every interaction then runs once
// per packed cluster of each of its cells, the own side only — for a pair (A, B)
// A's packed clusters against B's clusters and B's against A's, for the self
// interaction of A its packed clusters against all of A's clusters with the
// particle itself left out.  A pair with r < H_i of an iterating particle i lies
// in exactly one interaction (Section II-B), and there it is taken once, from i.

// The packing runs for the later passes only (the first pass of a captured
// iteration returns at once, and so does a stopped iteration).
__device__ __forceinline__ bool later_pass(const int* it_dev) { return it_dev[0] > 1 && it_dev[2] == 0; }

// After the scan of the counts (rank[t]: iterating particles before cluster t):
// the packed clusters of each leaf, at its first cluster (0 elsewhere).
__global__ void k_pack_leaf(long long ntcap, const unsigned int* __restrict__ ntile_dev, const int* __restrict__ it_dev,
                            Tree T, Tiles TL, const unsigned int* __restrict__ rank, unsigned int* __restrict__ v) {
  pdl_wait();
  if (!later_pass(it_dev)) return;
  const long long nt = ntile_dev ? min(ntcap, (long long)*ntile_dev) : ntcap;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t <= nt;
       t += (long long)gridDim.x * blockDim.x) {
    unsigned int val = 0;
    if (t < nt) {
      const unsigned int L = TL.leaf[t];
      if (T.tile0[L] == (unsigned int)t) val = (rank[t + T.ntile[L]] - rank[t] + 31u) >> 5;
    }
    v[t] = val;
  }
}

// The packed clusters of a later pass, when it gathers (after the scan of k_pack_leaf's
// counts: pk0[t], the first packed cluster of the leaf whose first cluster is t): the
// sorted indices of the iterating particles by rank (idx), and per packed cluster its
// first rank and its leaf's first cluster (info) and its size (pn).  The pass gathers
// when it is a later one and at most an eighth of the particles iterate (gflag[0]).  One
// warp per cluster.
__global__ void k_pack_fill(long long ntcap, const unsigned int* __restrict__ ntile_dev, const int* __restrict__ it_dev,
                            long long N, Tree T, Tiles TL, const unsigned char* __restrict__ act,
                            const unsigned int* __restrict__ rank, const unsigned int* __restrict__ pk0,
                            const unsigned int* __restrict__ pk_tot, unsigned int* __restrict__ idx,
                            uint2* __restrict__ info, unsigned char* __restrict__ pn, int* __restrict__ gflag) {
  pdl_wait();
  const bool on = later_pass(it_dev) && GATHER_SHARE * pk_tot[0] <= (unsigned long long)N;
  if (blockIdx.x == 0 && threadIdx.x == 0) gflag[0] = on ? 1 : 0;
  if (!on) return;
  const long long nt = ntile_dev ? min(ntcap, (long long)*ntile_dev) : ntcap;
  const int lane = threadIdx.x & 31;
  const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long t = warp; t < nt; t += nwarps) {
    const unsigned int s = TL.start[t];
    const bool a = (unsigned int)lane < TL.n[t] && act[s + lane];
    const unsigned int bal = __ballot_sync(0xffffffffu, a);
    if (!bal || !a) continue;
    const unsigned int L = TL.leaf[t], t0 = T.tile0[L];
    const unsigned int r0 = rank[t0];                        // the leaf's first rank
    const unsigned int na = rank[t0 + T.ntile[L]] - r0;       // its iterating particles
    const unsigned int k = rank[t] - r0 + __popc(bal & ((1u << lane) - 1u));
    idx[r0 + k] = s + (unsigned int)lane;
    if ((k & 31u) == 0u) {
      const unsigned int pid = pk0[t0] + (k >> 5);
      info[pid] = make_uint2(r0 + k, t0);
      pn[pid] = (unsigned char)min(32u, na - k);
    }
  }
}

// One batch of q <= 32 staged partners, the own side only; in a self interaction
// the particle itself (staged with its cell) is left out.
template <bool KAHAN>
__device__ __forceinline__ void gather_batch(const DensI& I, DensShared& S, unsigned int q, unsigned int segs, bool self,
                                             const float4* __restrict__ cen4, DensAcc<KAHAN>& acc, unsigned int& cnt,
                                             const unsigned int* perm, const double* x,
                                             const float4* __restrict__ pos4, const BoxDesc* __restrict__ box,
                                             float4* dacc, unsigned int* dcnt, float4* dcomp) {
  const int lane = threadIdx.x & 31;
  const bool v = (unsigned int)lane < q;
  __syncwarp();
  float jm = 0.0f;
  if (v) {
    jm = cen4[S.g[lane]].w;       // needed after the mask
  } else {
    S.x[lane] = 1e30f;
    S.y[lane] = 1e30f;
    S.z[lane] = 1e30f;
  }
  const unsigned int jvalid = __ballot_sync(0xffffffffu, v);
  __syncwarp();
  unsigned int m, none;
  const float iband = BAND_REL * I.H * (S.tk.eb + I.H), ilo = I.H * I.H - iband;
  near_masks<false>(I.p, I.H * I.H + iband, S.x, S.y, S.z, nullptr, (int)((q + 3u) & ~3u), m, none);
  m &= I.valid ? jvalid : 0u;
  S.m[lane] = jm;
  __syncwarp();
  if (self)
    for (unsigned int b = m; b; b &= b - 1)
      if (S.g[__ffs(b) - 1] == I.g) m &= ~(b & (0u - b));
  dens_row(I, ilo, S, m, segs, acc, cnt, perm, x, pos4, box, dacc, dcnt, dcomp);
  __syncwarp();
}

// One unit of a gathered pass: packed cluster pid, a part of its interactions: those of
// every cell on its leaf's chain, in both directions of the pairs, walked as in
// density_unit (a task per interaction set up, boxed and flushed a packed cluster 27
// times, in batches mostly partly filled).  The frame is the leaf's centre, as there.
template <bool KAHAN>
__device__ __forceinline__ void gather_unit(unsigned int pid, unsigned int part, unsigned int parts, const Lists& Lq,
                                            const Tree& T, const Tiles& TL, const BoxDesc* __restrict__ box,
                                            const float4* __restrict__ pos4, const float4* __restrict__ cen4,
                                            const float* __restrict__ sort_r, const unsigned int* __restrict__ sort_i,
                                            const unsigned int* __restrict__ perm, const double* __restrict__ x,
                                            float4* dacc, unsigned int* dcnt, float4* dcomp,
                                            const uint2* __restrict__ pk_info, const unsigned char* __restrict__ pk_n,
                                            const unsigned int* __restrict__ pk_idx, DensShared& S) {
  const int lane = threadIdx.x & 31;
  UnitShared& K = S.tk;
  const uint2 info = pk_info[pid];
  const unsigned int n = pk_n[pid];
  unit_begin(K, info.y, T, TL, box, part, parts);
  const bool vi = (unsigned int)lane < n;
  const DensI I = load_dens(vi, vi ? pk_idx[info.x + lane] : 0u, pos4, cen4, nullptr, K.bhi.w);
  S.ip[lane] = make_float4(I.p.x, I.p.y, I.p.z, I.m);
  S.ig[lane] = I.g;
  // the packed particles' box and largest H: the own side reaches no further
  Box3 bo;
  bo.lo = make_float3(warp_min(vi ? I.p.x : 1e30f), warp_min(vi ? I.p.y : 1e30f), warp_min(vi ? I.p.z : 1e30f));
  bo.hi = make_float3(warp_max(vi ? I.p.x : -1e30f), warp_max(vi ? I.p.y : -1e30f), warp_max(vi ? I.p.z : -1e30f));
  const float Ho = warp_max(vi ? I.H : 0.0f);
  const float invL = K.bhi.w;
  __syncwarp();
  if (lane == 0) {
    K.blo = K.clo = make_float4(bo.lo.x, bo.lo.y, bo.lo.z, Ho);
    K.bhi = K.chi = make_float4(bo.hi.x, bo.hi.y, bo.hi.z, invL);
  }
  __syncwarp();
  DensAcc<KAHAN> acc;
  unsigned int cnt = 0, q = 0, cur = 0, segs = 0;
  S.is[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  Walk Wk;
  bool own = false;      // the batch holds particles of the own leaf
  int k = -1;
  float4 nr = make_float4(0.f, 0.f, 0.f, 0.f);
  for (;;) {
    if (k < 0 && unit_next<false, true, false>(K, Wk, S.jlo, S.jhi, Lq, T, TL, sort_r, sort_i, true, true, I.p,
                                        vi ? I.H : 0.0f)) {
      k = __ffs(Wk.mask) - 1;
      Wk.mask &= Wk.mask - 1;
      if ((unsigned int)lane < K.cn[k]) nr = pos4[__float_as_uint(K.co[k].w) + lane];
    }
    const bool last = k < 0;
    unsigned int bal = 0, gj = 0;
    float4 pj = make_float4(0.f, 0.f, 0.f, 0.f);
    bool pass = false;
    if (!last) {
      const float4 o = K.co[k];
      const bool vj = (unsigned int)lane < K.cn[k];
      gj = __float_as_uint(o.w) + lane;
      pj = make_float4(nr.x + o.x, nr.y + o.y, nr.z + o.z, nr.w);
      k = -1;
      if (Wk.mask) {
        k = __ffs(Wk.mask) - 1;
        Wk.mask &= Wk.mask - 1;
        if ((unsigned int)lane < K.cn[k]) nr = pos4[__float_as_uint(K.co[k].w) + lane];
      }
      pass = vj && near_box(make_float3(pj.x, pj.y, pj.z), bo, Ho + K.gsh[Wk.it].w);
      bal = __ballot_sync(0xffffffffu, pass);
    }
    const unsigned int np = __popc(bal), rank = __popc(bal & ((1u << lane) - 1u));
    const unsigned int now = K.gidx + (unsigned int)Wk.it;
    if (last || q + np > 32u) {
      const unsigned int room = last ? 0u : 32u - q;
      if (room && now != cur) {
        if (q) segs |= 1u << q;
        else if (!KAHAN) sum_done(S, acc);
        cur = now;
      }
      if (pass && rank < room) dens_put(S, (int)(q + rank), make_float3(pj.x, pj.y, pj.z), pj.w, gj, true);
      pass = pass && rank >= room;
      q += room;
      own = own || (room && Wk.it == K.selfit);
      if (q) gather_batch<KAHAN>(I, S, q, KAHAN ? 0u : segs, own, cen4, acc, cnt, perm, x, pos4, box, dacc, dcnt, dcomp);
      q = 0u - room;
      segs = 0;
      own = false;
    }
    if (last) break;
    if (np && now != cur) {
      if (q) segs |= 1u << q;
      else if (!KAHAN) sum_done(S, acc);
      cur = now;
    }
    if (pass) dens_put(S, (int)(q + rank), make_float3(pj.x, pj.y, pj.z), pj.w, gj, true);
    own = own || Wk.it == K.selfit;
    q += np;
  }
  if (!KAHAN) {
    const float4 t = S.is[lane];
    acc.s = make_float4(t.x + acc.s.x, t.y + acc.s.y, t.z + acc.s.z, t.w + acc.s.w);
  }
  flush_dens(I.g, acc, cnt, dacc, dcnt, dcomp);
}

#ifndef GATHER_BLOCKS
#define GATHER_BLOCKS 7
#endif
// The gathered density pass (a later pass of the h iteration that gathers): units of the
// packed clusters; g_n[1] counts the passes that gathered.  Returns at once when the pass
// takes the clusters' units instead.
template <bool KAHAN>
__global__ void __launch_bounds__(SPH_THREADS, GATHER_BLOCKS) k_density_gather(
    Lists Lq, Tree T, Tiles TL, const BoxDesc* __restrict__ box, const float4* __restrict__ pos4,
    const float4* __restrict__ cen4, const float* __restrict__ sort_r, const unsigned int* __restrict__ sort_i,
    const unsigned int* __restrict__ perm, const double* __restrict__ x, float4* dacc, unsigned int* dcnt,
    float4* dcomp, unsigned int* __restrict__ g_n, const int* __restrict__ gflag, const uint2* __restrict__ pk_info,
    const unsigned char* __restrict__ pk_n, const unsigned int* __restrict__ pk_idx,
    const unsigned int* __restrict__ pk_tot, unsigned int* __restrict__ task_ctr) {
  pdl_wait();
  if (gflag[0] == 0) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) g_n[1] += 1u;
  __shared__ DensShared SH[SPH_WARPS_PER_CTA];
  const int lane = threadIdx.x & 31;
  DensShared& S = SH[threadIdx.x >> 5];
  const unsigned int npk = pk_tot[1], parts = unit_parts(npk), nunit = npk * parts;
  unsigned int t = 0;
  if (lane == 0) t = atomicAdd(task_ctr, 1u);
  for (t = __shfl_sync(0xffffffffu, t, 0); t < nunit; t = __shfl_sync(0xffffffffu, t, 0)) {
    gather_unit<KAHAN>(t / parts, t % parts, parts, Lq, T, TL, box, pos4, cen4, sort_r, sort_i, perm, x, dacc, dcnt,
                       dcomp, pk_info, pk_n, pk_idx, S);
    if (lane == 0) t = atomicAdd(task_ctr, 1u);
  }
}

// =========================================================================== ghost
// mode 0: finalise every particle at its current h (one density pass);
// mode 1: one h iteration (Newton on N~ = n_ngb, bracket, clamp) for the
//         active particles, finalising those that converged or ran out.
__global__ void k_ghost(long long N, int mode, int it_host, const int* __restrict__ it_dev, int max_iter,
                        float gamma_k, float n_ngb, float tol,
                        float gamma_gas, const unsigned int* __restrict__ perm, float* __restrict__ Hs,
                        float4* __restrict__ pos4, const float4* __restrict__ cen4, const float4* __restrict__ vel4,
                        float4* __restrict__ dacc, unsigned int* __restrict__ dcnt, float4* __restrict__ dcomp,
                        unsigned char* __restrict__ act, float* __restrict__ h,
                        float* __restrict__ hlo, float* __restrict__ hhi, int* __restrict__ conv,
                        const float* __restrict__ hlimp, const unsigned int* __restrict__ leaf_of, Tree T,
                        float4* __restrict__ ghost4, float4* __restrict__ hhist, int* __restrict__ n_active,
                        unsigned int* __restrict__ err_all, long long nnodes, long long ntile,
                        unsigned char* __restrict__ t_active, unsigned char* __restrict__ tl_active,
                        unsigned int* __restrict__ t_alo, unsigned int* __restrict__ t_ahi) {
  pdl_wait();
  // the iteration number: the host's, or in a captured step the device counter
  const int it = it_dev ? *it_dev : it_host;
  if (it_dev && it_dev[2] != 0) return;    // the iteration has stopped (batched iterations)
  if (mode == 1) {
    // the marks of this pass's cells and clusters, and the boxes of their iterating
    // particles (those of the next pass are set anew)
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, nth = (long long)gridDim.x * blockDim.x;
    for (long long k = t0; k < 3 * nnodes; k += nth) {
      t_alo[k] = 0xffffffffu;
      t_ahi[k] = 0u;
      if (k < nnodes) t_active[k] = 0;
    }
    for (long long k = t0; k < ntile; k += nth) tl_active[k] = 0;
  }
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < N; p += (long long)gridDim.x * blockDim.x) {
    if (mode == 1 && !act[p]) continue;
    const unsigned int i = perm[p];
    const float H = Hs[p];
    const float m = cen4[p].w;
    float4 a = dacc[p];
    if (dcomp) {      // compensated sums: the rounding of their additions
      const float4 c = dcomp[p];
      a = make_float4(a.x + c.x, a.y + c.y, a.z + c.z, a.w + c.w);
      dacc[p] = a;
    }
    const float sw = a.z + 1.0f;          // self term w(0) = 1
    const float Nw = (32.0f / 3.0f) * sw; // (4 pi / 3) H^3 n with n = (8/pi) sum w / H^3
    const float F = Nw - n_ngb;
    const bool ok = fabsf(F) <= tol * n_ngb;
    if (mode == 1 && !ok && it < max_iter) {
      const float hc = h[i];
      float lo = hlo[i], hi = hhi[i];
      if (F < 0.0f) lo = hc;
      else hi = hc;
      // dN~/dh = gamma_K (4 pi/3) H^2 (3 n - sum (3W + r W')) = -gamma_K (32/3) sum q w' / H
      const float dN = -gamma_k * (32.0f / 3.0f) * a.w / H;
      float hn = dN > 0.0f ? hc - F / dN : (F < 0.0f ? 2.0f * hc : 0.5f * hc);
      hn = fminf(fmaxf(hn, 0.5f * hc), 2.0f * hc);
      if (lo > 0.0f && isfinite(hi) && !(hn > lo && hn < hi)) hn = 0.5f * (lo + hi);
      hlo[i] = lo;
      hhi[i] = hi;
      h[i] = hn;
      const float Hn = __fmul_rn(gamma_k, hn);
      Hs[p] = Hn;
      pos4[p].w = Hn;
      if (!(Hn < hlimp[p])) atomicOr(err_all, ERR_REBUILD);
      if (Hn > H) {
        // a cell's H_max bounds its children's: the climb ends at the first cell
        // that already covers Hn
        for (int id = (int)leaf_of[p]; id >= 0; id = T.parent[id]) {
          if (T.hmax[id] >= Hn) break;
          atomic_max_pos(&T.hmax[id], Hn);
        }
      }
      {
        // one atomic for the lanes here (every particle of a first pass may iterate)
        const unsigned int am = __activemask();
        if ((threadIdx.x & 31) == __ffs(am) - 1) atomicAdd(n_active, __popc(am));
      }
      // the next pass sums anew
      dacc[p] = make_float4(0.f, 0.f, 0.f, 0.f);
      dcnt[p] = 0;
      if (dcomp) dcomp[p] = make_float4(0.f, 0.f, 0.f, 0.f);
      continue;
    }
    act[p] = 0;
    conv[i] = ok ? 1 : 0;
    {
      // the root of N~(h) = N_ngb one Newton step from the final h: where the next
      // step's h iteration extrapolates from
      const float hc = h[i];
      const float dN = -gamma_k * (32.0f / 3.0f) * a.w / H;
      const float hr = dN > 0.0f ? hc - F / dN : hc;
      hhist[i].x = fminf(fmaxf(hr, 0.9f * hc), 1.1f * hc);
    }
    const float ih = 1.0f / H;
    const float K3 = SPH_KNORM * ih * ih * ih;
    const float rho = K3 * (a.x + m);
    const float u = vel4[p].w;
    const float P = (gamma_gas - 1.0f) * rho * u;
    const float c = sqrtf(gamma_gas * P / rho);
    // f = [1 + h/(3 rho) d rho/dh]^-1 = 3 rho / (-sum_j m_j r W'), without cancellation;
    // 1 when no other particle lies inside the support
    const float f = a.y < 0.0f ? -3.0f * (a.x + m) / a.y : 1.0f;
    ghost4[p] = make_float4(rho, f * P / (rho * rho), c, ih);
  }
}

// After an h iteration: marks the clusters and cells that still hold a particle iterating
// h (a cluster's largest H follows the H its particles took), with the box of those
// particles in each cell's frame.  One warp per cluster; the cluster's box of active
// particles is added to every cell on its chain with ordered-key atomics.  With pair
// records (rec) also the clusters and cells that changed since the recording, and the
// boxes of the particles that did.  Counts the particles still iterating per cluster
// (cnt[t], and cnt[ntile] = 0) for the packing that follows.
__global__ void k_mark_active(long long ntile, const unsigned int* __restrict__ ntile_dev,
                              const unsigned char* __restrict__ act, const float4* __restrict__ pos4, Tree T, Tiles TL,
                              unsigned int* __restrict__ cnt, int rec) {
  pdl_wait();
  if (ntile_dev) ntile = min(ntile, (long long)*ntile_dev);   // a captured step: this build's clusters
  const int lane = threadIdx.x & 31;
  const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  if (blockIdx.x == 0 && threadIdx.x == 0) cnt[ntile] = 0;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long t = warp; t < ntile; t += nwarps) {
    const unsigned int n = TL.n[t], s0 = TL.start[t];
    const bool a = (unsigned int)lane < n && act[s0 + lane];
    const unsigned int bal = __ballot_sync(0xffffffffu, a);
    if (lane == 0) cnt[t] = __popc(bal);
    if (!bal) continue;
    float3 lo = make_float3(FLT_MAX, FLT_MAX, FLT_MAX), hi = make_float3(-FLT_MAX, -FLT_MAX, -FLT_MAX);
    float hm = 0.0f;
    if (a) {
      const float4 p = pos4[s0 + lane];
      lo = make_float3(p.x, p.y, p.z);
      hi = lo;
      hm = p.w;
    }
    lo.x = warp_min(lo.x); lo.y = warp_min(lo.y); lo.z = warp_min(lo.z);
    hi.x = warp_max(hi.x); hi.y = warp_max(hi.y); hi.z = warp_max(hi.z);
    // only particles that iterate change H: the cluster's largest H grows to theirs
    hm = warp_max(hm);
    if (lane == 0) {
      if (hm > TL.lo[t].w) TL.lo[t].w = hm;
      TL.active[t] = 1;
      if (rec) TL.changed[t] = 1;
    }
    if (lane >= (rec ? 12 : 6)) continue;
    // a lane per bound: the lower and upper corners of the iterating particles' box, then
    // of those that took a new h since the recording
    const int k = lane % 3;
    const bool up = (lane / 3) & 1;
    const float4 lc = TL.cen[t];
    const float mine = up ? (k == 0 ? hi.x : (k == 1 ? hi.y : hi.z)) : (k == 0 ? lo.x : (k == 1 ? lo.y : lo.z));
    const float lck = k == 0 ? lc.x : (k == 1 ? lc.y : lc.z);
    unsigned int* arr = lane < 6 ? (up ? T.ahi : T.alo) : (up ? T.chi : T.clo);
    for (int id = (int)TL.leaf[t]; id >= 0; id = T.parent[id]) {
      if (lane == 0) {
        T.active[id] = 1;
        if (rec) T.changed[id] = 1;
      }
      const float key_at = mine + (lck - reinterpret_cast<const float*>(&T.cen[id])[k]);   // the offset is exact
      if (up) atomicMax(&arr[3 * id + k], float_key(key_at));
      else atomicMin(&arr[3 * id + k], float_key(key_at));
    }
  }
}

// Tasks: one per (interaction, cluster of its first cell).  Counts per
// interaction over the whole list capacity (zero past the list), so that the
// prefix and the task totals are ready before the host reads the list sizes.
__global__ void k_task_tiles(Lists Lq, Tree T, int cap_pair, int cap_self) {
  pdl_wait();
  const int npair = min(Lq.counts[1], cap_pair), nself = min(Lq.counts[0], cap_self);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < cap_pair + cap_self; i += gridDim.x * blockDim.x) {
    if (i < cap_pair) Lq.p_toff[i] = i < npair ? T.ntile[Lq.pair_a[i]] : 0u;
    else Lq.s_toff[i - cap_pair] = i - cap_pair < nself ? T.ntile[Lq.self_a[i - cap_pair]] : 0u;
  }
}

// task -> interaction tables (one warp per interaction)
// The tables hold cap_p pair tasks and cap_s self tasks, and nothing is written past them.
__global__ void k_task_items(Lists Lq, Tree T, int npair, int nself, unsigned int cap_p, unsigned int cap_s) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int i = warp; i < npair + nself; i += nwarps) {
    const bool pr = i < npair;
    const int it = pr ? i : i - npair;
    const unsigned int t0 = pr ? Lq.p_toff[it] : Lq.s_toff[it];
    const unsigned int n = T.ntile[pr ? Lq.pair_a[it] : Lq.self_a[it]];
    unsigned int* dst = pr ? Lq.p_task : Lq.s_task;
    const unsigned int cap = pr ? cap_p : cap_s;
    for (unsigned int k = lane; k < n && t0 + k < cap; k += 32) dst[t0 + k] = (unsigned int)it;
  }
}

__global__ void k_count_unconverged(long long N, const int* __restrict__ conv, int* __restrict__ out) {
  pdl_wait();
  int c = 0;
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < N; p += (long long)gridDim.x * blockDim.x)
    c += conv[p] ? 0 : 1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

// Sets up a first pass: every particle, cell and cluster takes part, with fresh sums;
// in an h iteration (hlo given) also fresh brackets and flags, and the iteration's state
// on the device (it > 0: that iteration comes next).
__global__ void k_pass_setup(long long N, unsigned char* __restrict__ act, float4* __restrict__ dacc,
                             unsigned int* __restrict__ dcnt, float4* __restrict__ dcomp, float* __restrict__ hlo,
                             float* __restrict__ hhi, int* __restrict__ conv, long long nnodes,
                             unsigned char* __restrict__ t_active, long long ntile,
                             unsigned char* __restrict__ tl_active, unsigned int* __restrict__ task_ctr,
                             int* __restrict__ dev_counters, unsigned int* __restrict__ err_all,
                             int* __restrict__ gflag, int* __restrict__ it_dev, int it, unsigned int* __restrict__ g_n) {
  pdl_wait();
  const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, nth = (long long)gridDim.x * blockDim.x;
  if (t0 < 4) {
    task_ctr[t0] = 0;
    dev_counters[t0] = 0;
    if (err_all) err_all[t0] = 0;
  }
  if (t0 == 0) {
    gflag[0] = 0;
    if (it > 0) {
      it_dev[0] = it;
      it_dev[2] = 0;
      if (it == 1) {
        it_dev[1] = 0;
        g_n[1] = 0;
      }
    }
  }
  for (long long p = t0; p < N; p += nth) {
    act[p] = 1;
    dacc[p] = make_float4(0.f, 0.f, 0.f, 0.f);
    dcnt[p] = 0;
    if (dcomp) dcomp[p] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (hlo) {
      hlo[p] = 0.0f;
      hhi[p] = __int_as_float(0x7f800000);
      conv[p] = 0;
    }
  }
  for (long long k = t0; k < nnodes; k += nth) t_active[k] = 1;
  for (long long k = t0; k < ntile; k += nth) tl_active[k] = 1;
}

// =========================================================================== captured steps
// Conditions of a step captured as a CUDA graph with conditional nodes (one
// thread each).  keep: the decomposition stays (no particle outgrew the limits).
__global__ void k_cond_keep(cudaGraphConditionalHandle keep, const unsigned int* __restrict__ reuse_flag) {
  pdl_wait();
  cudaGraphSetConditional(keep, *reuse_flag == 0u ? 1u : 0u);
}

// start of the h iteration: iteration 1 runs
__global__ void k_iter_start(cudaGraphConditionalHandle iter, int* __restrict__ it_dev) {
  pdl_wait();
  it_dev[0] = 1;
  it_dev[2] = 0;
  cudaGraphSetConditional(iter, 1u);
}

// The same control without a graph: after iteration it_dev[0], stop (it_dev[2] =
// 1: every particle finalised or the limit reached; 2: a rebuild is needed) or
// advance to the next iteration.  Kernels of later iterations launched ahead
// return at once after a stop.
__global__ void k_iter_step(int* __restrict__ it_dev, int* __restrict__ n_active,
                            const unsigned int* __restrict__ err_all, int max_iter, unsigned int* __restrict__ task_ctr) {
  pdl_wait();
  if (it_dev[2] != 0) return;
  task_ctr[0] = task_ctr[1] = task_ctr[3] = 0;      // the density passes' queues
  const int na = *n_active;
  if (it_dev[0] == 1) it_dev[1] = na;
  if ((*err_all & ERR_REBUILD) != 0u) it_dev[2] = 2;
  else if (na == 0 || it_dev[0] >= max_iter) it_dev[2] = 1;
  else it_dev[0] += 1;
  *n_active = 0;
}

// after iteration *it_dev: another while particles still iterate, no rebuild is
// needed and the limit is not reached; the force pass follows unless a rebuild is
// needed (the host then takes over).  n_active is cleared for the next iteration.
__global__ void k_iter_next(cudaGraphConditionalHandle iter, cudaGraphConditionalHandle force, int* __restrict__ it_dev,
                            int* __restrict__ n_active, const unsigned int* __restrict__ err_all, int max_iter,
                            int* __restrict__ first_active, unsigned int* __restrict__ task_ctr) {
  pdl_wait();
  task_ctr[0] = task_ctr[1] = task_ctr[3] = 0;      // the density passes' queues
  const bool rebuild = (*err_all & ERR_REBUILD) != 0u;
  const int na = *n_active;
  if (*it_dev == 1) *first_active = na;
  const bool more = !rebuild && na > 0 && *it_dev < max_iter;
  if (more) *it_dev += 1;
  *n_active = 0;
  it_dev[3] = (!more && !rebuild) ? 1 : 0;     // for the conditions of later force phases
  cudaGraphSetConditional(iter, more ? 1u : 0u);
  cudaGraphSetConditional(force, (!more && !rebuild) ? 1u : 0u);
}

// a condition taken from a flag in device memory (a graph node of its own)
__global__ void k_cond_set(cudaGraphConditionalHandle h, const int* __restrict__ flag) {
  cudaGraphSetConditional(h, *flag != 0 ? 1u : 0u);
}

// the displacement of every box, written into its descriptor on the device
__global__ void k_set_drift(int nbox, BoxDesc* __restrict__ box, const unsigned long long* __restrict__ dmax) {
  pdl_wait();
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += gridDim.x * blockDim.x) {
    const double d = __longlong_as_double((long long)dmax[b]);
    box[b].drift2 = (float)(2.0 * d);
    box[b].drift_u = (float)(d * box[b].invL);
  }
}

// =========================================================================== reductions
// FP64 conservation sums per box: sum m a (3), sum m (v.a + du/dt), sum m v (3),
// sum m (v^2/2 + u).  Block row y reduces boxes y, y + gridDim.y, ...: every
// thread accumulates its particles of the box in FP64 registers, then one block
// reduction and eight atomics per box.
__global__ void __launch_bounds__(256) k_reduce(int nbox, const long long* __restrict__ boff,
                                                const BoxDesc* __restrict__ box, const unsigned int* __restrict__ perm,
                                                const float4* __restrict__ cen4, const float4* __restrict__ vel4,
                                                const float4* __restrict__ facc, float4* __restrict__ a_in,
                                                double* __restrict__ red) {
  pdl_wait();
  __shared__ double part[8][8];
  for (int b = blockIdx.y; b < nbox; b += gridDim.y) {
    const long long p0 = boff[b], p1 = boff[b + 1];
    if (p0 + blockIdx.x * (long long)blockDim.x >= p1) continue;
    const long long nown = box[b].nown;
    double val[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (long long p = p0 + blockIdx.x * (long long)blockDim.x + threadIdx.x; p < p1;
         p += (long long)gridDim.x * blockDim.x) {
      const unsigned int i = perm[p];
      const float4 a = facc[p];
      a_in[i] = a;
      if ((long long)i - p0 >= nown) continue;   // a halo particle: summed by its owner
      const float4 vv = vel4[p];
      const double m = widen_any(cen4[p].w);
      const double vx = widen_any(vv.x), vy = widen_any(vv.y), vz = widen_any(vv.z);
      const double ax = widen_any(a.x), ay = widen_any(a.y), az = widen_any(a.z);
      val[0] += m * ax;
      val[1] += m * ay;
      val[2] += m * az;
      val[3] += m * (vx * ax + vy * ay + vz * az + widen_any(a.w));
      val[4] += m * vx;
      val[5] += m * vy;
      val[6] += m * vz;
      val[7] += m * (0.5 * (vx * vx + vy * vy + vz * vz) + widen_any(vv.w));
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      double v = val[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) part[w][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < 8) {
      double v = 0.0;
      for (int q = 0; q < (int)(blockDim.x >> 5); ++q) v += part[q][threadIdx.x];
      atomicAdd(&red[8 * b + threadIdx.x], v);
    }
    __syncthreads();
  }
}

// =========================================================================== time stepping
// caller-order (a, du/dt) into the saved accelerations: which = 0 sets a (n x 3), 1 sets du/dt
__global__ void k_set_acc(long long off, long long n, int which, const float* __restrict__ src,
                          float4* __restrict__ a_in) {
  pdl_wait();
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
    float4 a = a_in[off + q];
    if (which == 0) {
      a.x = src[3 * q];
      a.y = src[3 * q + 1];
      a.z = src[3 * q + 2];
    } else {
      a.w = src[q];
    }
    a_in[off + q] = a;
  }
}

void launch_set_acc(Engine& E, long long off, long long n, int which, const float* src) {
  launch_pdl(k_set_acc, E.grid(n), 256, E.st, off, n, which, src, E.a_in.p); count_launch();
}

// half kick with the box's dt: v += a dt/2, u += du/dt dt/2 (u kept >= 0)
__global__ void k_kick(long long N, const int* __restrict__ bid, const BoxDesc* __restrict__ box,
                       const float4* __restrict__ a_in, float* __restrict__ v, float* __restrict__ u) {
  pdl_wait();
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const float hdt = (float)(0.5 * box[bid[i]].dt);      // (kept from round to round it held the loads up: 0.26 -> 0.54 ms)
    if (hdt == 0.0f) continue;
    const float4 a = a_in[i];
    v[3 * i] += a.x * hdt;
    v[3 * i + 1] += a.y * hdt;
    v[3 * i + 2] += a.z * hdt;
    u[i] = fmaxf(u[i] + a.w * hdt, 0.0f);
  }
}

// drift in FP64 with the box's dt, wrapped into [0, L) (periodic) or clamped (open).
// The h iteration of the new step then starts from the extrapolation of the
// last roots of N~(h) = N_ngb (hhist x: this step's, written by the ghost pass;
// y, z, w: the three before) to the new time: the polynomial through them, cubic
// once four are known, with the box's weights hc, kept within 10 % of h.  A
// particle's root moves smoothly with its neighbours, so the extrapolation is
// off by a fourth-order term in dt and most particles meet the N~ tolerance in
// the first density pass.  hlev[b] counts the earlier roots a box holds (0..3); it
// restarts at 0 when the box's h is set to other values.  Without a history y, z,
// w take the current h.
__global__ void k_drift(long long N, const int* __restrict__ bid, const BoxDesc* __restrict__ box,
                        double* __restrict__ x, const float* __restrict__ v, float* __restrict__ h,
                        float4* __restrict__ hhist, const int* __restrict__ hlev) {
  pdl_wait();
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < N; p += (long long)gridDim.x * blockDim.x) {
    const int b = bid[p];
    const BoxDesc& bd = box[b];
    if (bd.dt == 0.0) continue;
    const float hc = h[p];
    float4 hh = hhist[p];
    const int lev = hlev[b];
    if (lev > 0) {
      const float* w = bd.hw[lev];
      const float hn = fmaf(w[0], hh.x, fmaf(w[1], hh.y, fmaf(w[2], hh.z, w[3] * hh.w)));
      h[p] = fminf(fmaxf(hn, 0.9f * hc), 1.1f * hc);
      hh.w = hh.z;
      hh.z = hh.y;
      hh.y = hh.x;
    } else {
      hh.y = hc;
      hh.z = hc;
      hh.w = hc;
    }
    hhist[p] = hh;
    for (int k = 0; k < 3; ++k) {
      double xn = x[3 * p + k] + (double)v[3 * p + k] * bd.dt;
      // inside by more than the rounding of x / L: nothing to wrap or clamp
      if (dbits(xn) + 16 < dbits(bd.L)) {
      } else if (bd.periodic) {
        xn -= bd.L * floor(xn * bd.invL);
        if (xn >= bd.L) xn -= bd.L;
        if (xn < 0.0 || xn >= bd.L) xn = 0.0;
      } else {
        xn = fmin(fmax(xn, 0.0), nextafter(bd.L, 0.0));
      }
      x[3 * p + k] = xn;
    }
  }
}

// =========================================================================== FP32 peak
// Independent FMA chains (8 per thread) with no memory traffic between the first
// load and the final store: the FP32 pipe's throughput.  The store depends on
// every chain so the compiler keeps them.
__global__ void __launch_bounds__(256) k_fma_peak(int iters, float a, float b, float* __restrict__ out) {
  pdl_wait();
  float v[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = (float)(threadIdx.x + k) * 1e-3f;
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = fmaf(v[k], a, b);
  }
  float s = 0.0f;
#pragma unroll
  for (int k = 0; k < 8; ++k) s += v[k];
  if (s == 12345.678f) out[blockIdx.x] = s;   // practically never: keeps the chains live
}

double measure_fp32_peak(cudaStream_t st, int nsm, float* scratch) {
  const int blocks = nsm * 8, threads = 256, iters = 8192;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  k_fma_peak<<<blocks, threads, 0, st>>>(iters, 0.9999f, 1e-4f, scratch); count_launch();
  cudaEventRecord(e0, st);
  k_fma_peak<<<blocks, threads, 0, st>>>(iters, 0.9999f, 1e-4f, scratch); count_launch();
  cudaEventRecord(e1, st);
  cudaEventSynchronize(e1);
  float ms = 0.0f;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  const double flops = 2.0 * 8.0 * iters * (double)blocks * threads;
  return ms > 0.0f ? flops / (ms * 1e-3) / 1e12 : 0.0;
}

// =========================================================================== outputs
// Write field `field` of the particles of one box [off, off + n) in caller order.
__global__ void k_get_field(long long off, long long n, int field, const unsigned int* __restrict__ perm,
                            const float* __restrict__ Hs, const float4* __restrict__ cen4,
                            const float4* __restrict__ vel4, const float4* __restrict__ dacc,
                            const unsigned int* __restrict__ dcnt, const float4* __restrict__ ghost4,
                            const float4* __restrict__ facc, const float* __restrict__ fvsig,
                            const unsigned int* __restrict__ fcnt, const float* __restrict__ h, float gamma_gas,
                            void* out) {
  pdl_wait();
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
    const long long p = off + q;
    const long long i = (long long)perm[p] - off;
    const float H = Hs[p];
    const float ih = 1.0f / H;
    const float K3 = SPH_KNORM * ih * ih * ih;
    const float4 a = dacc[p];
    const float m = cen4[p].w;
    float* fo = reinterpret_cast<float*>(out);
    switch (field) {
      case SPH_FIELD_RHO: fo[i] = K3 * (a.x + m); break;
      case SPH_FIELD_DRHO_DH: fo[i] = -K3 * fmaf(3.0f, a.x + m, a.y) / h[perm[p]]; break;
      case SPH_FIELD_NW: fo[i] = K3 * (a.z + 1.0f); break;
      case SPH_FIELD_NNGB: fo[i] = (32.0f / 3.0f) * (a.z + 1.0f); break;
      case SPH_FIELD_COUNT: reinterpret_cast<int*>(out)[i] = (int)dcnt[p]; break;
      case SPH_FIELD_P: fo[i] = (gamma_gas - 1.0f) * ghost4[p].x * vel4[p].w; break;
      case SPH_FIELD_C: fo[i] = ghost4[p].z; break;
      case SPH_FIELD_F: fo[i] = a.y < 0.0f ? -3.0f * (a.x + m) / a.y : 1.0f; break;   // as the ghost pass
      case SPH_FIELD_A: {
        const float4 f = facc[p];
        fo[3 * i] = f.x;
        fo[3 * i + 1] = f.y;
        fo[3 * i + 2] = f.z;
        break;
      }
      case SPH_FIELD_DUDT: fo[i] = facc[p].w; break;
      case SPH_FIELD_VSIG: fo[i] = fvsig[p]; break;
      case SPH_FIELD_FORCE_COUNT: reinterpret_cast<int*>(out)[i] = (int)fcnt[p]; break;
      default: break;
    }
  }
}

// =========================================================================== launchers
// CTAs of a kernel resident per SM at SPH_THREADS threads (looked up once; engines
// may run in several host threads)
static int resident_ctas(const void* fn) {
  static std::mutex mu;
  static const void* fns[16] = {nullptr};   // the 10 density, 2 gathered density and 3 force instances
  static int val[16] = {0};
  std::lock_guard<std::mutex> lock(mu);
  for (int k = 0; k < 16; ++k) {
    if (fns[k] == fn) return val[k];
    if (!fns[k]) {
      int nb = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, SPH_THREADS, 0) != cudaSuccess || nb < 1) nb = 4;
      fns[k] = fn;
      val[k] = nb;
      return nb;
    }
  }
  return 4;
}

void launch_live_tasks(Engine& E) {
  if (!E.rec_for_force().pool) return;     // the passes walk their clusters' interactions (with pair records they list their tasks)
  cudaMemsetAsync(E.Lq.n_live, 0, sizeof(unsigned int), E.st);
  const long long n = E.n_ptasks + E.n_stasks;
  if (n == 0) return;
  launch_pdl(k_live_tasks, (int)std::min<long long>((n + 255) / 256, (long long)E.nsm * 16), 256, E.st, E.Lq, E.T, E.TL,
             E.box.p, E.n_ptasks, E.n_stasks);
  count_launch();
}

// One density pass.  The kernel instance (first pass or later pass) follows the
// iteration counter it_dev when given, else E.partial_pass.  only: the instance
// the caller knows the pass needs (-1: both, as in a captured step, where the
// one that does not match the counter returns at once).
void launch_density(Engine& E, const int* it_dev, int only) {
  for (int part = 0; part < 2; ++part) {
    if (!it_dev && part != (E.partial_pass ? 1 : 0)) continue;
    if (it_dev && only >= 0 && part != only) continue;
    const bool kahan = E.kahan();
    // the first pass records its pairs for the force pass when the records are on
    const bool rec = part == 0 && E.rec_for_force().pool != nullptr;
    decltype(&k_density<false, false, false, false>) k;
    if (kahan)
      k = E.count_pairs ? (part ? k_density<true, true, true, false>
                                : (rec ? k_density<true, false, true, true> : k_density<true, false, true, false>))
                        : (part ? k_density<false, true, true, false> : k_density<false, false, true, false>);
    else
      k = E.count_pairs ? (part ? k_density<true, true, false, false>
                                : (rec ? k_density<true, false, false, true> : k_density<true, false, false, false>))
                        : (part ? k_density<false, true, false, false> : k_density<false, false, false, false>);
    launch_pdl(k, E.nsm * resident_ctas((const void*)k), SPH_THREADS, E.st,
        E.Lq, E.T, E.TL, E.box.p, E.pos4.p, E.cen4.p, E.sort_r.p, E.sort_i.p, E.act.p, E.perm.p, E.x.p, E.dacc.p,
        E.dcnt.p, E.dcomp.p, E.pc.p, E.task_ctr.p + part, E.partial_pass, it_dev, it_dev ? E.gflag.p : nullptr,
        (unsigned int)(E.gcap ? E.N : E.n_tiles),
        E.gcap ? reinterpret_cast<const unsigned int*>(E.dev_counters.p + 4) : nullptr,
        E.unit_list ? E.units.p : nullptr, E.n_units.p, (unsigned int)E.units.n, E.rec_for_force());
    count_launch();
  }
}

// The packing of a gathered later pass (a pass of the h
// iteration given by it_dev; the kernels decide on the device whether it gathers).
void launch_gather_prep(Engine& E, const int* it_dev) {
  if (E.prm.h_gather == 0 || E.count_pairs) return;      // (gflag stays 0: no pass gathers)
  // a captured rebuild step covers the capacities (this build's sizes are on the device)
  const long long nt = E.gcap ? E.N : E.n_tiles;
  const unsigned int* ntd = E.gcap ? reinterpret_cast<const unsigned int*>(E.dev_counters.p + 4) : nullptr;
  if (E.N <= PACK_ONE) {
    launch_pack_scan(E, nt, ntd, it_dev);
  } else {
    exclusive_scan(E.pk_cnt.p, E.pk_cnt.p, nt + 1, E.pk_sums.p, E.pk_tot.p + 0, E.st, ntd, it_dev);
    launch_pdl(k_pack_leaf, E.grid(nt + 1), 256, E.st, nt, ntd, it_dev, E.T, E.TL, E.pk_cnt.p, E.pk_v.p);
    count_launch();
    exclusive_scan(E.pk_v.p, E.pk_v.p, nt + 1, E.pk_sums.p, E.pk_tot.p + 1, E.st, ntd, it_dev);
  }
  launch_pdl(k_pack_fill, E.grid(32 * nt), 256, E.st, nt, ntd, it_dev, (long long)E.N, E.T, E.TL, E.act.p, E.pk_cnt.p,
             E.pk_v.p, E.pk_tot.p, E.pk_idx.p, E.pk_info.p, E.pk_n.p, E.gflag.p);
  count_launch();
}

// The gathered density pass; returns at once unless the pass gathers.
void launch_density_gather(Engine& E) {
  const bool kahan = E.kahan();
  const auto k = kahan ? k_density_gather<true> : k_density_gather<false>;
  launch_pdl(k, E.nsm * resident_ctas((const void*)k), SPH_THREADS, E.st, E.Lq, E.T, E.TL, E.box.p, E.pos4.p,
             E.cen4.p, E.sort_r.p, E.sort_i.p, E.perm.p, E.x.p, E.dacc.p, E.dcnt.p, E.dcomp.p, E.g_n.p, E.gflag.p,
             E.pk_info.p, E.pk_n.p, E.pk_idx.p, E.pk_tot.p, E.task_ctr.p + 3);
  count_launch();
}

void launch_force(Engine& E) {
  const bool rec = E.rec_for_force().pool != nullptr;
  const auto k = E.count_pairs ? (rec ? k_force<true, true> : k_force<true, false>) : k_force<false, false>;
  cudaMemsetAsync(E.task_ctr.p + 2, 0, sizeof(unsigned int), E.st);
  launch_pdl(k, E.nsm * resident_ctas((const void*)k), SPH_THREADS, E.st,
      E.Lq, E.T, E.TL, E.box.p, E.pos4.p, E.cen4.p, E.vel4.p, E.ghost4.p, E.sort_r.p, E.sort_i.p, E.perm.p, E.x.p,
      E.prm.alpha_visc, E.facc.p, E.fvsig.p, E.fcnt.p, E.pc.p, E.task_ctr.p + 2,
      (unsigned int)(E.gcap ? E.N : E.n_tiles),
      E.gcap ? reinterpret_cast<const unsigned int*>(E.dev_counters.p + 4) : nullptr,
      E.unit_list ? E.units.p : nullptr, E.n_units.p, (unsigned int)E.units.n, E.rec_for_force());
  count_launch();
}

// The unit list of a decomposition (built with it; see k_unit_list).
void launch_unit_list(Engine& E) {
  if (!E.unit_list) return;
  cudaMemsetAsync(E.n_units.p, 0, sizeof(unsigned int), E.st);
  const long long nt = E.gcap ? E.N : E.n_tiles;
  launch_pdl(k_unit_list, E.grid(32 * nt), 256, E.st, (unsigned int)nt,
             E.gcap ? reinterpret_cast<const unsigned int*>(E.dev_counters.p + 4) : nullptr, E.Lq, E.T, E.TL, E.box.p,
             E.units.p, E.n_units.p, (unsigned int)E.units.n);
  count_launch();
}

void launch_ghost(Engine& E, int mode, int it, const int* it_dev) {
  launch_pdl(k_ghost, E.grid(E.N), 256, E.st, E.N, mode, it, it_dev, E.prm.h_max_iter, E.prm.gamma_kernel, E.prm.n_ngb,
                                          E.prm.h_tol, E.prm.gamma_gas, E.perm.p, E.Hs.p, E.pos4.p, E.cen4.p,
                                          E.vel4.p, E.dacc.p, E.dcnt.p, E.dcomp.p, E.act.p, E.h.p, E.hlo.p, E.hhi.p, E.conv.p,
                                          E.hlimp.p, E.leaf_of.p, E.T, E.ghost4.p, E.hhist.p, E.dev_counters.p,
                                          E.err_all.p, (long long)(E.gcap ? E.cap_nodes : E.n_nodes),
                                          (long long)(E.gcap ? E.N : E.n_tiles), E.t_active.p, E.tl_active.p, E.t_alo.p,
                                          E.t_ahi.p); count_launch();
}

void launch_pass_setup(Engine& E, bool brackets, bool errors, int it) {
  E.partial_pass = 0;
  launch_pdl(k_pass_setup, E.grid(E.N), 256, E.st, E.N, E.act.p, E.dacc.p, E.dcnt.p, E.dcomp.p,
             brackets ? E.hlo.p : nullptr, E.hhi.p, E.conv.p, (long long)(E.gcap ? E.cap_nodes : E.n_nodes),
             E.t_active.p, (long long)(E.gcap ? E.N : E.n_tiles), E.tl_active.p, E.task_ctr.p, E.dev_counters.p,
             errors ? E.err_all.p : nullptr, E.gflag.p, E.it_dev.p, it, E.g_n.p);
  count_launch();
}

void launch_count_unconverged(Engine& E, int* out) {
  launch_pdl(k_count_unconverged, E.grid(E.N), 256, E.st, E.N, E.conv.p, out); count_launch();
}

void launch_mark_active_cells(Engine& E) {
  E.partial_pass = 1;
  // a captured rebuild step covers the capacities (this build's sizes are on the device)
  const long long nt = E.gcap ? E.N : E.n_tiles;
  launch_pdl(k_mark_active, E.grid(32 * nt), 256, E.st, nt,
             E.gcap ? reinterpret_cast<const unsigned int*>(E.dev_counters.p + 4) : nullptr, E.act.p, E.pos4.p, E.T,
             E.TL, E.pk_cnt.p, E.rec_for_force().pool ? 1 : 0);
  count_launch();
}

void launch_task_offsets(Engine& E) {
  launch_pdl(k_task_tiles, E.grid(E.cap_pair + E.cap_self), 256, E.st, E.Lq, E.T, E.cap_pair, E.cap_self); count_launch();
  exclusive_scan(E.Lq.p_toff, E.Lq.p_toff, E.cap_pair, E.scan_tmp.p,
                 reinterpret_cast<unsigned int*>(E.Lq.counts + 6), E.st);
  exclusive_scan(E.Lq.s_toff, E.Lq.s_toff, E.cap_self, E.scan_tmp.p,
                 reinterpret_cast<unsigned int*>(E.Lq.counts + 7), E.st);
}

void launch_task_items(Engine& E) {
  launch_pdl(k_task_items, E.nsm * 8, 256, E.st, E.Lq, E.T, E.n_pairs, E.n_selfs, (unsigned int)E.l_ptask.n, (unsigned int)E.l_stask.n);
  count_launch();
}

void launch_reduce(Engine& E) {
  cudaMemsetAsync(E.red.p, 0, sizeof(double) * 8 * E.nbox, E.st);
  long long maxn = 1;
  for (int b = 0; b < E.nbox; ++b) maxn = std::max(maxn, E.spec[b].n);
  // blocks enough for the largest box alone (a small one's others return at once): shared
  // out evenly, the largest of twelve boxes had a twelfth of them and took 74 us
  const int gx = (int)std::max<long long>(1, std::min<long long>((maxn + 255) / 256, std::max(E.nsm * 4 / E.nbox, std::min(E.nsm * 4, 65536 / E.nbox))));
  launch_pdl(k_reduce, dim3(gx, std::min(E.nbox, 65535)), 256, E.st, E.nbox, E.boff.p, E.box.p, E.perm.p, E.cen4.p,
             E.vel4.p, E.facc.p,
                                                                 E.a_in.p, E.red.p); count_launch();
}

cudaError_t add_cond_set_node(cudaGraphNode_t* node, cudaGraph_t g, const cudaGraphNode_t* deps, size_t ndeps,
                              cudaGraphConditionalHandle h, const int* flag) {
  cudaKernelNodeParams kp = {};
  void* args[2] = {&h, &flag};
  kp.func = (void*)k_cond_set;
  kp.gridDim = dim3(1);
  kp.blockDim = dim3(1);
  kp.sharedMemBytes = 0;
  kp.kernelParams = args;
  kp.extra = nullptr;
  return cudaGraphAddKernelNode(node, g, deps, ndeps, &kp);
}

void launch_cond_keep(Engine& E, cudaGraphConditionalHandle keep) {
  launch_pdl(k_cond_keep, 1, 1, E.st, keep, E.reuse_flag.p); count_launch();
}

void launch_iter_start(Engine& E, cudaGraphConditionalHandle iter) {
  launch_pdl(k_iter_start, 1, 1, E.st, iter, E.it_dev.p); count_launch();
}

void launch_iter_step(Engine& E) {
  launch_pdl(k_iter_step, 1, 1, E.st, E.it_dev.p, E.dev_counters.p, E.err_all.p, E.prm.h_max_iter,
             E.task_ctr.p); count_launch();
}

void launch_iter_next(Engine& E, cudaGraphConditionalHandle iter, cudaGraphConditionalHandle force) {
  launch_pdl(k_iter_next, 1, 1, E.st, iter, force, E.it_dev.p, E.dev_counters.p, E.err_all.p, E.prm.h_max_iter,
                                 E.it_dev.p + 1, E.task_ctr.p); count_launch();
}

void launch_set_drift(Engine& E) {
  launch_pdl(k_set_drift, 1, 256, E.st, E.nbox, E.box.p, E.dmax_bits.p); count_launch();
}

void launch_kick(Engine& E) { launch_pdl(k_kick, E.grid(E.N), 256, E.st, E.N, E.bid.p, E.box.p, E.a_in.p, E.v.p, E.u.p); count_launch(); }

// one more root kept by every moving box (the ghost pass of the step writes it)
__global__ void k_hlev_next(int nbox, const BoxDesc* __restrict__ box, int* __restrict__ hlev) {
  pdl_wait();
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += gridDim.x * blockDim.x)
    if (box[b].dt != 0.0) hlev[b] = min(hlev[b] + 1, 3);
}

// history levels of the boxes of a new layout: a moved box keeps its own
__global__ void k_remap_hlev(int nbox, const long long* __restrict__ src_tab, const int* __restrict__ old_lev,
                             int* __restrict__ lev) {
  pdl_wait();
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += gridDim.x * blockDim.x) {
    const long long s = src_tab[b];
    lev[b] = s >= 0 ? old_lev[s] : 0;
  }
}

// h of one box set from src (device); the box's root history restarts when any h changes
__global__ void k_set_h(long long n, const float* __restrict__ src, float* __restrict__ h, int* __restrict__ hlev) {
  pdl_wait();
  bool diff = false;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float s = src[i];
    diff |= __float_as_uint(s) != __float_as_uint(h[i]);
    h[i] = s;
  }
  if (__syncthreads_or(diff) && threadIdx.x == 0) *hlev = 0;
}

void launch_drift(Engine& E) {
  launch_pdl(k_drift, E.grid(E.N), 256, E.st, E.N, E.bid.p, E.box.p, E.x.p, E.v.p, E.h.p, E.hhist.p, E.hlev.p);
  count_launch();
  launch_pdl(k_hlev_next, 1, 256, E.st, E.nbox, E.box.p, E.hlev.p); count_launch();
}

// The particles of a small box from device arrays, in one launch (five copies and the
// kernel above take 30 us for 4096 particles, this 15).
__global__ void k_set_particles(long long n, const double* __restrict__ xs, const float* __restrict__ vs,
                                const float* __restrict__ ms, const float* __restrict__ us,
                                const float* __restrict__ hs, double* __restrict__ x, float* __restrict__ v,
                                float* __restrict__ m, float* __restrict__ u, float* __restrict__ h,
                                int* __restrict__ hlev) {
  pdl_wait();
  const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, nth = (long long)gridDim.x * blockDim.x;
  bool diff = false;
  for (long long i = t0; i < 3 * n; i += nth) {
    x[i] = xs[i];
    v[i] = vs[i];
    if (i < n) {
      m[i] = ms[i];
      u[i] = us[i];
      const float s = hs[i];
      diff |= __float_as_uint(s) != __float_as_uint(h[i]);
      h[i] = s;
    }
  }
  if (__syncthreads_or(diff) && threadIdx.x == 0) *hlev = 0;
}

void launch_set_particles(Engine& E, int b, const double* x, const float* v, const float* m, const float* u,
                          const float* h) {
  const long long n = E.spec[b].n, o = E.off[b];
  launch_pdl(k_set_particles, E.grid(3 * n), 256, E.st, n, x, v, m, u, h, E.x.p + 3 * o, E.v.p + 3 * o, E.m.p + o,
             E.u.p + o, E.h.p + o, E.hlev.p + b);
  count_launch();
}

void launch_set_h(Engine& E, int b, const float* src) {
  const long long n = E.spec[b].n;
  if (n == 0) return;
  launch_pdl(k_set_h, E.grid(n), 256, E.st, n, src, E.h.p + E.off[b], E.hlev.p + b); count_launch();
}

// The accelerations and du/dt of the last force pass from their copy in caller order,
// which needs no scatter (1.28 and 0.57 ms for 33.5M particles through the permutation).
__global__ void k_get_acc(long long off, long long n, int field, const float4* __restrict__ a_in, float* __restrict__ out) {
  pdl_wait();
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
    const float4 a = a_in[off + q];
    if (field == SPH_FIELD_DUDT) {
      out[q] = a.w;
    } else {
      out[3 * q] = a.x;
      out[3 * q + 1] = a.y;
      out[3 * q + 2] = a.z;
    }
  }
}

void launch_get_field(Engine& E, long long off, long long n, int field, void* out) {
  if ((field == SPH_FIELD_A || field == SPH_FIELD_DUDT) && !E.acc_edited) {
    launch_pdl(k_get_acc, E.grid(n), 256, E.st, off, n, field, E.a_in.p, reinterpret_cast<float*>(out));
    count_launch();
    return;
  }
  launch_pdl(k_get_field, E.grid(n), 256, E.st, off, n, field, E.perm.p, E.Hs.p, E.cen4.p, E.vel4.p, E.dacc.p, E.dcnt.p,
                                           E.ghost4.p, E.facc.p, E.fvsig.p, E.fcnt.p, E.h.p, E.prm.gamma_gas, out);
  count_launch();
}

}  // namespace sph

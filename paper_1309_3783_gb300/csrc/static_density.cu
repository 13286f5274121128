// Density pass that allocates nothing, for callers that cannot call cudaMalloc.
//
// Some callers run where device allocation is not allowed: inside an
// allocator-free embedding (a pre-sized arena owned by someone else), from code
// that must not trigger the driver's allocator after start-up, or where every
// allocation has to be accounted for up front.  sph_density_static serves them:
// it takes device pointers for its inputs and outputs and keeps all of its
// working memory in one fixed device array that exists from the moment the
// library is loaded, so no call allocates.
//
// The working memory is the static array below: a uniform cell list of the box (cell
// offsets, and the particles sorted by cell).  One cluster of thread blocks checks the
// inputs and builds it; then a warp per particle evaluates rho_i = sum_{r_ij < H_i} m_j W(r_ij,
// H_i) (j = i included) and the neighbour count over the whole chip, with the neighbour
// decision r_ij < H taken in FP64 in the same fixed evaluation order as the main path's
// exact decision, so counts match it bit for bit.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>

#include "sph.h"
#include "sph_internal.cuh"

namespace {

constexpr int kMaxN = SPH_STATIC_MAX_N;           // particles per call
constexpr int kMaxSide = 20;                      // cells per dimension of the cell list (its counts fit shared memory)
constexpr int kMaxCells = kMaxSide * kMaxSide * kMaxSide;
constexpr int kThreads = 1024;                    // per block of the cluster that builds the cell list
constexpr int kBlocks = 8;                        // blocks of that cluster
constexpr int kPer = kMaxN / (kThreads * kBlocks);   // particles per thread of it
static_assert(kPer * kThreads * kBlocks == kMaxN, "every particle has a thread");
constexpr int kWarps = 4;                         // warps (particles) per block of the density kernel

// The working memory: the particles sorted by cell as (position about the box centre
// in units of L, mass), their indices, the exclusive cell offsets, the side of the
// cell list and the status of the call.
struct Scratch {
  float4 pos[kMaxN];
  unsigned int order[kMaxN];
  unsigned int cells[kMaxCells + 1];
  int side;
  int status;
};

// The working memory: held by every device that loads the library, for the
// life of the process.  Host code must not use this name as a device address.
static __device__ __align__(256) Scratch g_scratch;

// Device address of g_scratch per device, looked up once per device.  Host
// threads that make their first calls at the same time may each look it up; they
// store the same value, through atomics.
static std::atomic<Scratch*> g_scratch_ptr[64];

// Cell of a coordinate about the box centre in units of L.  Its FP32 rounding may put
// a particle next to its cell's border into the next cell; the cells' edge allows for it.
__device__ __forceinline__ int cell_of(float u, int side) {
  return min(max((int)floorf((u + 0.5f) * (float)side), 0), side - 1);
}

// Input checks and cell list: one cluster of 8 blocks, a thread per particle or two,
// which stay in registers; counts and fill cursors live in the first block's shared
// memory.  (FP64 runs at 2 lanes per clock and SM here: one block spent 60 us on the
// conversions and cell indices of 4096 particles; the checks are integer comparisons
// and the indices FP32.)
__global__ void __cluster_dims__(kBlocks, 1, 1) __launch_bounds__(kThreads)
    k_static_cells(const double* __restrict__ x, const float* __restrict__ m, const float* __restrict__ h, int n,
                   double L, int periodic, float gamma_k, Scratch* __restrict__ ws) {
  namespace cg = cooperative_groups;
  __shared__ unsigned int s_cnt[kMaxCells];
  __shared__ unsigned int s_tmp[kThreads / 32];
  __shared__ float s_h[kThreads / 32];
  __shared__ float s_hall[kBlocks];
  __shared__ int s_badall[kBlocks];
  __shared__ int s_side;
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, rank = (int)cl.block_rank();
  unsigned int* cnt0 = cl.map_shared_rank(s_cnt, 0);
  // input checks (those of the main path's ingest: 0 <= x < L, by the order of the
  // bit patterns, h and m finite and positive) and the largest support radius
  const unsigned long long Lbits = (unsigned long long)__double_as_longlong(L);
  const double invL = 1.0 / L;
  float hm = 0.0f;
  bool bad = false;
  float4 u[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int i = (k * kBlocks + rank) * kThreads + tid;
    if (i >= n) break;
    const float hi = h[i], mi = m[i];
    const double xi[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
    for (int d = 0; d < 3; ++d) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(xi[d]);
      bad |= !(b < Lbits || b == 0x8000000000000000ull);
    }
    bad |= !(isfinite(hi) && hi > 0.0f) || !(isfinite(mi) && mi > 0.0f);
    hm = fmaxf(hm, __fmul_rn(gamma_k, hi));
    u[k] = make_float4((float)fma(xi[0], invL, -0.5), (float)fma(xi[1], invL, -0.5), (float)fma(xi[2], invL, -0.5), mi);
  }
  hm = warp_max(hm);
  if (lane == 0) s_h[w] = hm;
  const int block_bad = __syncthreads_or(bad ? 1 : 0);
  if (w == 0) {
    hm = warp_max(s_h[lane]);
    if (lane < kBlocks) {
      cl.map_shared_rank(s_hall, lane)[rank] = hm;
      cl.map_shared_rank(s_badall, lane)[rank] = block_bad;
    }
  }
  if (rank == 0)
    for (int c = tid; c < kMaxCells; c += kThreads) s_cnt[c] = 0;
  cl.sync();
  if (tid == 0) {
    int any_bad = 0;
    hm = 0.0f;
    for (int b = 0; b < kBlocks; ++b) {
      hm = fmaxf(hm, s_hall[b]);
      any_bad |= s_badall[b];
    }
    int side = 1, status = 0;
    if (any_bad || !(hm > 0.0f) || !isfinite(hm)) {
      status = SPH_E_INVALID;
    } else if (periodic && !(floor(L / ((double)hm * (1.0 + 1e-9))) >= 3.0)) {
      status = SPH_E_H_TOO_LARGE;      // (a relative margin far above the rounding of the quotient)
    } else {
      // cells of edge >= H_max and the rounding of a cell index; 3 per dimension of a
      // periodic box are all of it, whatever their edge
      const double sd = floor(1.0 / ((double)hm * invL + 1e-6));
      side = sd > (double)kMaxSide ? kMaxSide : max((int)sd, periodic ? 3 : 1);
    }
    if (rank == 0) {
      ws->side = side;
      ws->status = status;
    }
    s_side = status == 0 ? side : 0;
  }
  __syncthreads();
  const int side = s_side;
  if (side == 0) return;      // (every block)
  const int ncell = side * side * side;
  int cell[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    if ((k * kBlocks + rank) * kThreads + tid >= n) break;
    cell[k] = (cell_of(u[k].z, side) * side + cell_of(u[k].y, side)) * side + cell_of(u[k].x, side);
    atomicAdd(&cnt0[cell[k]], 1u);
  }
  cl.sync();
  if (rank == 0) {
    // exclusive scan: every thread a run of cells, then the runs' sums over the block
    const int per = (ncell + kThreads - 1) / kThreads;
    const int c0 = min(tid * per, ncell), c1 = min(c0 + per, ncell);
    unsigned int sum = 0;
    for (int c = c0; c < c1; ++c) sum += s_cnt[c];
    unsigned int incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_tmp[w] = incl;
    __syncthreads();
    if (w == 0) {
      unsigned int t = s_tmp[lane];
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned int y = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += y;
      }
      s_tmp[lane] = t;
    }
    __syncthreads();
    unsigned int at = (w > 0 ? s_tmp[w - 1] : 0u) + incl - sum;
    for (int c = c0; c < c1; ++c) {
      const unsigned int v = s_cnt[c];
      ws->cells[c] = at;
      s_cnt[c] = at;          // from here on the cell's fill cursor
      at += v;
    }
    if (tid == 0) ws->cells[ncell] = (unsigned int)n;
  }
  cl.sync();
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int i = (k * kBlocks + rank) * kThreads + tid;
    if (i >= n) break;
    const unsigned int o = atomicAdd(&cnt0[cell[k]], 1u);
    ws->order[o] = (unsigned int)i;
    ws->pos[o] = u[k];
  }
  cl.sync();                  // (the first block's shared memory stays until all are done)
}

// Density of the particles, a warp each, in cell order: its lanes take the particles
// of the 27 cells (runs of adjacent cells per row) and drop those out of reach in FP32;
// the others are gathered in a list, and full warps of them decided and evaluated from
// FP64 distances.  FP64 runs at 1/60 of the FP32 rate here, so only the pairs that are
// neighbours (one candidate in eight in a uniform box), or within rounding of one,
// take it, and of them only the subtractions, squares and sums.
// FP32 distances in units of L are off by less than 4e-7 (two positions rounded to
// 2^-25, three differences below 1 rounded to 2^-25 twice, their squares' sum to a few
// 2^-24 of itself): REACH covers it.
// The call took 15.4 ms for 4096 particles and 59 ms for 16384 as one block with every
// candidate in FP64; it takes 52 and 105 us, a third of it the host's share.  (Built by
// one block in FP64, the cell list alone made these 95 and 254 us.)
constexpr float REACH = 1e-6f;

__global__ void __launch_bounds__(32 * kWarps) k_static_density(const double* __restrict__ x,
                                                                const float* __restrict__ h, int n, double L,
                                                                double invL, int periodic, float gamma_k, float* __restrict__ rho,
                                                                int* __restrict__ count,
                                                                const Scratch* __restrict__ ws) {
  pdl_wait();
  __shared__ unsigned int s_list[kWarps][64];
  if (ws->status != 0) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int at = blockIdx.x * kWarps + w;
  if (at >= n) return;
  const int side = ws->side;
  const float4 pi = ws->pos[at];
  const unsigned int i = ws->order[at];
  const double xi[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
  const float Hi = __fmul_rn(gamma_k, h[i]), invH = 1.0f / Hi;
  const unsigned long long h2 = (unsigned long long)__double_as_longlong(__dmul_rn((double)Hi, (double)Hi));   // exact
  const float reach = __double2float_ru((double)Hi * invL) + REACH;
  const float reach2 = reach * reach * 1.000001f;
  // H = Hn 2^eh with Hn in [1, 2) (a subnormal H too)
  const int eh = ilogbf(Hi);
  const float invHn = 1.0f / scalbnf(Hi, -eh);
  // the runs of cells: lane 2 r + p has part p of row r (a periodic row that leaves
  // the box has two parts)
  unsigned int lo = 0, len = 0;
  {
    const int cx = cell_of(pi.x, side), r = lane >> 1;
    int cy = cell_of(pi.y, side) + r % 3 - 1, cz = cell_of(pi.z, side) + r / 3 - 1;
    if (periodic) {
      cy = (cy + side) % side;
      cz = (cz + side) % side;
    }
    int a = max(cx - 1, 0), b = min(cx + 1, side - 1);
    bool on = r < 9 && cy >= 0 && cz >= 0 && cy < side && cz < side;
    if (lane & 1) {
      on = on && periodic && (cx == 0 || cx == side - 1);
      a = b = cx == 0 ? side - 1 : 0;
    }
    if (on) {
      const int row = (cz * side + cy) * side;
      lo = ws->cells[row + a];
      len = ws->cells[row + b + 1] - lo;
    }
  }
  float sw = 0.0f;
  int cnt = 0;
  unsigned int held = 0;       // listed candidates not yet decided
  const auto decide = [&](bool on, unsigned int q) {
    if (!on) return;
    const unsigned int j = ws->order[q];
    const float4 pj = ws->pos[q];
    // canonical_r2; a component is within rounding of L/2 only in pairs beyond reach
    // (H <= L / 3), so FP32 tells which image is the nearest
    const float du[3] = {pi.x - pj.x, pi.y - pj.y, pi.z - pj.z};
    double d[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      d[k] = __dsub_rn(xi[k], x[3 * (size_t)j + k]);
      if (periodic) {
        if (du[k] > 0.5f) d[k] = __dsub_rn(d[k], L);
        else if (du[k] < -0.5f) d[k] = __dadd_rn(d[k], L);
      }
    }
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
    const unsigned long long b2 = (unsigned long long)__double_as_longlong(r2);
    if (!(b2 < h2)) return;      // r2 < H^2: the order of their bit patterns
    // r / 2^eh to FP32 rounding: r2 / 2^(2 eh) split into its leading 24 bits and the
    // other 29, the root of the first corrected once for both
    const int e = (int)(b2 >> 52) - 1023 - 2 * eh;
    float rn = 0.0f;
    if (e > -70) {      // (below, the kernel is 1 to rounding)
      const float hi = __uint_as_float(((unsigned int)(e + 127) << 23) | ((unsigned int)(b2 >> 29) & 0x7fffffu));
      const float lo = (float)((unsigned int)b2 & 0x1fffffffu) * __uint_as_float((unsigned int)(e - 52 + 127) << 23);
      const float rt = sqrtf(hi);
      rn = rt + (fmaf(-rt, rt, hi) + lo) / (2.0f * rt);
    }
    const float qn = rn * invHn;
    float wq, dw;
    spline_w_dw(qn, wq, dw);
    sw = fmaf(pj.w, wq, sw);
    ++cnt;
  };
  for (unsigned int runs = __ballot_sync(0xffffffffu, len != 0u); runs; runs &= runs - 1) {
    const int l = __ffs(runs) - 1;
    const unsigned int b = __shfl_sync(0xffffffffu, lo, l), e = b + __shfl_sync(0xffffffffu, len, l);
    for (unsigned int q0 = b; q0 < e; q0 += 32) {
      const unsigned int q = q0 + lane;
      bool near = false;
      if (q < e) {
        const float4 pj = ws->pos[q];
        float dx = fabsf(pi.x - pj.x), dy = fabsf(pi.y - pj.y), dz = fabsf(pi.z - pj.z);
        if (periodic) {
          dx = fminf(dx, 1.0f - dx);
          dy = fminf(dy, 1.0f - dy);
          dz = fminf(dz, 1.0f - dz);
        }
        near = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= reach2 && q != (unsigned int)at;
      }
      const unsigned int bal = __ballot_sync(0xffffffffu, near);
      if (near) s_list[w][held + __popc(bal & ((1u << lane) - 1u))] = q;
      held += __popc(bal);
      __syncwarp();
      if (held >= 32u) {
        decide(true, s_list[w][lane]);
        held -= 32u;
        const unsigned int rest = s_list[w][32 + lane];
        __syncwarp();
        s_list[w][lane] = rest;
        __syncwarp();
      }
    }
  }
  decide((unsigned int)lane < held, s_list[w][lane]);
  sw = warp_sum(sw);
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) {
    const float K3 = SPH_KNORM * invH * invH * invH;
    rho[i] = K3 * (sw + pi.w);
    count[i] = cnt;
  }
}

}  // namespace

extern "C" sph_status sph_density_static(const double* x, const float* m, const float* h, int64_t n, double box_len,
                                         int periodic, float* rho, int32_t* count, void* stream) {
  if (!x || !m || !h || !rho || !count || !(box_len > 0)) return SPH_E_INVALID;
  if (n < 1 || n > kMaxN) return SPH_E_INVALID;      // beyond the static working memory
  if (!std::isfinite(box_len)) return SPH_E_INVALID;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SPH_E_CUDA;
  Scratch* ws = g_scratch_ptr[dev].load(std::memory_order_acquire);
  if (!ws) {
    // first call on this device: look up the array's device address (call it
    // before any stream capture)
    Scratch* ptr = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_scratch) != cudaSuccess || !ptr) return SPH_E_CUDA;
    g_scratch_ptr[dev].store(ptr, std::memory_order_release);
    ws = ptr;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int ni = (int)n, per = periodic ? 1 : 0;
  k_static_cells<<<kBlocks, kThreads, 0, st>>>(x, m, h, ni, box_len, per, SPH_STATIC_GAMMA_K, ws);
  if (cudaGetLastError() != cudaSuccess) return SPH_E_CUDA;
  if (launch_pdl(k_static_density, (ni + kWarps - 1) / kWarps, 32 * kWarps, st, x, h, ni, box_len, 1.0 / box_len, per,
                 SPH_STATIC_GAMMA_K, rho, count, static_cast<const Scratch*>(ws)) != cudaSuccess)
    return SPH_E_CUDA;
  int hs = 0;
  if (cudaMemcpyAsync(&hs, &ws->status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return SPH_E_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return SPH_E_CUDA;
  return hs == 0 ? SPH_OK : (sph_status)hs;
}

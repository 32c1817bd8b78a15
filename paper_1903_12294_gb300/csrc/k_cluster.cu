// The paper's multifaceted 4D clustering (§3.2) over the resident dataset: k_i centres seeded on
// a 4D rectilinear grid (§3.2.1), every field and point sample assigned to a centre, centres
// moved to the means of their samples, samples reassigned by D_f = w_f |f_s - f_c| + w_d S_st and
// D_p = w_p |p_s - p_c| + w_d S_st among the centres whose 2C search region holds them (§3.2.3),
// until no centre value changes by more than eps_c relative (§3.2.2).
//
//   k_slic_valid    samples that take part, and the largest |value| of each kind (fixed-point
//                   scales for the centre sums)
//   k_slic_seed     centres at the grid cells' centres
//   k_slic_assign_* the best centre of every sample among its candidates, and the sample's
//                   fixed-point contribution to that centre's sums: the first pass one thread
//                   per sample; later field passes a tile of voxels of one step per block, later
//                   point passes one cell's grouped samples per block (k_slic_pgroup groups them
//                   once), both against a shared candidate list that every warp cuts down to the
//                   centres its own samples can reach
//   k_slic_update   one thread per centre: means of its sums, counts, change test
//   k_slic_cells*   centres sorted into the cells of the seed grid for the next assignment
//
// Candidates: a centre whose search region holds a sample lies within C_i of it along every
// axis, so its cell is the sample's cell or a neighbour (cells are the seed grid, size C_i). A
// centre within a small margin of a cell border is filed in the neighbouring cell as well, so
// rounding in the cell computation cannot lose it. The first assignment takes the nearest seed
// by S_st; the seeds are the cells' centres, so it is among the sample's cell and neighbours.
//
// Every decision is taken in IEEE fp32 with the operations in a fixed order (no contraction),
// ties to the lower centre index; centre sums are exact int64 fixed point and the means are
// formed in fp64 from them, so the result does not depend on the order of the atomics.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "msf_internal.cuh"

namespace msf {

int scan_exclusive_u32(msf_ctx* ctx, const uint32_t* in, uint32_t* out, int64_t n, DevBuf& tmp,
                       uint32_t* total);

// How the approximate scan forms a distance: sqrt(k2 * (dx^2 + dy^2 + dz^2) + kt * dt^2) + |dv|,
// the distance divided by the value's weight (values == false, a zero weight: |dv| is left out and
// nothing divided). ok == false: the weights are outside what its error bound covers.
struct ScanScale {
  float k2, kt, slack;
  bool ok, values;
};

struct SlicArgs {
  int nx, ny, nz, T, A;
  int64_t V, P;
  int t0, tw;
  int j0, nj;                   // the window's point steps [j0, j0 + nj)
  int attr;
  int k[4];
  float C[4];
  float w_p, w_f, w_d, c_f, eps_c;
  int kpos, kf, kp;
  int K;
  const float* field;
  const float* pos;
  const float* attrp;
  const int32_t* key;
  const int32_t* fstep;         // [Tp] field step of each point step
  const int32_t* pj0;           // [T + 1] first point step of each field step
  float* centers;               // [K][6] x, y, z, t, p_c, f_c
  float* prev;                  // [K][6]
  unsigned long long* sums;     // [K][8] x, y, z, t, p, f, n_field, n_point
  long long* counts;            // [K][2]
  uint32_t* cell_start;         // [K + 1] (cells = seed grid)
  uint32_t* cell_cursor;        // [K]
  uint32_t* cell_items;         // [16 K]
  int32_t* flabel;              // [tw][V]
  int32_t* plabel;              // [nj][P]
  unsigned* moved;
  unsigned long long* valid;    // [0] samples, [1] max|f| bits, [2] max|p| bits
  uint32_t* pcell_start;        // [K * nsub + 1] first slot of each subcell's point samples
  uint32_t* pcell_cursor;       // [K * nsub]
  float4* psample;              // [slots] x, y, z, value of the point sample in the slot
  float* ptime;                 // [slots] its time
  uint32_t* pindex;             // [slots] its index t * P + p in the window (t: point step)
  int sub[4], nsub;             // subcells of a cell along x, y, z, t, and their number
  bool plain;                   // sizes and scales the packed sums allow
  ScanScale scan_f, scan_p;     // the approximate scan of the field and of the point samples
};

// Time of window point step t: with r point steps in field step f, the i-th (0-based) sits at
// f + (i + 0.5) / r, spreading them evenly over the field step's unit of time (one per field
// step: f + 0.5, as a field sample of step f).
__device__ __forceinline__ float point_time(const SlicArgs& a, int t) {
  const int j = a.j0 + t;
  const int f = __ldg(a.fstep + j);
  const int p0 = __ldg(a.pj0 + f), r = __ldg(a.pj0 + f + 1) - p0;
  return __fadd_rn((float)f, __fdiv_rn(__fadd_rn((float)(j - p0), 0.5f), (float)r));
}

constexpr float kCellMargin = 1e-3f;

__device__ __forceinline__ float s_st(const float* c, float xs, float ys, float zs, float ts,
                                      float cf) {
  const float dx = __fsub_rn(c[0], xs), dy = __fsub_rn(c[1], ys), dz = __fsub_rn(c[2], zs);
  const float dt = __fmul_rn(cf, __fsub_rn(c[3], ts));
  const float s = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)),
                                      __fmul_rn(dz, dz)),
                            __fmul_rn(dt, dt));
  return __fsqrt_rn(s);
}

__device__ __forceinline__ bool in_region(const float* c, const float* C, float xs, float ys,
                                          float zs, float ts) {
  return fabsf(__fsub_rn(xs, c[0])) <= C[0] && fabsf(__fsub_rn(ys, c[1])) <= C[1] &&
         fabsf(__fsub_rn(zs, c[2])) <= C[2] && fabsf(__fsub_rn(ts, c[3])) <= C[3];
}

// cell along one axis: floor(u / C) clamped to [0, k)
__device__ __forceinline__ int cell_of(float u, float C, int k) {
  const int c = (int)floorf(__fdiv_rn(u, C));
  return min(max(c, 0), k - 1);
}

__device__ __forceinline__ bool better(float d, int c, float bd, int bc) {
  return bc < 0 || d < bd || (d == bd && c < bc);
}

// ---- sums of one warp's samples into their centres -------------------------------------------
// v[0..4]: fixed-point x, y, z, t and the value; slot: 4 (point value) or 5 (field value).
__device__ __forceinline__ void warp_accumulate(unsigned long long* sums, int best,
                                                const long long* v, int slot) {
  const bool ok = best >= 0;
  const unsigned act = __ballot_sync(0xFFFFFFFFu, ok);
  if (!act) return;
  const int lane = threadIdx.x & 31, first = __ffs(act) - 1;
  const int b0 = __shfl_sync(0xFFFFFFFFu, best, first);
  const int cslot = slot == 5 ? 6 : 7;
  if (__all_sync(0xFFFFFFFFu, !ok || best == b0)) {
    unsigned long long tot[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const unsigned long long u = ok ? (unsigned long long)v[q] : 0ull;
      const uint32_t s0 = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(u & 0x1FFFFFull));
      const uint32_t s1 = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)((u >> 21) & 0x1FFFFFull));
      const uint32_t s2 = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(u >> 42));
      tot[q] = (unsigned long long)s0 + ((unsigned long long)s1 << 21) +
               ((unsigned long long)s2 << 42);
    }
    if (lane == first) {
      unsigned long long* s = sums + 8 * (int64_t)b0;
#pragma unroll
      for (int q = 0; q < 4; ++q) atomicAdd(s + q, tot[q]);
      atomicAdd(s + slot, tot[4]);
      atomicAdd(s + cslot, (unsigned long long)__popc(act));
    }
    return;
  }
  if (!ok) return;
  const unsigned grp = __match_any_sync(act, best);
  const int leader = __ffs(grp) - 1;
  unsigned long long tot[5] = {0ull, 0ull, 0ull, 0ull, 0ull};
  for (unsigned m = grp; m; m &= m - 1) {
    const int src = __ffs(m) - 1;
#pragma unroll
    for (int q = 0; q < 5; ++q) tot[q] += (unsigned long long)__shfl_sync(grp, v[q], src);
  }
  if (lane == leader) {
    unsigned long long* s = sums + 8 * (int64_t)best;
#pragma unroll
    for (int q = 0; q < 4; ++q) atomicAdd(s + q, tot[q]);
    atomicAdd(s + slot, tot[4]);
    atomicAdd(s + cslot, (unsigned long long)__popc(grp));
  }
}

// ---- samples that take part, and value ranges ------------------------------------------------
__global__ void __launch_bounds__(256) k_slic_valid(const __grid_constant__ SlicArgs a) {
  const int64_t nf = (int64_t)a.tw * a.V, np = (int64_t)a.nj * a.P;
  unsigned long long n = 0;
  unsigned fm = 0, pm = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nf + np;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (i < nf) {
      const float f = __ldg(a.field + (int64_t)a.t0 * a.V + i);
      if (isfinite(f)) {
        ++n;
        fm = max(fm, __float_as_uint(fabsf(f)));
      }
    } else {
      const int64_t j = i - nf, t = j / a.P, p = j - t * a.P;
      const float v = __ldg(a.attrp + ((a.j0 + t) * a.A + a.attr) * a.P + p);
      if (__ldg(a.key + (a.j0 + t) * a.P + p) >= 0 && isfinite(v)) {
        ++n;
        pm = max(pm, __float_as_uint(fabsf(v)));
      }
    }
  }
  n = __reduce_add_sync(0xFFFFFFFFu, (unsigned)n);
  fm = __reduce_max_sync(0xFFFFFFFFu, fm);
  pm = __reduce_max_sync(0xFFFFFFFFu, pm);
  if ((threadIdx.x & 31) == 0) {
    if (n) atomicAdd(a.valid, n);
    if (fm) atomicMax(reinterpret_cast<unsigned*>(a.valid + 1), fm);
    if (pm) atomicMax(reinterpret_cast<unsigned*>(a.valid + 2), pm);
  }
}

// ---- seeds -----------------------------------------------------------------------------------
__global__ void k_slic_seed(const __grid_constant__ SlicArgs a) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= a.K) return;
  const int i = c % a.k[0], j = (c / a.k[0]) % a.k[1], l = (c / (a.k[0] * a.k[1])) % a.k[2];
  const int m = c / (a.k[0] * a.k[1] * a.k[2]);
  float* cc = a.centers + 6 * (int64_t)c;
  cc[0] = __fmul_rn(__fadd_rn((float)i, 0.5f), a.C[0]);
  cc[1] = __fmul_rn(__fadd_rn((float)j, 0.5f), a.C[1]);
  cc[2] = __fmul_rn(__fadd_rn((float)l, 0.5f), a.C[2]);
  cc[3] = __fadd_rn((float)a.t0, __fmul_rn(__fadd_rn((float)m, 0.5f), a.C[3]));
  cc[4] = 0.f;
  cc[5] = 0.f;
  for (int q = 0; q < 8; ++q) a.sums[8 * (int64_t)c + q] = 0ull;
}

// ---- the best centre of one sample -------------------------------------------------------------
// Smallest D among the filed centres of the sample's cell and its neighbours whose search region
// holds the sample (-1: none).
__device__ __forceinline__ int best_centre(const SlicArgs& a, float xs, float ys, float zs,
                                           float ts, float w, float vs, int vslot) {
  const int ci = cell_of(xs, a.C[0], a.k[0]), cj = cell_of(ys, a.C[1], a.k[1]);
  const int cl = cell_of(zs, a.C[2], a.k[2]);
  const int cm = cell_of(__fsub_rn(ts, (float)a.t0), a.C[3], a.k[3]);
  int bc = -1;
  float bd = 0.f;
  for (int m = max(cm - 1, 0); m <= min(cm + 1, a.k[3] - 1); ++m)
    for (int l = max(cl - 1, 0); l <= min(cl + 1, a.k[2] - 1); ++l)
      for (int j = max(cj - 1, 0); j <= min(cj + 1, a.k[1] - 1); ++j)
        for (int i = max(ci - 1, 0); i <= min(ci + 1, a.k[0] - 1); ++i) {
          const int cell = ((m * a.k[2] + l) * a.k[1] + j) * a.k[0] + i;
          const uint32_t e = __ldg(a.cell_start + cell + 1);
          for (uint32_t q = __ldg(a.cell_start + cell); q < e; ++q) {
            const int c = (int)__ldg(a.cell_items + q);
            const float* cc = a.centers + 6 * (int64_t)c;
            if (!in_region(cc, a.C, xs, ys, zs, ts)) continue;
            const float d = __fadd_rn(__fmul_rn(w, fabsf(__fsub_rn(vs, cc[vslot]))),
                                      __fmul_rn(a.w_d, s_st(cc, xs, ys, zs, ts, a.c_f)));
            if (better(d, c, bd, bc)) {
              bd = d;
              bc = c;
            }
          }
        }
  return bc;
}

// Coordinate of the seeds of grid index i along axis q (as k_slic_seed forms it).
__device__ __forceinline__ float seed_coord(const SlicArgs& a, int q, int i) {
  const float u = __fmul_rn(__fadd_rn((float)i, 0.5f), a.C[q]);
  return q == 3 ? __fadd_rn((float)a.t0, u) : u;
}

// First assignment: the nearest seed by S_st, the lowest index on a tie. The seeds are a grid, so
// S_st^2 is a sum of one term per axis, added in a fixed order, and rounded additions and square
// root never decrease: the smallest distance is that of the axes' smallest terms, each at the
// sample's grid index or a neighbour, and a tie at a lower index of one axis exists exactly when
// it does with the other axes at their smallest (the later ones) or at the index already taken
// (the earlier ones). So the axes are walked down from the nearest index, the slowest-running
// one first, as long as the distance stays the same: mostly not at all. Computing the 81
// distances of the neighbourhood was a tenth of a ten-update clustering.
__device__ __forceinline__ int nearest_seed(const SlicArgs& a, float xs, float ys, float zs,
                                            float ts) {
  const float u[4] = {xs, ys, zs, ts};
  auto term = [&](int q, int i) {
    float d = __fsub_rn(seed_coord(a, q, i), u[q]);
    if (q == 3) d = __fmul_rn(a.c_f, d);
    return __fmul_rn(d, d);
  };
  auto sum = [](const float (&e)[4]) {
    return __fadd_rn(__fadd_rn(__fadd_rn(e[0], e[1]), e[2]), e[3]);
  };
  int at[4];
  float e[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = cell_of(q == 3 ? __fsub_rn(ts, (float)a.t0) : u[q], a.C[q], a.k[q]);
    at[q] = c;
    e[q] = term(q, c);
    const float lo = c > 0 ? term(q, c - 1) : INFINITY;
    const float hi = c + 1 < a.k[q] ? term(q, c + 1) : INFINITY;
    if (lo <= e[q] && c > 0) {
      at[q] = c - 1;
      e[q] = lo;
    }
    if (hi < e[q]) {
      at[q] = c + 1;
      e[q] = hi;
    }
  }
  const float smin = sum(e), dmin = __fsqrt_rn(smin), most = __fmaf_rn(smin, 1e-6f, smin);
#pragma unroll
  for (int q = 3; q >= 0; --q)
    while (at[q] > 0) {
      const float keep = e[q];
      e[q] = term(q, at[q] - 1);
      const float s2 = sum(e);
      if (!(s2 <= most) || __fsqrt_rn(s2) != dmin) {
        e[q] = keep;
        break;
      }
      --at[q];
    }
  return ((at[3] * a.k[2] + at[2]) * a.k[1] + at[1]) * a.k[0] + at[0];
}

__global__ void __launch_bounds__(256, 4) k_slic_assign_field(const __grid_constant__ SlicArgs a) {
  const int64_t n = (int64_t)a.tw * a.V;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t li = base + threadIdx.x;
    int best = -1;
    long long v[5] = {0, 0, 0, 0, 0};
    if (li < n) {
      const uint32_t t = (uint32_t)li / (uint32_t)a.V, vox = (uint32_t)li - t * (uint32_t)a.V;
      const uint32_t yz = vox / (uint32_t)a.nx, x = vox - yz * (uint32_t)a.nx;
      const uint32_t z = yz / (uint32_t)a.ny, y = yz - z * (uint32_t)a.ny;
      const float f = __ldg(a.field + (int64_t)a.t0 * a.V + li);
      if (isfinite(f)) {
        const float xs = __fadd_rn((float)(int)x, 0.5f), ys = __fadd_rn((float)(int)y, 0.5f);
        const float zs = __fadd_rn((float)(int)z, 0.5f);
        const float ts = __fadd_rn((float)(a.t0 + (int)t), 0.5f);
        best = nearest_seed(a, xs, ys, zs, ts);
        v[0] = quantise(xs, a.kpos);
        v[1] = quantise(ys, a.kpos);
        v[2] = quantise(zs, a.kpos);
        v[3] = quantise(ts, a.kpos);
        v[4] = quantise(f, a.kf);
      }
      a.flabel[li] = best;
    }
    warp_accumulate(a.sums, best, v, 5);
  }
}

// ---- later assignments: shared candidate lists ----------------------------------------------
// The centres filed in the cells around a block's samples (a tile of field voxels of one step, or
// a cell's point samples) are gathered into shared memory once. A warp's samples are close to
// each other, so it copies the centres whose search region reaches the box of its samples into a
// list of its own (the box test is the region test at the box's nearest point, in the same
// rounded operations, so it never drops a centre that some sample's test would pass) and every
// lane scans that.
//
// Only the arg-min is needed, not the distance: the scan uses an approximate distance (fused
// operations and the hardware's approximate square root, within 2^-20 of the rounded sequence
// that decides; the region test is exact) and keeps the two smallest. When the second exceeds the
// first by more than 4e-6 of it, the first is the answer; otherwise, and with weights or values
// that the error bound does not cover, the lane scans the list again with the deciding
// operations. 54 to 81 candidates in the deciding operations, an IEEE square root each, bounded
// the passes by instruction issue, and the scan still does: it divides the distance by the value's
// weight (no multiplication after the root), lets the root flush denormals (an absolute error
// that the slack of the comparison covers) and takes two steps or two centres per packed fp32
// instruction.
//
// Sums: a sample adds to its centre's place in shared memory, and the block commits each place
// once (adding up in the warp took a loop over the members of every group with 64-bit shuffles).
//
// 128^3 x 32 field and 1M x 32 point samples, 16,384 centres, ten assignments: field 68.2 -> 34.0
// ms, points 60.2 -> 18.2 ms; in packed operations 18.1 -> 16.9 and 18.2 -> 16.2 ms.
constexpr int kCand = 384;   // centres in a block's list; more: the per-sample lookup
constexpr int kWCand = 96;   // centres in a warp's list; more: the warp scans the block's list

struct CandList {
  float4 pos[kCand];   // x, y, z, t
  float val[kCand];    // the value the pass compares
  int id[kCand];
};

struct __align__(16) WarpList {    // two centres side by side
  float xy[kWCand / 2][4], zt[kWCand / 2][4];  // x, x, y, y; z, z, t, t
  float val[kWCand];
  uint16_t q[kWCand];  // place in the block's list
};
static_assert(kWCand % 2 == 0, "the list is padded to pairs");

// distance between u and the nearest point of [lo, hi], in the rounding of the region test
__device__ __forceinline__ float box_dist(float u, float lo, float hi) {
  return u < lo ? __fsub_rn(lo, u) : u > hi ? __fsub_rn(u, hi) : 0.f;
}

// centre q of the block's list, when it reaches the box, into the warp's list; returns the
// number listed (-1: too many; an odd list is padded with a centre out of reach). All lanes.
__device__ __forceinline__ int warp_list(const SlicArgs& a, const CandList& c, int nc, WarpList& w,
                                         const float (&lo)[4], const float (&hi)[4], bool values) {
  const int lane = threadIdx.x & 31;
  int n = 0;
  for (int b = 0; b < nc; b += 32) {
    const int q = b + lane;
    bool in = q < nc;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    if (in) {
      p = c.pos[q];
      in = box_dist(p.x, lo[0], hi[0]) <= a.C[0] && box_dist(p.y, lo[1], hi[1]) <= a.C[1] &&
           box_dist(p.z, lo[2], hi[2]) <= a.C[2] && box_dist(p.w, lo[3], hi[3]) <= a.C[3];
    }
    const unsigned m = __ballot_sync(0xFFFFFFFFu, in);
    const int at = n + __popc(m & ((1u << lane) - 1u));
    n += __popc(m);
    if (n > kWCand) return -1;  // warp-uniform
    if (in) {
      const int h = at >> 1, o = at & 1;
      w.xy[h][o] = p.x, w.xy[h][2 + o] = p.y;
      w.zt[h][o] = p.z, w.zt[h][2 + o] = p.w;
      w.val[at] = values ? c.val[q] : __fmul_rn(0.f, c.val[q]);  // (a NaN stays one)
      w.q[at] = (uint16_t)q;
    }
  }
  if ((n & 1) && lane == 0) {
    w.xy[n >> 1][1] = w.xy[n >> 1][3] = w.zt[n >> 1][1] = w.zt[n >> 1][3] = INFINITY;
    w.val[n] = 0.f;
  }
  __syncwarp();
  return n;
}

// place in the block's list of the best centre among n listed ones by the deciding operations
// (list: the warp's places, or null for the whole block's list), or -1
__device__ __noinline__ int exact_best(const SlicArgs& a, const CandList& c, const uint16_t* list,
                                          int n, float xs, float ys, float zs, float ts, float wv,
                                          float vs) {
  int best = -1, bc = -1;
  float bd = 0.f;
  for (int i = 0; i < n; ++i) {
    const int q = list ? (int)list[i] : i;
    const float4 p = c.pos[q];
    const float cc[4] = {p.x, p.y, p.z, p.w};
    if (!in_region(cc, a.C, xs, ys, zs, ts)) continue;
    const float d = __fadd_rn(__fmul_rn(wv, fabsf(__fsub_rn(vs, c.val[q]))),
                              __fmul_rn(a.w_d, s_st(cc, xs, ys, zs, ts, a.c_f)));
    if (better(d, c.id[q], bd, bc)) {
      bd = d;
      bc = c.id[q];
      best = q;
    }
  }
  return best;
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// two fp32 values in one 64-bit register pair: packed operations, each rounded as the single one
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
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

// the two smallest so far (m1, m2) and the place of the smallest, with candidate i at distance e
__device__ __forceinline__ void best_two(float e, int i, float& m1, float& m2, int& best) {
  m2 = fminf(m2, fmaxf(m1, e));
  best = e < m1 ? i : best;
  m1 = fminf(m1, e);
}

// does the smallest approximate distance decide?
__device__ __forceinline__ bool decided(const ScanScale& k, float m1, float m2) {
  return m1 < 1e18f && m2 > fmaf(m1, 4e-6f, m1) + k.slack;
}

// the same by the approximate scan of the warp's list where that decides
__device__ __forceinline__ int list_best(const SlicArgs& a, const ScanScale& k, const CandList& c,
                                         const WarpList& w, int n, int nc, float xs, float ys,
                                         float zs, float ts, float wv, float vs) {
  if (n < 0) return exact_best(a, c, nullptr, nc, xs, ys, zs, ts, wv, vs);
  if (!k.ok) return exact_best(a, c, w.q, n, xs, ys, zs, ts, wv, vs);
  const float C0 = a.C[0], C1 = a.C[1], C2 = a.C[2], C3 = a.C[3];
  const f32x2 nx = pack2(-xs, -xs), ny = pack2(-ys, -ys), nz = pack2(-zs, -zs);
  const f32x2 nt = pack2(-ts, -ts), nv = k.values ? pack2(-vs, -vs) : 0ull;
  const f32x2 k2 = pack2(k.k2, k.k2), kt = pack2(k.kt, k.kt);
  float m1 = INFINITY, m2 = INFINITY;
  int best = -1;
#pragma unroll 2
  for (int i = 0; i < n; i += 2) {
    const ulonglong2 xy = *reinterpret_cast<const ulonglong2*>(w.xy[i >> 1]);
    const ulonglong2 zt = *reinterpret_cast<const ulonglong2*>(w.zt[i >> 1]);
    const f32x2 v = *reinterpret_cast<const f32x2*>(w.val + i);
    const f32x2 dx = add2(xy.x, nx), dy = add2(xy.y, ny), dz = add2(zt.x, nz), dt = add2(zt.y, nt);
    const f32x2 s3 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
    const float2 s = unpack2(fma2(mul2(dt, kt), dt, mul2(s3, k2)));
    const float2 d = unpack2(add2(v, nv));
    const float2 ux = unpack2(dx), uy = unpack2(dy), uz = unpack2(dz), ut = unpack2(dt);
    const bool in0 = fabsf(ux.x) <= C0 && fabsf(uy.x) <= C1 && fabsf(uz.x) <= C2 && fabsf(ut.x) <= C3;
    const bool in1 = fabsf(ux.y) <= C0 && fabsf(uy.y) <= C1 && fabsf(uz.y) <= C2 && fabsf(ut.y) <= C3;
    const float e0 = in0 ? sqrt_approx(s.x) + fabsf(d.x) : INFINITY;
    const float e1 = in1 ? sqrt_approx(s.y) + fabsf(d.y) : INFINITY;
    best_two(e0, i, m1, m2, best);
    best_two(e1, i + 1, m1, m2, best);
  }
  // (no centre in reach, or distances too large: the deciding scan tells)
  if (best >= 0 && decided(k, m1, m2)) return w.q[best];
  return exact_best(a, c, w.q, n, xs, ys, zs, ts, wv, vs);
}

// The filed centres of the cells [lo, lo + nn) into the block's list, except those whose time
// fails the search region for every time in [ta, tb]. Returns their number, -1 for more than
// kCand (or more than 256 cells). One neighbouring cell per thread; all threads.
__device__ __forceinline__ int block_list(const SlicArgs& a, const int (&lo)[4], const int (&nn)[4],
                                          float ta, float tb, int vslot, CandList& c, int* s_warp) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int ncell = nn[0] * nn[1] * nn[2] * nn[3];
  if (ncell > 256) return -1;  // block-uniform
  int cnt = 0, kept = 0;
  uint32_t c0 = 0;
  if (tid < ncell) {
    int q = tid;
    const int i = lo[0] + q % nn[0]; q /= nn[0];
    const int j = lo[1] + q % nn[1]; q /= nn[1];
    const int l = lo[2] + q % nn[2]; q /= nn[2];
    const int m = lo[3] + q;
    const int cell = ((m * a.k[2] + l) * a.k[1] + j) * a.k[0] + i;
    c0 = __ldg(a.cell_start + cell);
    cnt = (int)(__ldg(a.cell_start + cell + 1) - c0);
    for (int r = 0; r < cnt; ++r) {
      const int id = (int)__ldg(a.cell_items + c0 + r);
      kept += box_dist(__ldg(a.centers + 6 * (int64_t)id + 3), ta, tb) <= a.C[3];
    }
  }
  int x = kept;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[w] = x;
  __syncthreads();
  int off = x - kept, total = 0;
  for (int q = 0; q < 8; ++q) {
    const int t = s_warp[q];
    if (q < w) off += t;
    total += t;
  }
  if (total <= kCand)
    for (int q = 0; q < cnt; ++q) {
      const int id = (int)__ldg(a.cell_items + c0 + q);
      const float* cc = a.centers + 6 * (int64_t)id;
      const float ct = __ldg(cc + 3);
      if (!(box_dist(ct, ta, tb) <= a.C[3])) continue;
      c.pos[off] = make_float4(__ldg(cc), __ldg(cc + 1), __ldg(cc + 2), ct);
      c.val[off] = __ldg(cc + vslot);
      c.id[off] = id;
      ++off;
    }
  __syncthreads();
  return total <= kCand ? total : -1;
}

// one sample's sums straight to its centre (no place in the block's list)
__device__ __forceinline__ void commit_sample(unsigned long long* sums, int c, const long long* v,
                                              int slot) {
  unsigned long long* s = sums + 8 * (int64_t)c;
#pragma unroll
  for (int q = 0; q < 4; ++q) atomicAdd(s + q, (unsigned long long)v[q]);
  atomicAdd(s + slot, (unsigned long long)v[4]);
  atomicAdd(s + (slot == 5 ? 6 : 7), 1ull);
}

// 64-bit addition in shared memory as two 32-bit atomics, the carry with the second
__device__ __forceinline__ void add64(uint32_t* p, unsigned long long v) {
  const uint32_t lo = (uint32_t)v, old = atomicAdd(p, lo);
  const uint32_t hi = (uint32_t)(v >> 32) + (old + lo < old ? 1u : 0u);
  if (hi) atomicAdd(p + 1, hi);
}

// Field samples: a tile of TX x TY x TZ voxels (256, 8 x 4 of them per warp) over kFieldSteps
// steps per block. A thread takes its voxel at all of the steps at once: the spatial part of the
// region test and of the distance is the same for them, and so is the list; a listed centre
// carries the squared time term of every step, infinite where its region does not reach the step
// (the time test of the step, in the deciding operations, made once per centre). One step at a
// time the passes took 34.0 ms (ten assignments of 67M samples), so 18.1 ms. A sample's place
// adds its tile coordinates as packed counters: count and x in one word, y and z in another, and
// the steps' sum (1024 samples: no counter exceeds 16 bits). Where four steps together would reach
// more cells or centres than the lists hold (cells of a step or two), two steps go together or one
// (field_steps).
constexpr int kFieldSteps = 4;

template <int S>
struct __align__(16) FieldList {
  float4 pv[kWCand];    // x, y, z, -value
  float dt[kWCand][S];  // kt (t - step)^2, or infinity
  uint16_t q[kWCand];
};

// S: steps a thread has room for, 4 or 2; most: how many of them a tile takes (S = 4: all)
template <int TX, int TY, int TZ, int S>
__global__ void __launch_bounds__(256, 4) k_slic_assign_field_tiled(const __grid_constant__ SlicArgs a,
                                                                    int most) {
  static_assert(TX * TY * TZ == 256 && TX % 8 == 0 && TY % 4 == 0, "8 x 4 voxels per warp");
  static_assert(S == 2 || S == kFieldSteps, "pairs of steps");
  const int steps = S == 2 ? most : S;
  __shared__ CandList s_c;
  __shared__ FieldList<S> s_w[8];
  __shared__ uint32_t s_acc[kCand][5];  // count | x, y | z, step, the value sum's halves
  __shared__ int s_warp[8];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int ntx = (a.nx + TX - 1) / TX, nty = (a.ny + TY - 1) / TY, ntz = (a.nz + TZ - 1) / TZ;
  const int ntt = (a.tw + steps - 1) / steps;
  const int64_t ntiles = (int64_t)ntx * nty * ntz * ntt;
  const int wx = (w % (TX / 8)) * 8, wy = (w / (TX / 8)) % (TY / 4) * 4;
  const int wz = w / ((TX / 8) * (TY / 4));
  const float C0 = a.C[0], C1 = a.C[1], C2 = a.C[2], C3 = a.C[3];
  const ScanScale& k = a.scan_f;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    int64_t r = tile;
    const int bx = (int)(r % ntx); r /= ntx;
    const int by = (int)(r % nty); r /= nty;
    const int bz = (int)(r % ntz);
    const int t0 = (int)(r / ntz) * steps, nt = min(steps, a.tw - t0);
    const int x0 = bx * TX, y0 = by * TY, z0 = bz * TZ;
    auto step_time = [&](int s) { return __fadd_rn((float)(a.t0 + t0 + s), 0.5f); };
    int lo[4], nn[4];
    {
      const int e0[3] = {x0, y0, z0};
      const int e1[3] = {min(x0 + TX, a.nx) - 1, min(y0 + TY, a.ny) - 1, min(z0 + TZ, a.nz) - 1};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float u0 = q < 3 ? __fadd_rn((float)e0[q < 3 ? q : 0], 0.5f)
                               : __fsub_rn(step_time(0), (float)a.t0);
        const float u1 = q < 3 ? __fadd_rn((float)e1[q < 3 ? q : 0], 0.5f)
                               : __fsub_rn(step_time(nt - 1), (float)a.t0);
        lo[q] = max(cell_of(u0, a.C[q], a.k[q]) - 1, 0);
        nn[q] = min(cell_of(u1, a.C[q], a.k[q]) + 1, a.k[q] - 1) - lo[q] + 1;
      }
    }
    const int nc = block_list(a, lo, nn, step_time(0), step_time(nt - 1), 5, s_c, s_warp);
    for (int q = tid; q < nc * 5; q += 256) (&s_acc[0][0])[q] = 0u;
    __syncthreads();
    const int lx = wx + (lane & 7), ly = wy + (lane >> 3), lz = wz;
    const int xv = x0 + lx, yv = y0 + ly, zv = z0 + lz;
    const float xs = __fadd_rn((float)xv, 0.5f), ys = __fadd_rn((float)yv, 0.5f);
    const float zs = __fadd_rn((float)zv, 0.5f);
    // the warp's list: centres whose region reaches the box of its voxels (and some step)
    FieldList<S>& L = s_w[w];
    int n = nc >= 0 ? 0 : -1;
    for (int b = 0; b < nc; b += 32) {
      const int q = b + lane;
      bool in = q < nc;
      float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
      if (in) {
        p = s_c.pos[q];
        in = box_dist(p.x, __fadd_rn((float)(x0 + wx), 0.5f),
                      __fadd_rn((float)(x0 + wx + 7), 0.5f)) <= C0 &&
             box_dist(p.y, __fadd_rn((float)(y0 + wy), 0.5f),
                      __fadd_rn((float)(y0 + wy + 3), 0.5f)) <= C1 &&
             box_dist(p.z, zs, zs) <= C2;
      }
      const unsigned m = __ballot_sync(0xFFFFFFFFu, in);
      const int at = n + __popc(m & ((1u << lane) - 1u));
      n += __popc(m);
      if (n > kWCand) {  // warp-uniform
        n = -1;
        break;
      }
      if (in) {
        const float v = s_c.val[q];
        L.pv[at] = make_float4(p.x, p.y, p.z, k.values ? -v : __fmul_rn(0.f, v));  // (NaN stays)
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const float dt = __fsub_rn(p.w, step_time(s));
          L.dt[at][s] = fabsf(dt) <= C3 ? k.kt * (dt * dt) : INFINITY;
        }
        L.q[at] = (uint16_t)q;
      }
    }
    __syncwarp();
    if (xv < a.nx && yv < a.ny && zv < a.nz) {
      const int64_t l0 = ((int64_t)t0 * a.nz + zv) * a.ny * a.nx + (int64_t)yv * a.nx + xv;
      int old[S];
      float f[S], m1[S], m2[S];
      int best[S];
#pragma unroll
      for (int s = 0; s < S; ++s) {
        old[s] = s < nt ? a.flabel[l0 + s * a.V] : -1;
        f[s] = s < nt ? __ldg(a.field + (int64_t)a.t0 * a.V + l0 + s * a.V) : 0.f;
        m1[s] = m2[s] = INFINITY;
        best[s] = -1;
      }
      if (n >= 0 && k.ok) {
        f32x2 ff[S / 2];
#pragma unroll
        for (int s = 0; s < S; s += 2) ff[s / 2] = k.values ? pack2(f[s], f[s + 1]) : 0ull;
#pragma unroll 2
        for (int i = 0; i < n; ++i) {
          const float4 p = L.pv[i];
          const float dx = __fsub_rn(p.x, xs), dy = __fsub_rn(p.y, ys), dz = __fsub_rn(p.z, zs);
          const bool in = fabsf(dx) <= C0 && fabsf(dy) <= C1 && fabsf(dz) <= C2;
          const float s3 = in ? k.k2 * fmaf(dx, dx, fmaf(dy, dy, dz * dz)) : INFINITY;
          const f32x2 ss = pack2(s3, s3), vv = pack2(p.w, p.w);
#pragma unroll
          for (int s = 0; s < S; s += 2) {
            const float2 s4 = unpack2(add2(ss, *reinterpret_cast<const f32x2*>(&L.dt[i][s])));
            const float2 d = unpack2(add2(ff[s / 2], vv));
            best_two(sqrt_approx(s4.x) + fabsf(d.x), i, m1[s], m2[s], best[s]);
            best_two(sqrt_approx(s4.y) + fabsf(d.y), i, m1[s + 1], m2[s + 1], best[s + 1]);
          }
        }
      }
#pragma unroll
      for (int s = 0; s < S; ++s) {
        if (old[s] < 0) continue;
        const float ts = step_time(s);
        int q, c;
        if (nc < 0) {
          q = -1;
          c = best_centre(a, xs, ys, zs, ts, a.w_f, f[s], 5);
        } else {
          if (best[s] >= 0 && decided(k, m1[s], m2[s]))
            q = L.q[best[s]];
          else
            q = exact_best(a, s_c, n >= 0 ? L.q : nullptr, n >= 0 ? n : nc, xs, ys, zs, ts, a.w_f,
                           f[s]);
          c = q >= 0 ? s_c.id[q] : -1;
        }
        if (c < 0) c = old[s];  // no centre in range: keeps its centre
        a.flabel[l0 + s * a.V] = c;
        const long long qf = quantise(f[s], a.kf);
        if (q >= 0 && a.plain) {
          uint32_t* p = s_acc[q];
          atomicAdd(p, 1u + ((uint32_t)lx << 16));
          atomicAdd(p + 1, (uint32_t)ly + ((uint32_t)lz << 16));
          if (s) atomicAdd(p + 2, (uint32_t)s);
          add64(p + 3, (unsigned long long)qf);
        } else {
          const long long v[5] = {quantise(xs, a.kpos), quantise(ys, a.kpos), quantise(zs, a.kpos),
                                  quantise(ts, a.kpos), qf};
          commit_sample(a.sums, c, v, 5);
        }
      }
    }
    __syncthreads();
    // a place's coordinate sums are sums of (2 x + 1) / 2 at the position scale: exact shifts
    for (int q = tid; q < nc; q += 256) {
      const uint32_t* p = s_acc[q];
      const uint32_t m = p[0] & 0xFFFFu;
      if (!m) continue;
      unsigned long long* sm = a.sums + 8 * (int64_t)s_c.id[q];
      const int e0[4] = {x0, y0, z0, a.t0 + t0};
      const uint32_t l[4] = {p[0] >> 16, p[1] & 0xFFFFu, p[1] >> 16, p[2]};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        atomicAdd(sm + j, (unsigned long long)(2ull * ((unsigned long long)m * e0[j] + l[j]) + m)
                              << (a.kpos - 1));
      atomicAdd(sm + 5, ((unsigned long long)p[4] << 32) | p[3]);
      atomicAdd(sm + 6, (unsigned long long)m);
    }
    __syncthreads();  // the lists are rebuilt for the next tile
  }
}

__global__ void __launch_bounds__(256, 4) k_slic_assign_points(const __grid_constant__ SlicArgs a) {
  const int64_t n = (int64_t)a.nj * a.P;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t li = base + threadIdx.x;
    int best = -1;
    long long v[5] = {0, 0, 0, 0, 0};
    if (li < n) {
      const int t = (int)((uint32_t)li / (uint32_t)a.P);
      const int64_t p = li - (int64_t)t * a.P;
      const int64_t si = (int64_t)(a.j0 + t) * a.P + p;
      const float pv = __ldg(a.attrp + ((int64_t)(a.j0 + t) * a.A + a.attr) * a.P + p);
      if (__ldg(a.key + si) >= 0 && isfinite(pv)) {
        const float* ps = a.pos + (int64_t)(a.j0 + t) * 3 * a.P;
        const float xs = __ldg(ps + p), ys = __ldg(ps + a.P + p), zs = __ldg(ps + 2 * a.P + p);
        const float ts = point_time(a, t);
        best = nearest_seed(a, xs, ys, zs, ts);
        v[0] = quantise(xs, a.kpos);
        v[1] = quantise(ys, a.kpos);
        v[2] = quantise(zs, a.kpos);
        v[3] = quantise(ts, a.kpos);
        v[4] = quantise(pv, a.kp);
      }
      a.plabel[li] = best;
    }
    warp_accumulate(a.sums, best, v, 4);
  }
}

// ---- point samples grouped by cell ----------------------------------------------------------
// The seed-grid cell of a point sample does not change between updates (its position is fixed),
// and every sample of one cell searches the same 3^4 neighbourhood of cells. So the point samples
// that take part are grouped by cell once per call (a counting sort; the order within a group is
// whatever the atomics give, which changes nothing: each sample's result depends on it alone and
// the centre sums are exact), and each update then takes a cell at a time against a shared list
// of its neighbourhood's centres, reading the grouped samples in order. Within a cell they are
// grouped by subcell (halves in space, steps in time), so that the 32 samples of a warp span a
// small box and few of the list's centres reach it. (Field samples are taken in tiles of voxels
// that lie in one cell already, so they need no grouping.)
__device__ __forceinline__ uint32_t sample_cell(const SlicArgs& a, float xs, float ys, float zs,
                                                float ts) {
  const float u[4] = {xs, ys, zs, __fsub_rn(ts, (float)a.t0)};
  int c[4], h[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    c[q] = cell_of(u[q], a.C[q], a.k[q]);
    // the subcell only orders samples: any rounding does
    const float fr = u[q] / a.C[q] - (float)c[q];
    h[q] = min(max((int)(fr * (float)a.sub[q]), 0), a.sub[q] - 1);
  }
  const uint32_t cell = (uint32_t)(((c[3] * a.k[2] + c[2]) * a.k[1] + c[1]) * a.k[0] + c[0]);
  return cell * (uint32_t)a.nsub +
         (uint32_t)(((h[3] * a.sub[2] + h[2]) * a.sub[1] + h[1]) * a.sub[0] + h[0]);
}

// point sample li (taking part after the first assignment): position and value
__device__ __forceinline__ bool point_sample(const SlicArgs& a, int64_t li, float4& s, float& ts) {
  if (a.plabel[li] < 0) return false;
  const int t = (int)((uint32_t)li / (uint32_t)a.P);
  const int64_t p = li - (int64_t)t * a.P;
  const float* ps = a.pos + (int64_t)(a.j0 + t) * 3 * a.P;
  s = make_float4(__ldg(ps + p), __ldg(ps + a.P + p), __ldg(ps + 2 * a.P + p),
                  __ldg(a.attrp + ((int64_t)(a.j0 + t) * a.A + a.attr) * a.P + p));
  ts = point_time(a, t);
  return true;
}

template <bool FILL>
__global__ void __launch_bounds__(256) k_slic_pgroup(const __grid_constant__ SlicArgs a) {
  const int64_t n = (int64_t)a.nj * a.P;
  uint32_t* cursor = a.pcell_cursor;
  for (int64_t li = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; li < n;
       li += (int64_t)gridDim.x * blockDim.x) {
    float4 sm;
    float ts;
    if (!point_sample(a, li, sm, ts)) continue;
    const uint32_t cell = sample_cell(a, sm.x, sm.y, sm.z, ts);
    if (!FILL) {
      atomicAdd(cursor + cell, 1u);
    } else {
      const uint32_t slot = atomicAdd(cursor + cell, 1u);
      a.psample[slot] = sm;
      a.ptime[slot] = ts;
      a.pindex[slot] = (uint32_t)li;
    }
  }
}

// One cell at a time (persistent blocks; grid y splits the samples of a cell where there are few
// cells): its neighbourhood's filed centres into shared memory, then its samples in slot order,
// 32 consecutive ones per warp. A sample's place adds its count and its five fixed-point values.
struct PointAcc {
  uint32_t n[kCand];
  uint32_t v[kCand][10];  // x, y, z, t, value: low and high halves
};

__global__ void __launch_bounds__(256, 4) k_slic_assign_points_cells(const __grid_constant__ SlicArgs a) {
  constexpr int VS = 4;  // the centre's value slot (p_c)
  __shared__ CandList s_c;
  __shared__ WarpList s_w[8];
  __shared__ PointAcc s_acc;
  __shared__ int s_warp[8];
  const int tid = threadIdx.x, w = tid >> 5;
  for (int cell = blockIdx.x; cell < a.K; cell += gridDim.x) {
    const uint32_t first = __ldg(a.pcell_start + (int64_t)cell * a.nsub);
    const uint32_t last = __ldg(a.pcell_start + (int64_t)(cell + 1) * a.nsub);
    if (first + 256u * blockIdx.y >= last) continue;  // block-uniform
    int lo[4], nn[4];
    int q0 = cell;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = q0 % a.k[q];
      q0 /= a.k[q];
      lo[q] = max(c - 1, 0);
      nn[q] = min(c + 1, a.k[q] - 1) - lo[q] + 1;
    }
    const int nc = block_list(a, lo, nn, -INFINITY, INFINITY, VS, s_c, s_warp);
    for (int q = tid; q < nc; q += 256) {
      s_acc.n[q] = 0u;
#pragma unroll
      for (int j = 0; j < 10; ++j) s_acc.v[q][j] = 0u;
    }
    __syncthreads();
    for (uint32_t b0 = first + 256u * blockIdx.y; b0 < last; b0 += 256u * gridDim.y) {
      const uint32_t slot = b0 + tid;
      const bool take = slot < last;
      // (lanes past the end stand in for the last sample, so that they do not widen the box)
      const uint32_t sl = min(slot, last - 1u);
      const float4 sm = a.psample[sl];
      const float ts = a.ptime[sl];
      int n = -1;
      if (nc >= 0) {
        // positions lie inside the grid and times are positive: fp32 bits order like the values
        // (-0 counts as 0)
        const float u[4] = {__fadd_rn(sm.x, 0.f), __fadd_rn(sm.y, 0.f), __fadd_rn(sm.z, 0.f), ts};
        float blo[4], bhi[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          blo[q] = __uint_as_float(__reduce_min_sync(0xFFFFFFFFu, __float_as_uint(u[q])));
          bhi[q] = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(u[q])));
        }
        n = warp_list(a, s_c, nc, s_w[w], blo, bhi, a.scan_p.values);
      }
      if (take) {
        const uint32_t li = a.pindex[slot];
        int q = -1, best;
        if (nc >= 0) {
          q = list_best(a, a.scan_p, s_c, s_w[w], n, nc, sm.x, sm.y, sm.z, ts, a.w_p, sm.w);
          best = q >= 0 ? s_c.id[q] : -1;
        } else {
          best = best_centre(a, sm.x, sm.y, sm.z, ts, a.w_p, sm.w, VS);
        }
        const long long v[5] = {quantise(sm.x, a.kpos), quantise(sm.y, a.kpos),
                                quantise(sm.z, a.kpos), quantise(ts, a.kpos), quantise(sm.w, a.kp)};
        if (best >= 0) a.plabel[li] = best;
        else best = a.plabel[li];  // no centre in range: keeps its centre
        if (q >= 0) {
          atomicAdd(s_acc.n + q, 1u);
#pragma unroll
          for (int j = 0; j < 5; ++j) add64(&s_acc.v[q][2 * j], (unsigned long long)v[j]);
        } else {
          commit_sample(a.sums, best, v, VS);
        }
      }
      __syncwarp();  // the warp's list is rebuilt for its next samples
    }
    __syncthreads();
    for (int q = tid; q < nc; q += 256) {
      const uint32_t m = s_acc.n[q];
      if (!m) continue;
      unsigned long long* sums = a.sums + 8 * (int64_t)s_c.id[q];
#pragma unroll
      for (int j = 0; j < 5; ++j)
        atomicAdd(sums + j,
                  ((unsigned long long)s_acc.v[q][2 * j + 1] << 32) | s_acc.v[q][2 * j]);
      atomicAdd(sums + 7, (unsigned long long)m);
    }
    __syncthreads();  // the lists are rebuilt for the next cell
  }
}

// ---- centre update ---------------------------------------------------------------------------
__device__ __forceinline__ float fixed_mean(long long sum, long long n, int k) {
  double m = __ll2double_rn(sum);
  m = __ddiv_rn(m, __ll2double_rn(n));
  m = __dmul_rn(m, __hiloint2double((1023 - k) << 20, 0));  // * 2^-k (k < 1023)
  return __double2float_rn(m);
}

__global__ void k_slic_update(const __grid_constant__ SlicArgs a, int check) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= a.K) return;
  unsigned long long* s = a.sums + 8 * (int64_t)c;
  float* cc = a.centers + 6 * (int64_t)c;
  float* pv = a.prev + 6 * (int64_t)c;
  const long long nf = (long long)s[6], np = (long long)s[7], n = nf + np;
  float nc[6];
  for (int q = 0; q < 6; ++q) nc[q] = cc[q];
  if (n > 0)
    for (int q = 0; q < 4; ++q) nc[q] = fixed_mean((long long)s[q], n, a.kpos);
  if (np > 0) nc[4] = fixed_mean((long long)s[4], np, a.kp);
  if (nf > 0) nc[5] = fixed_mean((long long)s[5], nf, a.kf);
  bool moved = false;
  for (int q = 0; q < 6; ++q) {
    moved |= !(fabsf(__fsub_rn(nc[q], cc[q])) <= __fmul_rn(a.eps_c, fabsf(cc[q])));
    pv[q] = cc[q];
    cc[q] = nc[q];
  }
  if (check && moved) atomicOr(a.moved, 1u);
  a.counts[2 * c] = nf;
  a.counts[2 * c + 1] = np;
  for (int q = 0; q < 8; ++q) s[q] = 0ull;
}

// ---- centres into cells ----------------------------------------------------------------------
// Cells along one axis that a centre at u is filed in: its own and a neighbour when it lies
// within the margin of the shared border.
__device__ __forceinline__ int axis_cells(float u, float C, int k, int* out) {
  const float r = __fdiv_rn(u, C);
  const int c = (int)floorf(r);
  const float fr = __fsub_rn(r, (float)c);
  int n = 0;
  const int cc = min(max(c, 0), k - 1);
  out[n++] = cc;
  if (fr < kCellMargin && c - 1 >= 0 && c - 1 < k && c - 1 != cc) out[n++] = c - 1;
  if (fr > 1.f - kCellMargin && c + 1 >= 0 && c + 1 < k && c + 1 != cc) out[n++] = c + 1;
  return n;
}

template <bool FILL>
__global__ void k_slic_cells(const __grid_constant__ SlicArgs a) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= a.K) return;
  const float* cc = a.centers + 6 * (int64_t)c;
  int xi[3], yi[3], zi[3], ti[3];
  const int nx = axis_cells(cc[0], a.C[0], a.k[0], xi);
  const int ny = axis_cells(cc[1], a.C[1], a.k[1], yi);
  const int nz = axis_cells(cc[2], a.C[2], a.k[2], zi);
  const int nt = axis_cells(__fsub_rn(cc[3], (float)a.t0), a.C[3], a.k[3], ti);
  for (int m = 0; m < nt; ++m)
    for (int l = 0; l < nz; ++l)
      for (int j = 0; j < ny; ++j)
        for (int i = 0; i < nx; ++i) {
          const int cell = ((ti[m] * a.k[2] + zi[l]) * a.k[1] + yi[j]) * a.k[0] + xi[i];
          if (FILL) {
            const uint32_t at = atomicAdd(a.cell_cursor + cell, 1u);
            a.cell_items[at] = (uint32_t)c;
          } else {
            atomicAdd(a.cell_cursor + cell, 1u);
          }
        }
}

// host side of the fixed-point scale: k = 62 - e - b (max|v| < 2^e, 2^b >= n + 1)
static int fixed_scale_host(double max_abs, long long n) {
  int e = 0;
  if (max_abs > 0) frexp(max_abs, &e);
  int b = 0;
  while ((1ll << b) < n + 1) ++b;
  return 62 - e - b;
}

// Steps of a field tile of TX x TY x TZ voxels: as many as leave its cells within a block's list and
// the centres that a warp's voxels reach (8 x 4 x 1 of them, a centre per cell) within a warp's, with
// some room for centres that have moved together; four where no number does. 64^3 x 8, six
// assignments, cells of 4 x 4 x 4 voxels and one step: four steps (each sample looked up by itself) 3.25
// ms, two 1.27; cells of 8 x 8 x 8 and four steps: four 0.33, two 0.40.
template <int TX, int TY, int TZ>
static int field_steps(const SlicArgs& a) {
  const int tile[3] = {TX - 1, TY - 1, TZ - 1}, warp[3] = {7, 3, 0};
  for (int s = kFieldSteps; s >= 1; s >>= 1) {
    double cells = 1.0, reach = 1.0;
    for (int q = 0; q < 4; ++q) {
      cells *= std::min<double>(a.k[q], std::floor((q < 3 ? tile[q] : s - 1) / (double)a.C[q]) + 3.0);
      reach *= std::min<double>(a.k[q], (q < 3 ? warp[q] : s - 1) / (double)a.C[q] + 2.0);
    }
    if (cells <= 256.0 && reach <= 0.9 * kWCand) return s;
  }
  return kFieldSteps;
}

template <int TX, int TY, int TZ>
static void launch_field_tiled(const SlicArgs& a, unsigned grid, cudaStream_t s) {
  const int steps = field_steps<TX, TY, TZ>(a);
  if (steps == kFieldSteps)
    k_slic_assign_field_tiled<TX, TY, TZ, kFieldSteps><<<grid, 256, 0, s>>>(a, steps);
  else
    k_slic_assign_field_tiled<TX, TY, TZ, 2><<<grid, 256, 0, s>>>(a, steps);
}

int cluster_run(msf_ctx* ctx, const msf_cluster_params* prm, int32_t* flabel, int32_t* plabel,
                float* centers_host, int64_t* counts_host, int* iters) {
  const Dataset& d = ctx->ds;
  ClusterScratch& S = ctx->clu;
  cudaStream_t s = ctx->stream;
  SlicArgs a{};
  a.nx = d.nx;
  a.ny = d.ny;
  a.nz = d.nz;
  a.T = d.T;
  a.A = d.A;
  a.V = d.V;
  a.P = d.A > 0 ? d.P : 0;
  a.t0 = prm->t0;
  a.tw = prm->t1 - prm->t0;
  a.j0 = d.h_pj0[prm->t0];
  a.nj = d.h_pj0[prm->t1] - a.j0;
  a.attr = prm->attr;
  for (int i = 0; i < 4; ++i) a.k[i] = prm->k[i];
  a.K = prm->k[0] * prm->k[1] * prm->k[2] * prm->k[3];
  // C_i = E_i / k_i, IEEE fp32 (the same division on any host)
  volatile float ex[4] = {(float)d.nx, (float)d.ny, (float)d.nz, (float)a.tw};
  for (int i = 0; i < 4; ++i) {
    volatile float ci = ex[i] / (float)prm->k[i];
    a.C[i] = ci;
  }
  a.w_p = prm->w_p;
  a.w_f = prm->w_f;
  a.w_d = prm->w_d;
  a.c_f = prm->c_f;
  a.eps_c = prm->eps_c;
  a.field = d.field.as<float>();
  a.pos = d.pos.as<float>();
  a.attrp = d.attr.as<float>();
  a.key = d.key.as<int32_t>();
  a.fstep = d.fstep.as<int32_t>();
  a.pj0 = d.pj0.as<int32_t>();
  MSF_TRY(S.centers.ensure(sizeof(float) * 6 * (size_t)a.K));
  MSF_TRY(S.prev.ensure(sizeof(float) * 6 * (size_t)a.K));
  MSF_TRY(S.sums.ensure(sizeof(unsigned long long) * 8 * (size_t)a.K));
  MSF_TRY(S.counts.ensure(sizeof(long long) * 2 * (size_t)a.K));
  MSF_TRY(S.cell_start.ensure(sizeof(uint32_t) * ((size_t)a.K + 1)));
  MSF_TRY(S.cell_cursor.ensure(sizeof(uint32_t) * (size_t)a.K));
  MSF_TRY(S.cell_items.ensure(sizeof(uint32_t) * 16 * (size_t)a.K));
  MSF_TRY(S.flags.ensure(sizeof(unsigned long long) * 4));
  a.centers = S.centers.as<float>();
  a.prev = S.prev.as<float>();
  a.sums = S.sums.as<unsigned long long>();
  a.counts = S.counts.as<long long>();
  a.cell_start = S.cell_start.as<uint32_t>();
  a.cell_cursor = S.cell_cursor.as<uint32_t>();
  a.cell_items = S.cell_items.as<uint32_t>();
  a.valid = S.flags.as<unsigned long long>();
  a.moved = reinterpret_cast<unsigned*>(a.valid + 3);
  a.flabel = flabel;
  a.plabel = plabel;
  // fixed-point scales from the samples that take part
  MSF_CUDA_TRY(cudaMemsetAsync(a.valid, 0, sizeof(unsigned long long) * 4, s));
  {
    ScopedKernel k(ctx, "k_slic_valid");
    k_slic_valid<<<ctx->sm_count * 8, 256, 0, s>>>(a);
  }
  unsigned long long hv[3];
  MSF_CUDA_TRY(cudaMemcpyAsync(hv, a.valid, sizeof(hv), cudaMemcpyDeviceToHost, s));
  MSF_CUDA_TRY(cudaStreamSynchronize(s));
  float fmax, pmax;
  const unsigned fb = (unsigned)hv[1], pb = (unsigned)hv[2];
  memcpy(&fmax, &fb, 4);
  memcpy(&pmax, &pb, 4);
  int ext = std::max(std::max(d.nx, d.ny), std::max(d.nz, d.T + 1));
  a.kpos = fixed_scale_host((double)ext, (long long)hv[0]);
  a.kf = fixed_scale_host((double)fmax, (long long)hv[0]);
  a.kp = fixed_scale_host((double)pmax, (long long)hv[0]);
  const unsigned kb = (unsigned)((a.K + 255) / 256);
  const int64_t nfs = (int64_t)a.tw * a.V, nps = (int64_t)a.nj * a.P;
  const unsigned gf = (unsigned)std::min<int64_t>((nfs + 255) / 256, (int64_t)ctx->sm_count * 32);
  const unsigned gp = (unsigned)std::max<int64_t>(1, std::min<int64_t>((nps + 255) / 256,
                                                                       (int64_t)ctx->sm_count * 32));
  const unsigned gt = (unsigned)ctx->sm_count * 8;  // tiled field pass: persistent blocks
  // The approximate scan's error bound wants weights that add up and are not far apart, and
  // distances far from overflow (1e18 and less decide: a squared term that overflows belongs to a
  // larger one). Absolute errors: a root below 2^-63 may be taken as zero, and the deciding
  // operations may lose products to underflow. The packed coordinate sums want voxel centres and
  // their scale to be exact in fp32.
  const bool small = std::max(std::max(d.nx, d.T), std::max(d.ny, d.nz)) <= (1 << 22);
  a.plain = a.kpos >= 1 && small;
  auto scan_scale = [&](float wv) {
    const double k = wv > 0.f ? (double)a.w_d / wv : (double)a.w_d;
    ScanScale r;
    r.k2 = (float)(k * k);
    r.kt = (float)(k * k * ((double)a.c_f * a.c_f));
    r.slack = 1e-18f + (wv > 0.f ? 1e-30f / wv : 0.f);
    r.values = wv > 0.f;
    r.ok = small && a.w_d >= 0.f && (wv == 0.f || (wv >= 1e-9f && wv <= 1e9f)) &&
           (k == 0.0 || (k >= 1e-9 && k <= 1e9)) && (double)r.kt <= 1e30;
    return r;
  };
  a.scan_f = scan_scale(a.w_f);
  a.scan_p = scan_scale(a.w_p);
  k_slic_seed<<<kb, 256, 0, s>>>(a);
  {
    ScopedKernel k(ctx, "k_slic_assign_field");
    k_slic_assign_field<<<gf, 256, 0, s>>>(a);
  }
  if (nps > 0) {
    ScopedKernel k(ctx, "k_slic_assign_points");
    k_slic_assign_points<<<gp, 256, 0, s>>>(a);
  }
  if (nps > 0) {  // the taking-part point samples grouped by cell, for every later assignment
    // subcells: halves of a cell in space, its point steps (up to eight) in time, at most 2^22
    // (or one per cell)
    for (int q = 0; q < 3; ++q) a.sub[q] = a.C[q] > 1.f ? 2 : 1;
    a.sub[3] = std::max(1, std::min(8, a.nj / a.k[3]));
    auto nsub = [&] { return a.sub[0] * a.sub[1] * a.sub[2] * a.sub[3]; };
    for (int q = 3; q >= 0; --q)
      while (a.sub[q] > 1 && (int64_t)a.K * nsub() > (1 << 22)) a.sub[q] >>= 1;
    a.nsub = nsub();
    const size_t ncs = (size_t)a.K * (size_t)a.nsub;
    MSF_TRY(S.pcell_start.ensure(sizeof(uint32_t) * (ncs + 1)));
    MSF_TRY(S.pcell_cursor.ensure(sizeof(uint32_t) * ncs));
    MSF_TRY(S.psample.ensure(sizeof(float4) * (size_t)nps));
    MSF_TRY(S.ptime.ensure(sizeof(float) * (size_t)nps));
    MSF_TRY(S.pindex.ensure(sizeof(uint32_t) * (size_t)nps));
    a.pcell_start = S.pcell_start.as<uint32_t>();
    a.pcell_cursor = S.pcell_cursor.as<uint32_t>();
    a.psample = S.psample.as<float4>();
    a.ptime = S.ptime.as<float>();
    a.pindex = S.pindex.as<uint32_t>();
    ScopedKernel k(ctx, "k_slic_pgroup");
    MSF_CUDA_TRY(cudaMemsetAsync(a.pcell_cursor, 0, sizeof(uint32_t) * ncs, s));
    k_slic_pgroup<false><<<gp, 256, 0, s>>>(a);
    MSF_TRY(scan_exclusive_u32(ctx, a.pcell_cursor, a.pcell_start, (int64_t)ncs, S.scan_tmp,
                               a.pcell_start + ncs));
    MSF_CUDA_TRY(cudaMemcpyAsync(a.pcell_cursor, a.pcell_start, sizeof(uint32_t) * ncs,
                                 cudaMemcpyDeviceToDevice, s));
    k_slic_pgroup<true><<<gp, 256, 0, s>>>(a);
  }
  // blocks of the point pass: a cell each; with few cells several share one
  const unsigned gpx = (unsigned)std::min<int64_t>(a.K, (int64_t)ctx->sm_count * 8);
  const int64_t want = ((int64_t)ctx->sm_count * 4 + gpx - 1) / gpx;
  const int64_t most = std::max<int64_t>(1, nps / ((int64_t)a.K * 512));
  const dim3 gpc(gpx, (unsigned)std::min<int64_t>(65535, std::min(want, most)));
  int it = 1;
  for (it = 1; it <= prm->max_iter; ++it) {
    MSF_CUDA_TRY(cudaMemsetAsync(a.moved, 0, sizeof(unsigned), s));
    {
      ScopedKernel k(ctx, "k_slic_update");
      k_slic_update<<<kb, 256, 0, s>>>(a, it >= 2 ? 1 : 0);
    }
    if (it >= 2) {
      unsigned mv = 0;
      MSF_CUDA_TRY(cudaMemcpyAsync(&mv, a.moved, sizeof(mv), cudaMemcpyDeviceToHost, s));
      MSF_CUDA_TRY(cudaStreamSynchronize(s));
      if (!mv) break;
    }
    if (it == prm->max_iter) break;
    {
      ScopedKernel k(ctx, "k_slic_cells");
      MSF_CUDA_TRY(cudaMemsetAsync(a.cell_cursor, 0, sizeof(uint32_t) * a.K, s));
      k_slic_cells<false><<<kb, 256, 0, s>>>(a);
      MSF_TRY(scan_exclusive_u32(ctx, a.cell_cursor, a.cell_start, a.K, S.scan_tmp,
                                 a.cell_start + a.K));
      MSF_CUDA_TRY(cudaMemcpyAsync(a.cell_cursor, a.cell_start, sizeof(uint32_t) * a.K,
                                   cudaMemcpyDeviceToDevice, s));
      k_slic_cells<true><<<kb, 256, 0, s>>>(a);
    }
    {
      ScopedKernel k(ctx, "k_slic_assign_field");
      if (d.nz > 1) launch_field_tiled<8, 8, 4>(a, gt, s);
      else launch_field_tiled<16, 16, 1>(a, gt, s);
    }
    if (nps > 0) {
      ScopedKernel k(ctx, "k_slic_assign_points");
      k_slic_assign_points_cells<<<gpc, 256, 0, s>>>(a);
    }
  }
  if (it > prm->max_iter) it = prm->max_iter;
  MSF_CUDA_TRY(cudaGetLastError());
  if (centers_host)
    MSF_CUDA_TRY(cudaMemcpyAsync(centers_host, a.centers, sizeof(float) * 6 * (size_t)a.K,
                                 cudaMemcpyDeviceToHost, s));
  if (counts_host)
    MSF_CUDA_TRY(cudaMemcpyAsync(counts_host, a.counts, sizeof(long long) * 2 * (size_t)a.K,
                                 cudaMemcpyDeviceToHost, s));
  MSF_CUDA_TRY(cudaStreamSynchronize(s));
  ctx->timer.flush();
  if (iters) *iters = it;
  return MSF_OK;
}

}  // namespace msf

// Steps that follow a clustering or a labelling: cluster merging (§3.3), the range query over
// centre properties and per-cluster summaries (§3.4), and trajectory splitting (§3.4).
//
// All of them are single passes over resident arrays with integer or fixed-order results:
//   merging    every pair of centres is tested once (tiles of pairs in shared memory) and
//              matching pairs are joined in a lock-free union-find whose roots are the smallest
//              index of their tree (a root is only ever hooked under a smaller one), so the
//              flattened parents are the groups' smallest indices whatever the order of joins;
//   select     a flag per centre, an exclusive scan, an ordered scatter;
//   summaries  three passes over the window: the scale of the fixed-point sums (largest value,
//              sample count), the counts / exact sums / extents, the squared deviations;
//   pieces     one thread per trajectory walks its timesteps twice (count, then write at the
//              scanned offset), so pieces come out in (point, t_start) order.
#include <cmath>
#include <cstring>

#include "msf_internal.cuh"

namespace msf {

int scan_exclusive_u32(msf_ctx* ctx, const uint32_t* in, uint32_t* out, int64_t n, DevBuf& tmp,
                       uint32_t* total);

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// Input staging: a host array is copied into `buf`; a device array is used where it is.
template <class T>
int stage_in(msf_ctx* c, const T* p, int kind, size_t n, DevBuf& buf, const T** dev) {
  if (kind == MSF_DEVICE) {
    *dev = p;
    return MSF_OK;
  }
  MSF_TRY(buf.ensure(sizeof(T) * std::max<size_t>(n, 1)));
  if (n)
    MSF_CUDA_TRY(cudaMemcpyAsync(buf.p, p, sizeof(T) * n, cudaMemcpyHostToDevice, c->stream));
  *dev = buf.as<T>();
  return MSF_OK;
}

// Output: device memory of the caller's, or staged and copied to the host afterwards.
template <class T>
int copy_out(msf_ctx* c, T* dst, int kind, const T* src, size_t n) {
  if (n && dst != src)
    MSF_CUDA_TRY(cudaMemcpyAsync(dst, src, sizeof(T) * n,
                                 kind == MSF_HOST ? cudaMemcpyDeviceToHost
                                                  : cudaMemcpyDeviceToDevice,
                                 c->stream));
  return MSF_OK;
}

unsigned blocks_for(int64_t n, int threads, int cap) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads, cap));
}

// ---------------------------------------------------------------------------------------------
// §3.3 merging
// ---------------------------------------------------------------------------------------------
// a == b, or 2|a - b| < eps (|a| + |b|): IEEE fp32 operations in that order (no contraction).
__device__ __forceinline__ bool value_match(float a, float b, float eps) {
  if (a == b) return true;
  const float lhs = __fmul_rn(2.0f, fabsf(__fsub_rn(a, b)));
  const float rhs = __fmul_rn(eps, __fadd_rn(fabsf(a), fabsf(b)));
  return lhs < rhs;
}

__device__ __forceinline__ int uf_find(const int* parent, int x) {
  int p = __ldcg(parent + x);
  while (p != x) {  // parents only decrease, and parent[x] <= x: the walk ends
    x = p;
    p = __ldcg(parent + x);
  }
  return x;
}

// Join the trees of a and b: the larger root is hooked under the smaller one. When the larger
// one has meanwhile been hooked elsewhere, atomicMin keeps the smaller parent and the join is
// retried from the parent it had, so no link is lost; each retry lowers a, so the loop ends.
__device__ void uf_union(int* parent, int a, int b) {
  for (;;) {
    a = uf_find(parent, a);
    b = uf_find(parent, b);
    if (a == b) return;
    if (a < b) {
      const int s = a;
      a = b;
      b = s;
    }
    const int old = atomicMin(parent + a, b);
    if (old == a) return;
    a = old;
  }
}

constexpr int kMergeTile = 256;
constexpr int kMergeNarrow = 32768;  // centres up to which a block takes 128 columns

__global__ void k_merge_init(int* parent, int K) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < K; i += gridDim.x * blockDim.x)
    parent[i] = i;
}

// Block (x, y): rows i of tile y (one per thread) against the columns j > i of the TC ones from x * TC.
// Most pairs of unlike centres fail on the first value compared, so nothing stands before that test.
// A pair whose roots were equal when the block started is joined already; where centres agree widely
// (the case merging is for) those are nearly all. The block joins its rows and columns in shared
// memory and then each with its set's first member in the map, one union per thread or two: a thread
// that joined every matching pair of its row in the map waited on L2 time and again while its warp
// stood still.
// One launch: with the first rows in one of their own, whose joins the rest then knew, centres that
// hardly agree waited for it (16,384 of them 94 us in one launch, 130 in two, 5000 of them 32 and 61).
// TC: few columns a block give more blocks and shorter chains, many fewer unions of the same sets in
// the map (all calls, one launch of 256 columns, then of 128: 16,384 centres without a match 107, 99
// us, in 1862 groups 282, 266, in 18 468, 270; 40,000 centres in 2310 groups 698, 835 us).
template <int TC>
__global__ void __launch_bounds__(kMergeTile) k_merge_pairs(const float* __restrict__ centers,
                                                            int K, float eps, int terms,
                                                            int* parent) {
  const int i0 = (int)blockIdx.y * kMergeTile, j0 = (int)blockIdx.x * TC;
  if (j0 + TC <= i0) return;
  __shared__ float s_p[TC], s_f[TC];
  __shared__ int s_root[TC];
  __shared__ uint32_t s_set[TC + kMergeTile];  // the columns, then the rows
  const int tid = threadIdx.x, i = i0 + tid;
  const int jn = min(TC, K - j0);
  const uint32_t row = i >= j0 && i < j0 + TC ? (uint32_t)(i - j0) : (uint32_t)(TC + tid);
  for (int n = tid; n < TC + kMergeTile; n += kMergeTile) s_set[n] = n;
  if (tid < jn) {
    s_p[tid] = centers[6 * (size_t)(j0 + tid) + 4];
    s_f[tid] = centers[6 * (size_t)(j0 + tid) + 5];
    s_root[tid] = uf_find(parent, j0 + tid);
  }
  __syncthreads();
  if (i < K) {
    const float pi = centers[6 * (size_t)i + 4], fi = centers[6 * (size_t)i + 5];
    const bool use_p = terms & MSF_MERGE_POINT, use_f = terms & MSF_MERGE_FIELD;
    const int root = uf_find(parent, i);
    for (int q = max(0, i + 1 - j0); q < jn; ++q) {
      if (use_p && !value_match(pi, s_p[q], eps)) continue;
      if (s_root[q] == root) continue;
      if (use_f && !value_match(fi, s_f[q], eps)) continue;
      sunion(s_set, row, q);
    }
  }
  __syncthreads();
  auto centre = [&](uint32_t n) { return n < TC ? j0 + (int)n : i0 + (int)n - TC; };
  for (uint32_t n = tid; n < TC + kMergeTile; n += kMergeTile) {
    const uint32_t first = sfind(s_set, n);
    if (first != n) uf_union(parent, centre(n), centre(first));
  }
}

__global__ void k_merge_flatten(int* parent, int K, uint32_t* n_groups) {
  int roots = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < K; i += gridDim.x * blockDim.x) {
    const int r = uf_find(parent, i);
    roots += (r == i);
    parent[i] = r;  // only lowers parent[i] to an ancestor: concurrent walks stay valid
  }
  roots = __reduce_add_sync(kFull, roots);
  if ((threadIdx.x & 31) == 0 && roots) atomicAdd(n_groups, (uint32_t)roots);
}

// ---------------------------------------------------------------------------------------------
// relabelling through a merge map
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_relabel_check(const int32_t* __restrict__ lab, int64_t n,
                                                       int K, uint32_t* bad) {
  bool b = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    b |= lab[i] >= K;
  if (__any_sync(kFull, b) && (threadIdx.x & 31) == 0) atomicOr(bad, 1u);
}

// VEC: labels in 16-byte units (an aligned buffer; the last n % 4 labels apart), four in flight per
// thread: the pass is bound by memory (50M labels, single ones 103 us, so 62; the check, which only
// reads, takes 47 us by single labels and 62 by units, and unaligned buffers 112 and 110 by single
// labels, one and four at a time).
template <bool VEC>
__global__ void __launch_bounds__(256) k_relabel_apply(int32_t* __restrict__ lab, int64_t n,
                                                       const int32_t* __restrict__ map,
                                                       const uint32_t* bad) {
  if (*bad) return;  // a label out of range: nothing changes
  auto one = [&](int32_t l) { return l >= 0 ? __ldg(map + l) : l; };
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if constexpr (VEC) {
    const int64_t units = n >> 2;
    int4* lab4 = reinterpret_cast<int4*>(lab);
    for (int64_t i = i0; i < units; i += 4 * stride) {
      int4 l[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        l[u] = i + u * stride < units ? lab4[i + u * stride] : make_int4(-1, -1, -1, -1);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        l[u] = make_int4(one(l[u].x), one(l[u].y), one(l[u].z), one(l[u].w));
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i + u * stride < units) lab4[i + u * stride] = l[u];
    }
    if (blockIdx.x == 0 && threadIdx.x < (n & 3)) {
      int32_t* p = lab + (n & ~3ll) + threadIdx.x;
      *p = one(*p);
    }
  } else {
    for (int64_t i = i0; i < n; i += stride) {
      const int32_t l = lab[i];
      if (l >= 0) lab[i] = __ldg(map + l);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// §3.4 range query
// ---------------------------------------------------------------------------------------------
struct Box {
  float lo[6], hi[6];
};

__device__ __forceinline__ bool in_box(const float* c, const Box& b) {
  bool in = true;
#pragma unroll
  for (int j = 0; j < 6; ++j) in &= (c[j] >= b.lo[j]) & (c[j] <= b.hi[j]);
  return in;
}

__global__ void k_select_flags(const float* __restrict__ centers, int K, Box box,
                               uint32_t* flags) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < K; i += gridDim.x * blockDim.x)
    flags[i] = in_box(centers + 6 * (size_t)i, box) ? 1u : 0u;
}

__global__ void k_select_write(const uint32_t* __restrict__ flags,
                               const uint32_t* __restrict__ offs, int K, int32_t* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < K; i += gridDim.x * blockDim.x)
    if (flags[i]) out[offs[i]] = i;
}

// ---------------------------------------------------------------------------------------------
// §3.4 per-cluster summaries
// ---------------------------------------------------------------------------------------------
// Accumulators (one DevBuf): per cluster n, fixed-point sum, extent bits, squared deviations and
// the mean, for field and point samples; then the scale inputs and a status word.
struct StatAcc {
  unsigned long long *nf, *np, *sf, *sp;  // [K] counts, int64 sums (two's complement)
  unsigned *lo, *hi;                      // [K][4] extent as fp32 bits (locations are >= 0)
  double *qf, *qp, *mf, *mp;              // [K] squared deviations, means
  unsigned* maxbits;                      // [2] largest |value| per kind, as fp32 bits
  unsigned long long* ntot;               // [2] summarised samples per kind
  unsigned* bad;                          // a label >= K
  static size_t bytes(int K) { return (size_t)K * (4 * 8 + 8 * 4 + 4 * 8) + 64; }
  static StatAcc carve(void* base, int K) {
    StatAcc a;
    char* p = static_cast<char*>(base);
    auto take = [&](size_t n) {
      char* r = p;
      p += n;
      return r;
    };
    a.nf = reinterpret_cast<unsigned long long*>(take(8 * (size_t)K));
    a.np = reinterpret_cast<unsigned long long*>(take(8 * (size_t)K));
    a.sf = reinterpret_cast<unsigned long long*>(take(8 * (size_t)K));
    a.sp = reinterpret_cast<unsigned long long*>(take(8 * (size_t)K));
    a.qf = reinterpret_cast<double*>(take(8 * (size_t)K));
    a.qp = reinterpret_cast<double*>(take(8 * (size_t)K));
    a.mf = reinterpret_cast<double*>(take(8 * (size_t)K));
    a.mp = reinterpret_cast<double*>(take(8 * (size_t)K));
    a.lo = reinterpret_cast<unsigned*>(take(16 * (size_t)K));
    a.hi = reinterpret_cast<unsigned*>(take(16 * (size_t)K));
    a.ntot = reinterpret_cast<unsigned long long*>(take(16));
    a.maxbits = reinterpret_cast<unsigned*>(take(8));
    a.bad = reinterpret_cast<unsigned*>(take(4));
    return a;
  }
};

struct StatArgs {
  const float* field;   // [T][V]
  const float* pos;     // [T][3][P]
  const float* attr;    // [T][A][P]
  const int32_t* key;   // [T][P]
  const int32_t* flab;  // [tw][V] or null
  const int32_t* plab;  // [tw][P] or null
  int64_t V, P;
  int nx, ny, nz, A, a, t0, tw, K;
  int kf, kp;
  StatAcc acc;
};

__global__ void k_cstat_init(StatAcc acc, int K) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < K; i += gridDim.x * blockDim.x) {
    acc.nf[i] = acc.np[i] = acc.sf[i] = acc.sp[i] = 0ull;
    acc.qf[i] = acc.qp[i] = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc.lo[4 * i + j] = 0x7F800000u;  // +inf
      acc.hi[4 * i + j] = 0u;           // +0
    }
  }
  if (blockIdx.x == 0 && threadIdx.x < 2) {
    acc.maxbits[threadIdx.x] = 0u;
    acc.ntot[threadIdx.x] = 0ull;
    if (threadIdx.x == 0) *acc.bad = 0u;
  }
}

// The samples a thread walks. Field: a column of the window's row table, that is the voxels
// col + r * nx of `rows` consecutive x-rows r (rows run on through z and t), so neighbouring
// threads read neighbouring voxels and a thread's samples are neighbours along y. Points: one
// trajectory over consecutive point steps. Either way a thread meets the same label several times
// in a row (a cluster is a few voxels wide and a point stays in it for a few steps), so it adds
// up a run of equal labels in registers and commits it once.
// 128^3 x 32 field and 1M x 32 point samples whose labels a merge left in 986 groups, one of them
// most samples: a commit per sample of every mixed warp queued on the large group's few
// addresses, sums 111.6 ms and deviations 62.5 ms; by runs and a table per block 0.66 and 1.78 ms
// (the scale pass, without its two 64-bit divisions per sample, 0.44 -> 0.21 ms).
constexpr int kCstatRun = 16;   // samples per thread and column (or trajectory) at most
constexpr int kCstatCols = 1024;  // columns per block at most (256 threads)

struct StatWalk {
  int rows;    // samples per column (field rows or point steps)
  int groups;  // field: row groups per block; each nx columns wide
  int cols;    // field: columns per block, of the groups' (blocks along y share longer rows)
  int nrows;   // field: x-rows of the window; points: its point steps
};

// Calls body(l, v, x, y, z, t) for every sample of the thread that takes part (label, value; the
// location only for LOC), column by column, and done() after each column. bad: set when a label is >= K.
template <bool POINTS, bool LOC, class Body, class Done>
__device__ __forceinline__ void stat_walk(const StatArgs& s, const StatWalk& w, bool& bad,
                                          Body&& body, Done&& done) {
  constexpr int U = 4;  // loads in flight
  if (POINTS) {
    const int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (p >= s.P) return;
    const int ta = blockIdx.y * w.rows, tb = min(ta + w.rows, w.nrows);
    for (int t0 = ta; t0 < tb; t0 += U) {
      int l[U], k[U];
      float v[U], px[U], py[U], pz[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const bool in = t0 + u < tb;
        const int64_t o = (int64_t)(s.t0 + t0 + u);
        l[u] = in ? __ldg(s.plab + (int64_t)(t0 + u) * s.P + p) : -1;
        k[u] = in ? __ldg(s.key + o * s.P + p) : -1;
        v[u] = in ? __ldg(s.attr + (o * s.A + s.a) * s.P + p) : 0.f;
        if (LOC) {
          const float* ps = s.pos + o * 3 * s.P + p;
          px[u] = in ? __ldg(ps) : 0.f;
          py[u] = in ? __ldg(ps + s.P) : 0.f;
          pz[u] = in ? __ldg(ps + 2 * s.P) : 0.f;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        bad |= l[u] >= s.K;
        if (l[u] < 0 || k[u] < 0 || !isfinite(v[u])) continue;
        // +0 for -0 so that the fp32 bits order like the values
        if (LOC)
          body(l[u], v[u], __fadd_rn(px[u], 0.0f), __fadd_rn(py[u], 0.0f),
               __fadd_rn(pz[u], 0.0f), __fadd_rn((float)(s.t0 + t0 + u), 0.5f));
        else body(l[u], v[u], 0.f, 0.f, 0.f, 0.f);
      }
    }
    done();
    return;
  }
  const unsigned c0 = blockIdx.y * (unsigned)w.cols, nx = (unsigned)s.nx;
  const unsigned cend = min(c0 + (unsigned)w.cols, (unsigned)w.groups * nx);
  const float* field = s.field + (int64_t)s.t0 * s.V;
  for (unsigned c = c0 + threadIdx.x; c < cend; c += 256u) {
    const int g = (int)(c / nx), x = (int)(c - (unsigned)g * nx);
    const int64_t rb = ((int64_t)blockIdx.x * w.groups + g) * w.rows;
    if (rb >= w.nrows) break;
    const int ra = (int)rb, re = (int)min(rb + w.rows, (int64_t)w.nrows);
    int y = 0, z = 0, t = 0;
    if (LOC) {
      const int zt = ra / s.ny;
      y = ra - zt * s.ny;
      t = zt / s.nz;
      z = zt - t * s.nz;
    }
    for (int r0 = ra; r0 < re; r0 += U) {
      int l[U];
      float v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t i = (int64_t)(r0 + u) * s.nx + x;
        const bool in = r0 + u < re;
        l[u] = in ? __ldg(s.flab + i) : -1;
        v[u] = in ? __ldg(field + i) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        bad |= l[u] >= s.K;
        if (l[u] >= 0 && isfinite(v[u]))
          body(l[u], v[u], __fadd_rn((float)x, 0.5f), __fadd_rn((float)y, 0.5f),
               __fadd_rn((float)z, 0.5f), __fadd_rn((float)(s.t0 + t), 0.5f));
        if (LOC && ++y == s.ny) {
          y = 0;
          if (++z == s.nz) {
            z = 0;
            ++t;
          }
        }
      }
    }
    done();
  }
}

// pass 1: labels in range, the largest |value| and the sample count per kind (no label's sums
// yet: the fixed-point scale needs both first)
template <bool POINTS>
__global__ void __launch_bounds__(256) k_cstat_scale(StatArgs s, StatWalk w) {
  unsigned m = 0u, c = 0u;
  bool bad = false;
  stat_walk<POINTS, false>(
      s, w, bad,
      [&](int, float v, float, float, float, float) {
        m = max(m, __float_as_uint(fabsf(v)));
        ++c;
      },
      [] {});
  __shared__ unsigned s_m, s_c;
  __shared__ int s_bad;
  if (threadIdx.x == 0) s_m = s_c = 0u, s_bad = 0;
  __syncthreads();
  m = __reduce_max_sync(kFull, m);
  c = __reduce_add_sync(kFull, c);
  if (__any_sync(kFull, bad) && (threadIdx.x & 31) == 0) s_bad = 1;
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&s_m, m);
    atomicAdd(&s_c, c);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_bad) atomicOr(s.acc.bad, 1u);
    if (s_m) atomicMax(s.acc.maxbits + (POINTS ? 1 : 0), s_m);
    if (s_c) atomicAdd(s.acc.ntot + (POINTS ? 1 : 0), (unsigned long long)s_c);
  }
}

// The labels a block meets, in a small open-addressing table of shared memory: runs commit there
// and the block commits each of its labels once. Without it every run of a label that most
// samples carry (what a merge leaves) would queue on one address in L2. A label that finds no
// place within a few probes (points in id order carry labels from everywhere) commits to the
// accumulators itself.
constexpr int kCtab = 512, kCtabProbes = 4;

__device__ __forceinline__ int ctab_slot(int* key, int l) {
  unsigned h = ((unsigned)l * 0x9E3779B1u) >> 23;
#pragma unroll 1
  for (int i = 0; i < kCtabProbes; ++i) {
    int k = *(volatile int*)(key + h);
    if (k == -1) {
      k = atomicCAS(key + h, -1, l);
      if (k == -1) return (int)h;
    }
    if (k == l) return (int)h;
    h = (h + 1) & (kCtab - 1);
  }
  return -1;
}

// Do all lanes of the warp end a run of the same label here (all of them converged)? Labels that lie
// along the rows make every sample a run of its own, and neighbouring lanes' the same: they add up in
// the warp, since 32 of them would queue at the label's place (5000 x 40 x 16, 1000 labels along the
// rows, the whole call 0.27 ms, so 0.19).
__device__ __forceinline__ bool warp_of_one(int label) {
  if (__activemask() != kFull) return false;
  int same;
  __match_all_sync(kFull, label, &same);
  return same && label >= 0;
}

struct SumTab {
  int key[kCtab];
  unsigned n[kCtab];
  unsigned slo[kCtab], shi[kCtab];   // the fixed-point sum's halves (mod 2^64)
  uint4 lo[kCtab], hi[kCtab];        // extent, fp32 bits
};

// extent words: an atomic only where the value extends what is there (a stale value read here
// only costs an atomic that changes nothing)
__device__ __forceinline__ void extend(unsigned* lo, unsigned* hi, const uint4& cl, const uint4& ch,
                                       const unsigned (&l)[4], const unsigned (&h)[4]) {
  const unsigned a[4] = {cl.x, cl.y, cl.z, cl.w}, b[4] = {ch.x, ch.y, ch.z, ch.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (l[j] < a[j]) atomicMin(lo + j, l[j]);
    if (h[j] > b[j]) atomicMax(hi + j, h[j]);
  }
}

template <bool POINTS>
__device__ __forceinline__ void commit_sum(const StatArgs& s, int l, unsigned n, long long q,
                                           const unsigned (&lo)[4], const unsigned (&hi)[4]) {
  atomicAdd((POINTS ? s.acc.np : s.acc.nf) + l, (unsigned long long)n);
  atomicAdd((POINTS ? s.acc.sp : s.acc.sf) + l, (unsigned long long)q);
  unsigned* gl = s.acc.lo + 4 * (size_t)l;
  unsigned* gh = s.acc.hi + 4 * (size_t)l;
  extend(gl, gh, __ldca(reinterpret_cast<const uint4*>(gl)),
         __ldca(reinterpret_cast<const uint4*>(gh)), lo, hi);
}

// pass 2: counts, exact sums and extents, by runs of equal labels
template <bool POINTS>
__global__ void __launch_bounds__(256) k_cstat_sum(StatArgs s, StatWalk w) {
  __shared__ SumTab tab;
  for (int i = threadIdx.x; i < kCtab; i += 256) {
    tab.key[i] = -1;
    tab.n[i] = tab.slo[i] = tab.shi[i] = 0u;
    tab.lo[i] = make_uint4(0x7F800000u, 0x7F800000u, 0x7F800000u, 0x7F800000u);
    tab.hi[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  __syncthreads();
  const int k = POINTS ? s.kp : s.kf;
  int rl = -1;  // the run at hand: label, samples, sum, extent
  unsigned rn = 0u, rlo[4], rhi[4];
  long long rq = 0;
  bool bad = false;  // (labels were checked by pass 1)
  auto flush = [&] {
    if (warp_of_one(rl)) {
      rq = (long long)limb_sum(kFull, (unsigned long long)rq);
      rn = __reduce_add_sync(kFull, rn);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        rlo[j] = __reduce_min_sync(kFull, rlo[j]);
        rhi[j] = __reduce_max_sync(kFull, rhi[j]);
      }
      if (threadIdx.x & 31) rl = -1;
    }
    if (rl < 0) return;
    const int h = ctab_slot(tab.key, rl);
    if (h < 0) {
      commit_sum<POINTS>(s, rl, rn, rq, rlo, rhi);
    } else {
      const unsigned ql = (unsigned)(unsigned long long)rq;
      const unsigned qh = (unsigned)((unsigned long long)rq >> 32);
      atomicAdd(tab.n + h, rn);
      const unsigned old = atomicAdd(tab.slo + h, ql);
      atomicAdd(tab.shi + h, qh + (old + ql < old ? 1u : 0u));  // with the carry
      extend(&tab.lo[h].x, &tab.hi[h].x, tab.lo[h], tab.hi[h], rlo, rhi);
    }
    rl = -1;
  };
  stat_walk<POINTS, true>(
      s, w, bad,
      [&](int l, float v, float x, float y, float z, float t) {
        const unsigned b[4] = {__float_as_uint(x), __float_as_uint(y), __float_as_uint(z),
                               __float_as_uint(t)};
        const long long q = quantise(v, k);
        if (l != rl) {
          flush();
          rl = l;
          rn = 0u;
          rq = 0;
#pragma unroll
          for (int j = 0; j < 4; ++j) rlo[j] = rhi[j] = b[j];
        }
        ++rn;
        rq += q;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          rlo[j] = min(rlo[j], b[j]);
          rhi[j] = max(rhi[j], b[j]);
        }
      },
      flush);
  __syncthreads();
  for (int i = threadIdx.x; i < kCtab; i += 256) {
    if (tab.key[i] < 0) continue;
    const uint4 a = tab.lo[i], b = tab.hi[i];
    const unsigned lo[4] = {a.x, a.y, a.z, a.w}, hi[4] = {b.x, b.y, b.z, b.w};
    commit_sum<POINTS>(s, tab.key[i], tab.n[i],
                       (long long)(((unsigned long long)tab.shi[i] << 32) | tab.slo[i]), lo, hi);
  }
}

// means from the exact sums: ((double)sum / n) * 2^-k
__device__ __forceinline__ double fixed_mean(unsigned long long s, unsigned long long n, int k) {
  if (!n) return __longlong_as_double(0x7FF8000000000000ll);
  const double m = __ddiv_rn(__ll2double_rn((long long)s), __ull2double_rn(n));
  return __dmul_rn(m, __longlong_as_double((long long)(1023 - k) << 52));
}

__global__ void k_cstat_means(StatAcc acc, int K, int kf, int kp) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < K; i += gridDim.x * blockDim.x) {
    acc.mf[i] = fixed_mean(acc.sf[i], acc.nf[i], kf);
    acc.mp[i] = fixed_mean(acc.sp[i], acc.np[i], kp);
  }
}

// pass 3: squared deviations from the means, in fp64, by runs of equal labels as in pass 2 (two
// fp64 operations per sample: this part's fp64 rate would make a warp reduction per label cost
// more than the pass's memory traffic). An fp64 addition in shared memory is a compare-and-swap
// loop, so lanes that commit one label at a time would take turns: a label has kDevCopies sums,
// a lane's by its index (one sum each 1.78 ms, now 0.74 ms, on the case above).
constexpr int kDevCopies = 8;

template <bool POINTS>
__global__ void __launch_bounds__(256) k_cstat_dev(StatArgs s, StatWalk w) {
  __shared__ int s_key[kCtab];
  __shared__ double s_q[kCtab][kDevCopies];
  for (int i = threadIdx.x; i < kCtab; i += 256) s_key[i] = -1;
  for (int i = threadIdx.x; i < kCtab * kDevCopies; i += 256) (&s_q[0][0])[i] = 0.0;
  __syncthreads();
  double* q = POINTS ? s.acc.qp : s.acc.qf;
  const double* mean = POINTS ? s.acc.mp : s.acc.mf;
  int rl = -1;
  double rd = 0.0, rm = 0.0;
  bool bad = false;
  auto flush = [&] {
    if (warp_of_one(rl)) {
#pragma unroll
      for (int o = 16; o; o >>= 1) rd += __shfl_xor_sync(kFull, rd, o);
      if (threadIdx.x & 31) rl = -1;
    }
    if (rl < 0) return;
    const int h = ctab_slot(s_key, rl);
    if (h < 0) atomicAdd(q + rl, rd);
    else atomicAdd(&s_q[h][threadIdx.x & (kDevCopies - 1)], rd);
    rl = -1;
  };
  stat_walk<POINTS, false>(
      s, w, bad,
      [&](int l, float v, float, float, float, float) {
        if (l != rl) {
          flush();
          rl = l;
          rd = 0.0;
          rm = __ldg(mean + l);
        }
        const double d = __dsub_rn(f2d(v), rm);
        rd = __fma_rn(d, d, rd);
      },
      flush);
  __syncthreads();
  for (int i = threadIdx.x; i < kCtab; i += 256) {
    if (s_key[i] < 0) continue;
    double t = 0.0;
#pragma unroll
    for (int j = 0; j < kDevCopies; ++j) t += s_q[i][j];
    atomicAdd(q + s_key[i], t);
  }
}

__global__ void k_cstat_final(StatAcc acc, int K, msf_cluster_stat* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < K; i += gridDim.x * blockDim.x) {
    msf_cluster_stat r;
    r.n_field = (int64_t)acc.nf[i];
    r.n_point = (int64_t)acc.np[i];
    const bool any = r.n_field + r.n_point > 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      r.lo[j] = __uint_as_float(acc.lo[4 * i + j]);
      r.hi[j] = any ? __uint_as_float(acc.hi[4 * i + j]) : -INFINITY;
    }
    const double qnan = __longlong_as_double(0x7FF8000000000000ll);
    r.mean_field = acc.mf[i];
    r.mean_point = acc.mp[i];
    r.std_field = r.n_field ? __dsqrt_rn(__ddiv_rn(acc.qf[i], (double)r.n_field)) : qnan;
    r.std_point = r.n_point ? __dsqrt_rn(__ddiv_rn(acc.qp[i], (double)r.n_point)) : qnan;
    out[i] = r;
  }
}

// Columns per block and samples per thread: as many as allowed, fewer while the pass would have
// less than four blocks per SM (short runs cost more commits, an idle GPU costs more). Rows longer
// than a block's columns are cut into pieces, one block each: with whole rows a block, few long rows
// left most of the GPU idle (2^20 x 8 steps 14.3 ms, so 0.4 ms; 5000 x 40 x 16, labels along the
// rows, 0.34 and 0.27 ms).
dim3 field_walk(const StatArgs& a, int64_t nrows, int sm_count, StatWalk* w) {
  w->nrows = (int)nrows;
  int cols = kCstatCols;
  w->rows = kCstatRun;
  int64_t gx = 1, gy = 1;
  auto blocks = [&] {
    w->groups = a.nx < cols ? (cols + a.nx - 1) / a.nx : 1;
    w->cols = a.nx < cols ? w->groups * a.nx : std::max<int>(cols, (a.nx / 65535 + 256) & ~255);
    const int64_t per = (int64_t)w->groups * w->rows;
    gx = std::max<int64_t>(1, (nrows + per - 1) / per);
    gy = a.nx < cols ? 1 : (a.nx + (int64_t)w->cols - 1) / w->cols;
    return gx * gy;
  };
  while (blocks() < 4 * (int64_t)sm_count && (cols > 256 || w->rows > 1)) {
    if (cols > 256) cols >>= 1;
    else w->rows >>= 1;
  }
  return dim3((unsigned)gx, (unsigned)gy);
}

dim3 point_walk(const StatArgs& a, int sm_count, StatWalk* w) {
  w->nrows = a.tw;
  w->groups = 1;
  w->rows = kCstatRun;
  const int64_t gx = (a.P + 255) / 256;
  auto gy = [&] { return (a.tw + w->rows - 1) / w->rows; };
  while (gx * gy() < 4 * (int64_t)sm_count && w->rows > 1) w->rows >>= 1;
  return dim3((unsigned)gx, (unsigned)gy());
}

// ---------------------------------------------------------------------------------------------
// §3.4 trajectory pieces
// ---------------------------------------------------------------------------------------------
struct PieceArgs {
  const int32_t* lab;  // [tw][P] (points) or [tw][V] (voxels)
  const int32_t* key;  // [T][P] binning keys (voxel space)
  int64_t P, V;
  int t0, tw, min_len;
  const uint32_t* offs;  // [P] first piece of each trajectory (write pass)
  int4* out;
};

template <bool VOX>
__device__ __forceinline__ int32_t sample_label(const PieceArgs& a, int t, int64_t p) {
  if (VOX) {
    const int32_t k = __ldg(a.key + (int64_t)(a.t0 + t) * a.P + p);
    return k >= 0 ? __ldg(a.lab + (int64_t)t * a.V + k) : -1;
  }
  return __ldg(a.lab + (int64_t)t * a.P + p);
}

// One thread per trajectory: the runs of equal labels along t; runs of a non-negative label and
// at least min_len steps are pieces. COUNT: pieces per trajectory; else write them in order.
template <bool VOX, bool COUNT>
__global__ void __launch_bounds__(256) k_pieces(PieceArgs a, uint32_t* cnt) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < a.P;
       p += (int64_t)gridDim.x * blockDim.x) {
    uint32_t n = 0, o = COUNT ? 0u : a.offs[p];
    int32_t cur = sample_label<VOX>(a, 0, p);
    int start = 0;
    for (int t = 1; t <= a.tw; ++t) {
      const int32_t l = t < a.tw ? sample_label<VOX>(a, t, p) : -1;
      if (t == a.tw || l != cur) {
        if (cur >= 0 && t - start >= a.min_len) {
          if (!COUNT) a.out[o + n] = make_int4((int)p, start, t - start, cur);
          ++n;
        }
        cur = l;
        start = t;
      }
    }
    if (COUNT) cnt[p] = n;
  }
}

}  // namespace
}  // namespace msf

using namespace msf;

extern "C" {

int msf_merge_clusters(msf_ctx* c, const float* centers, int centers_kind, int32_t K,
                       float eps_m, int terms, int32_t* map, int map_kind, int32_t* n_groups) {
  if (!c || !centers || !map) return MSF_ERR_INVALID_ARG;
  if ((centers_kind != MSF_HOST && centers_kind != MSF_DEVICE) ||
      (map_kind != MSF_HOST && map_kind != MSF_DEVICE))
    return MSF_ERR_INVALID_ARG;
  if (K < 1 || !std::isfinite(eps_m) || eps_m < 0.f) return MSF_ERR_INVALID_ARG;
  if (terms == 0 || (terms & ~(MSF_MERGE_POINT | MSF_MERGE_FIELD))) return MSF_ERR_INVALID_ARG;
  if (K > (1 << 18)) return MSF_ERR_TOO_LARGE;
  MSF_CUDA_TRY(cudaSetDevice(c->device));
  SpareScope spare(c);
  PostScratch& S = c->post;
  const float* dc;
  MSF_TRY(stage_in(c, centers, centers_kind, 6 * (size_t)K, S.in, &dc));
  int32_t* parent = map;
  if (map_kind == MSF_HOST) {
    MSF_TRY(S.out.ensure(sizeof(int32_t) * (size_t)K));
    parent = S.out.as<int32_t>();
  }
  MSF_TRY(S.total.ensure(sizeof(uint32_t)));
  uint32_t* ng = S.total.as<uint32_t>();
  cudaStream_t s = c->stream;
  MSF_CUDA_TRY(cudaMemsetAsync(ng, 0, sizeof(uint32_t), s));
  {
    ScopedKernel k(c, "k_merge_init");
    k_merge_init<<<blocks_for(K, 256, c->sm_count * 8), 256, 0, s>>>(parent, K);
  }
  {
    ScopedKernel k(c, "k_merge_pairs");
    const unsigned nt = (unsigned)((K + kMergeTile - 1) / kMergeTile);
    if (K <= kMergeNarrow)
      k_merge_pairs<128><<<dim3((unsigned)((K + 127) / 128), nt), kMergeTile, 0, s>>>(dc, K, eps_m,
                                                                                      terms, parent);
    else
      k_merge_pairs<256><<<dim3(nt, nt), kMergeTile, 0, s>>>(dc, K, eps_m, terms, parent);
  }
  {
    ScopedKernel k(c, "k_merge_flatten");
    k_merge_flatten<<<blocks_for(K, 256, c->sm_count * 8), 256, 0, s>>>(parent, K, ng);
  }
  MSF_CUDA_TRY(cudaGetLastError());
  if (map_kind == MSF_HOST) MSF_TRY(copy_out(c, map, MSF_HOST, (const int32_t*)parent, K));
  uint32_t g = 0;
  MSF_CUDA_TRY(cudaMemcpyAsync(&g, ng, sizeof(g), cudaMemcpyDeviceToHost, s));
  MSF_CUDA_TRY(cudaStreamSynchronize(s));
  c->timer.flush();
  if (n_groups) *n_groups = (int32_t)g;
  return MSF_OK;
}

int msf_relabel(msf_ctx* c, int32_t* labels, int labels_kind, int64_t n, const int32_t* map,
                int map_kind, int32_t K) {
  if (!c || (n > 0 && !labels) || !map || K < 1 || n < 0) return MSF_ERR_INVALID_ARG;
  if ((labels_kind != MSF_HOST && labels_kind != MSF_DEVICE) ||
      (map_kind != MSF_HOST && map_kind != MSF_DEVICE))
    return MSF_ERR_INVALID_ARG;
  if (n >= ((int64_t)1 << 31)) return MSF_ERR_TOO_LARGE;
  if (n == 0) return MSF_OK;
  // the labels may be the buffer of the retained segmentation: its features no longer describe
  // them, so msf_extract_features must read the buffer from now on
  c->last.valid = false;
  MSF_CUDA_TRY(cudaSetDevice(c->device));
  SpareScope spare(c);
  PostScratch& S = c->post;
  const int32_t* dm;
  MSF_TRY(stage_in(c, map, map_kind, (size_t)K, S.in2, &dm));
  int32_t* dl = labels;
  cudaStream_t s = c->stream;
  if (labels_kind == MSF_HOST) {
    MSF_TRY(S.out.ensure(sizeof(int32_t) * (size_t)n));
    dl = S.out.as<int32_t>();
    MSF_CUDA_TRY(cudaMemcpyAsync(dl, labels, sizeof(int32_t) * n, cudaMemcpyHostToDevice, s));
  }
  MSF_TRY(S.status.ensure(sizeof(uint32_t)));
  uint32_t* bad = S.status.as<uint32_t>();
  MSF_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(uint32_t), s));
  const bool vec = ((uintptr_t)dl & 15) == 0;
  const unsigned gc = blocks_for(n, 256, c->sm_count * 8);
  const unsigned g = vec ? blocks_for((n + 3) / 4, 256, c->sm_count * 8) : gc;
  {
    ScopedKernel k(c, "k_relabel_check");
    k_relabel_check<<<gc, 256, 0, s>>>(dl, n, K, bad);
  }
  {
    ScopedKernel k(c, "k_relabel_apply");
    if (vec) k_relabel_apply<true><<<g, 256, 0, s>>>(dl, n, dm, bad);
    else k_relabel_apply<false><<<g, 256, 0, s>>>(dl, n, dm, bad);
  }
  MSF_CUDA_TRY(cudaGetLastError());
  uint32_t hb = 0;
  MSF_CUDA_TRY(cudaMemcpyAsync(&hb, bad, sizeof(hb), cudaMemcpyDeviceToHost, s));
  MSF_CUDA_TRY(cudaStreamSynchronize(s));
  c->timer.flush();
  if (hb) return MSF_ERR_INVALID_ARG;
  if (labels_kind == MSF_HOST) {
    MSF_CUDA_TRY(cudaMemcpyAsync(labels, dl, sizeof(int32_t) * n, cudaMemcpyDeviceToHost, s));
    MSF_CUDA_TRY(cudaStreamSynchronize(s));
  }
  return MSF_OK;
}

int msf_select_clusters(msf_ctx* c, const float* centers, int centers_kind, int32_t K,
                        const float lo[6], const float hi[6], int32_t* out, int out_kind,
                        int32_t cap, int32_t* n_out) {
  if (!c || !centers || !lo || !hi || !n_out || K < 1 || cap < 0 || (cap > 0 && !out))
    return MSF_ERR_INVALID_ARG;
  if ((centers_kind != MSF_HOST && centers_kind != MSF_DEVICE) ||
      (out_kind != MSF_HOST && out_kind != MSF_DEVICE))
    return MSF_ERR_INVALID_ARG;
  Box box;
  for (int j = 0; j < 6; ++j) {
    if (std::isnan(lo[j]) || std::isnan(hi[j])) return MSF_ERR_INVALID_ARG;
    box.lo[j] = lo[j];
    box.hi[j] = hi[j];
  }
  if (K > (1 << 20)) return MSF_ERR_TOO_LARGE;
  MSF_CUDA_TRY(cudaSetDevice(c->device));
  SpareScope spare(c);
  PostScratch& S = c->post;
  const float* dc;
  MSF_TRY(stage_in(c, centers, centers_kind, 6 * (size_t)K, S.in, &dc));
  MSF_TRY(S.cnt.ensure(sizeof(uint32_t) * (size_t)K));
  MSF_TRY(S.offs.ensure(sizeof(uint32_t) * (size_t)K));
  MSF_TRY(S.total.ensure(sizeof(uint32_t)));
  uint32_t* flags = S.cnt.as<uint32_t>();
  uint32_t* offs = S.offs.as<uint32_t>();
  cudaStream_t s = c->stream;
  const unsigned g = blocks_for(K, 256, c->sm_count * 8);
  {
    ScopedKernel k(c, "k_select_flags");
    k_select_flags<<<g, 256, 0, s>>>(dc, K, box, flags);
  }
  MSF_TRY(scan_exclusive_u32(c, flags, offs, K, S.scan_tmp, S.total.as<uint32_t>()));
  uint32_t n = 0;
  MSF_CUDA_TRY(cudaMemcpyAsync(&n, S.total.p, sizeof(n), cudaMemcpyDeviceToHost, s));
  MSF_CUDA_TRY(cudaStreamSynchronize(s));
  *n_out = (int32_t)n;
  if ((int64_t)n > cap) {
    c->timer.flush();
    return MSF_ERR_CAPACITY;
  }
  if (n) {
    int32_t* dst = out;
    if (out_kind == MSF_HOST) {
      MSF_TRY(S.out.ensure(sizeof(int32_t) * (size_t)n));
      dst = S.out.as<int32_t>();
    }
    {
      ScopedKernel k(c, "k_select_write");
      k_select_write<<<g, 256, 0, s>>>(flags, offs, K, dst);
    }
    MSF_CUDA_TRY(cudaGetLastError());
    if (out_kind == MSF_HOST) MSF_TRY(copy_out(c, out, MSF_HOST, (const int32_t*)dst, n));
    MSF_CUDA_TRY(cudaStreamSynchronize(s));
  }
  c->timer.flush();
  return MSF_OK;
}

static int scale_bits(float max_abs, unsigned long long n) {
  int e = 0;
  if (max_abs > 0.f && std::isfinite(max_abs)) std::frexp((double)max_abs, &e);
  int b = 0;
  while ((1ull << b) < n + 1) ++b;
  return 62 - e - b;
}

int msf_cluster_stats(msf_ctx* c, int32_t t0, int32_t t1, int32_t attr,
                      const int32_t* field_labels, const int32_t* point_labels, int labels_kind,
                      int32_t K, msf_cluster_stat* out, int out_kind) {
  if (!c || !out || K < 1) return MSF_ERR_INVALID_ARG;
  if ((labels_kind != MSF_HOST && labels_kind != MSF_DEVICE) ||
      (out_kind != MSF_HOST && out_kind != MSF_DEVICE))
    return MSF_ERR_INVALID_ARG;
  const Dataset& d = c->ds;
  if (!d.loaded) return MSF_ERR_NOT_LOADED;
  if (t0 < 0 || t1 > d.T || t1 <= t0) return MSF_ERR_INVALID_ARG;
  const bool use_p = point_labels != nullptr && d.P > 0;
  if (use_p) {
    if (attr < 0 || attr >= d.A) return MSF_ERR_INVALID_ARG;
    if (!d.binned) return MSF_ERR_NOT_BINNED;
    if (d.multirate) return MSF_ERR_INVALID_ARG;  // point labels are [tw][P]: one step each
  }
  if (K > (1 << 20)) return MSF_ERR_TOO_LARGE;
  const int64_t tw = t1 - t0, nf = tw * d.V, np = use_p ? tw * d.P : 0;
  if (nf >= ((int64_t)1 << 31) || np >= ((int64_t)1 << 31)) return MSF_ERR_TOO_LARGE;
  MSF_CUDA_TRY(cudaSetDevice(c->device));
  SpareScope spare(c);
  MSF_TRY(ctx_field_ready(c));
  PostScratch& S = c->post;
  StatArgs a{};
  a.field = d.field.as<float>();
  a.pos = d.pos.as<float>();
  a.attr = d.attr.as<float>();
  a.key = d.key.as<int32_t>();
  a.V = d.V;
  a.P = d.P;
  a.nx = d.nx;
  a.ny = d.ny;
  a.nz = d.nz;
  a.A = d.A;
  a.a = attr;
  a.t0 = t0;
  a.tw = (int)tw;
  a.K = K;
  if (field_labels) MSF_TRY(stage_in(c, field_labels, labels_kind, (size_t)nf, S.in, &a.flab));
  if (use_p) MSF_TRY(stage_in(c, point_labels, labels_kind, (size_t)np, S.in2, &a.plab));
  MSF_TRY(S.acc.ensure(StatAcc::bytes(K)));
  a.acc = StatAcc::carve(S.acc.p, K);
  cudaStream_t s = c->stream;
  const unsigned gk = blocks_for(K, 256, c->sm_count * 8);
  StatWalk wf{}, wp{};
  const dim3 gf = a.flab ? field_walk(a, tw * d.nz * d.ny, c->sm_count, &wf) : dim3(1);
  const dim3 gp = a.plab ? point_walk(a, c->sm_count, &wp) : dim3(1);
  {
    ScopedKernel k(c, "k_cstat_init");
    k_cstat_init<<<gk, 256, 0, s>>>(a.acc, K);
  }
  {
    ScopedKernel k(c, "k_cstat_scale");
    if (a.flab) k_cstat_scale<false><<<gf, 256, 0, s>>>(a, wf);
    if (a.plab) k_cstat_scale<true><<<gp, 256, 0, s>>>(a, wp);
  }
  MSF_CUDA_TRY(cudaGetLastError());
  struct {
    unsigned long long ntot[2];
    unsigned maxbits[2];
    unsigned bad;
  } h;
  MSF_CUDA_TRY(cudaMemcpyAsync(&h, a.acc.ntot, sizeof(h.ntot) + sizeof(h.maxbits) + sizeof(h.bad),
                               cudaMemcpyDeviceToHost, s));
  MSF_CUDA_TRY(cudaStreamSynchronize(s));
  if (h.bad) {
    c->timer.flush();
    return MSF_ERR_INVALID_ARG;
  }
  float fm, pm;
  std::memcpy(&fm, &h.maxbits[0], 4);
  std::memcpy(&pm, &h.maxbits[1], 4);
  a.kf = scale_bits(fm, h.ntot[0]);
  a.kp = scale_bits(pm, h.ntot[1]);
  {
    ScopedKernel k(c, "k_cstat_sum");
    if (a.flab) k_cstat_sum<false><<<gf, 256, 0, s>>>(a, wf);
    if (a.plab) k_cstat_sum<true><<<gp, 256, 0, s>>>(a, wp);
  }
  {
    ScopedKernel k(c, "k_cstat_means");
    k_cstat_means<<<gk, 256, 0, s>>>(a.acc, K, a.kf, a.kp);
  }
  {
    ScopedKernel k(c, "k_cstat_dev");
    if (a.flab) k_cstat_dev<false><<<gf, 256, 0, s>>>(a, wf);
    if (a.plab) k_cstat_dev<true><<<gp, 256, 0, s>>>(a, wp);
  }
  msf_cluster_stat* dst = out;
  if (out_kind == MSF_HOST) {
    MSF_TRY(S.out.ensure(sizeof(msf_cluster_stat) * (size_t)K));
    dst = S.out.as<msf_cluster_stat>();
  }
  {
    ScopedKernel k(c, "k_cstat_final");
    k_cstat_final<<<gk, 256, 0, s>>>(a.acc, K, dst);
  }
  MSF_CUDA_TRY(cudaGetLastError());
  if (out_kind == MSF_HOST) MSF_TRY(copy_out(c, out, MSF_HOST, (const msf_cluster_stat*)dst, K));
  MSF_CUDA_TRY(cudaStreamSynchronize(s));
  c->timer.flush();
  return MSF_OK;
}

int msf_split_trajectories(msf_ctx* c, int32_t t0, int32_t t1, const int32_t* labels,
                           int labels_kind, int labels_space, int32_t min_len, msf_piece* pieces,
                           int pieces_kind, int64_t cap, int64_t* n_pieces) {
  if (!c || !n_pieces || min_len < 1 || cap < 0 || (cap > 0 && !pieces))
    return MSF_ERR_INVALID_ARG;
  if ((labels_kind != MSF_HOST && labels_kind != MSF_DEVICE) ||
      (pieces_kind != MSF_HOST && pieces_kind != MSF_DEVICE))
    return MSF_ERR_INVALID_ARG;
  if (labels_space != MSF_SPACE_POINTS && labels_space != MSF_SPACE_VOXELS)
    return MSF_ERR_INVALID_ARG;
  const Dataset& d = c->ds;
  if (!d.loaded) return MSF_ERR_NOT_LOADED;
  if (t0 < 0 || t1 > d.T || t1 <= t0) return MSF_ERR_INVALID_ARG;
  const bool vox = labels_space == MSF_SPACE_VOXELS;
  if (vox && !d.binned) return MSF_ERR_NOT_BINNED;
  if (vox && d.multirate) return MSF_ERR_INVALID_ARG;  // one point step per field step only
  const int64_t tw = t1 - t0;
  if (tw * d.P >= ((int64_t)1 << 31) || (vox && tw * d.V >= ((int64_t)1 << 31)))
    return MSF_ERR_TOO_LARGE;
  if (!labels && (vox || d.P > 0)) return MSF_ERR_INVALID_ARG;
  *n_pieces = 0;
  if (d.P == 0) return MSF_OK;
  MSF_CUDA_TRY(cudaSetDevice(c->device));
  SpareScope spare(c);
  PostScratch& S = c->post;
  PieceArgs a{};
  MSF_TRY(stage_in(c, labels, labels_kind, (size_t)(tw * (vox ? d.V : d.P)), S.in, &a.lab));
  a.key = d.key.as<int32_t>();
  a.P = d.P;
  a.V = d.V;
  a.t0 = t0;
  a.tw = (int)tw;
  a.min_len = min_len;
  MSF_TRY(S.cnt.ensure(sizeof(uint32_t) * (size_t)d.P));
  MSF_TRY(S.offs.ensure(sizeof(uint32_t) * (size_t)d.P));
  MSF_TRY(S.total.ensure(sizeof(uint32_t)));
  cudaStream_t s = c->stream;
  const unsigned g = blocks_for(d.P, 256, c->sm_count * 16);
  {
    ScopedKernel k(c, "k_pieces_count");
    if (vox) k_pieces<true, true><<<g, 256, 0, s>>>(a, S.cnt.as<uint32_t>());
    else k_pieces<false, true><<<g, 256, 0, s>>>(a, S.cnt.as<uint32_t>());
  }
  MSF_TRY(scan_exclusive_u32(c, S.cnt.as<uint32_t>(), S.offs.as<uint32_t>(), d.P, S.scan_tmp,
                             S.total.as<uint32_t>()));
  uint32_t n = 0;
  MSF_CUDA_TRY(cudaMemcpyAsync(&n, S.total.p, sizeof(n), cudaMemcpyDeviceToHost, s));
  MSF_CUDA_TRY(cudaStreamSynchronize(s));
  *n_pieces = n;
  if ((int64_t)n > cap) {
    c->timer.flush();
    return MSF_ERR_CAPACITY;
  }
  if (n) {
    int4* dst = reinterpret_cast<int4*>(pieces);
    if (pieces_kind == MSF_HOST) {
      MSF_TRY(S.out.ensure(sizeof(int4) * (size_t)n));
      dst = S.out.as<int4>();
    }
    a.offs = S.offs.as<uint32_t>();
    a.out = dst;
    {
      ScopedKernel k(c, "k_pieces_write");
      if (vox) k_pieces<true, false><<<g, 256, 0, s>>>(a, nullptr);
      else k_pieces<false, false><<<g, 256, 0, s>>>(a, nullptr);
    }
    MSF_CUDA_TRY(cudaGetLastError());
    if (pieces_kind == MSF_HOST)
      MSF_TRY(copy_out(c, reinterpret_cast<int4*>(pieces), MSF_HOST, (const int4*)dst, n));
    MSF_CUDA_TRY(cudaStreamSynchronize(s));
  }
  c->timer.flush();
  return MSF_OK;
}

}  // extern "C"

// crk_build.cu -- (a) cell-list build: validation and Morton keys, stable LSD
// radix sort, sorted particle arrays, a bounding-volume tree over buckets of
// eight consecutive sorted particles, and the per-particle union neighbor
// lists in a warp-interleaved layout.
//
// The paper's solver keeps particles in tree leaves of a few hundred
// particles and reuses that tree for hydro neighbor searches (Sec. 2.1,
// App. A.4); its GPU tree is built to minimise rebuild cost (Sec. 2.9).  Here
// the tree is a linear BVH over Morton-ordered buckets (one CUDA thread per
// node, no spin waits), and its only job is to produce neighbor lists that
// every later sweep reads without further distance tests.
#include <type_traits>

#include "crk_internal.cuh"

namespace crk {

// ---------------------------------------------------------------------------
// validation and keys
// ---------------------------------------------------------------------------
// What a build needs of each box: its side, cells per unit length of the Morton
// grid and the smallest float above half the side (h < L/2 for a float h is
// h < that).  Also clears the largest smoothing length of each box.
struct BoxScale {
  double cells_per_length;
  float half_up;
  int32_t pad;
};

__global__ void k_check_boxes(const int64_t* __restrict__ box_off, const double* __restrict__ box_L,
                              int32_t nb, int64_t n, int bits, double* __restrict__ wbox,
                              BoxScale* __restrict__ scale, unsigned int* __restrict__ hbox,
                              DevHeader* hdr) {
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b > nb) return;
  if (b == 0 && box_off[0] != 0) set_status(hdr, CRK_EINVAL);
  if (b == nb) {
    if (box_off[nb] != n) set_status(hdr, CRK_EINVAL);
    return;
  }
  if (box_off[b + 1] < box_off[b]) set_status(hdr, CRK_EINVAL);
  double L = box_L[b];
  if (!(L > 0.0) || !isfinite(L)) set_status(hdr, CRK_EINVAL);
  wbox[b] = L;
  scale[b] = BoxScale{(double)(1u << bits) / L, __double2float_ru(0.5 * L), 0};
  hbox[b] = 0u;
}

__device__ __forceinline__ int box_of(const int64_t* __restrict__ box_off, int32_t nb, int64_t i) {
  // largest b with box_off[b] <= i (empty boxes are skipped naturally)
  int lo = 0, hi = nb - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (box_off[mid] <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// 16 bits spread to every third of 48 by doubling steps
__device__ __forceinline__ uint64_t spread3(uint32_t v) {
  uint64_t r = v & 0xffffu;
  r = (r | (r << 16)) & 0x0000ff0000ffull;
  r = (r | (r << 8)) & 0x00f00f00f00full;
  r = (r | (r << 4)) & 0x0c30c30c30c3ull;
  return (r | (r << 2)) & 0x249249249249ull;
}

// Morton keys in caller order; also the largest smoothing length of each box
// (hbox, float bits): one atomic per block and box segment, since a block's
// consecutive particles lie in one box or a few; and, when cnt is given, the
// counts of each tile's first digits for the short sort.  FP64 arithmetic
// (1/64 of the FP32 rate here) is kept to the three products that place a
// particle in its cell; range checks compare bit patterns.
template <class R>
__global__ void __launch_bounds__(256) k_keys(const double* __restrict__ x, const R* __restrict__ h,
                       const int64_t* __restrict__ box_off, const double* __restrict__ wbox,
                       const BoxScale* __restrict__ scale, int32_t nb, int64_t n, int bits,
                       uint64_t* __restrict__ keys, int32_t* __restrict__ vals,
                       unsigned int* __restrict__ hbox, uint32_t* __restrict__ cnt, int tile_log2,
                       DevHeader* hdr) {
  __shared__ float wmax[8];
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x;
  int64_t i = i0 + threadIdx.x;
  const bool live = i < n;
  const int64_t ilast = min(i0 + (int64_t)blockDim.x, n) - 1;
  const int bfirst = box_of(box_off, nb, i0), blast = box_of(box_off, nb, ilast);
  const int b = bfirst == blast ? bfirst : (live ? box_of(box_off, nb, i) : bfirst);
  const R hi = live ? h[i] : R(1);
  float hmx = 0.f;
  if (live && isfinite(hi) && hi > R(0))
    hmx = sizeof(R) == 4 ? (float)hi : __double2float_ru((double)hi);
  if (bfirst == blast) {
    float m = hmx;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, wmax[w]);
      atomicMax(hbox + bfirst, __float_as_uint(m));
    }
  } else if (live) {
    atomicMax(hbox + b, __float_as_uint(hmx));
  }
  if (!live) return;
  const double L = wbox[b];
  const BoxScale sc = scale[b];
  const long long Lb = __double_as_longlong(L);
  const uint32_t cells = 1u << bits;
  uint32_t q[3];
  bool ok = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double xa = x[a * n + i];
    const long long xb = __double_as_longlong(xa);
    const bool finite = (xb & 0x7ff0000000000000ll) != 0x7ff0000000000000ll;
    // 0 <= x < L: order of the bit patterns of non-negative doubles (and -0)
    const bool inside = (xb >= 0 && xb < Lb) || (xb << 1) == 0;
    if (!finite) { set_status(hdr, CRK_ENONFINITE); ok = false; }
    else if (!inside) { set_status(hdr, CRK_EDOMAIN); ok = false; }
    const uint32_t t = ok ? __double2uint_rz(__dmul_rn(xa, sc.cells_per_length)) : 0u;
    q[a] = t < cells ? t : cells - 1u;
  }
  if (!isfinite(hi)) set_status(hdr, CRK_ENONFINITE);
  else if (!(hi > R(0) && (sizeof(R) == 4 ? (float)hi < sc.half_up : (double)hi < 0.5 * L)))
    set_status(hdr, CRK_EDOMAIN);
  const uint64_t key =
      ((uint64_t)b << 48) | (spread3(q[0]) << 2) | (spread3(q[1]) << 1) | spread3(q[2]);
  keys[i] = key;
  vals[i] = (int32_t)i;
  if (cnt) atomicAdd(cnt + ((i >> tile_log2) << 8) + (key & 0xff), 1u);
}

// ---------------------------------------------------------------------------
// device-wide exclusive scan (two levels of 4096-element blocks)
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanChunk = kScanThreads * kScanItems;

template <class T>
__device__ T block_exclusive_scan(T v, T* smem_warp, T& total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  T inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T t = __shfl_up_sync(kFull, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) smem_warp[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    T w = lane < (kScanThreads / 32) ? smem_warp[lane] : T(0);
    T wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T t = __shfl_up_sync(kFull, wi, o);
      if (lane >= o) wi += t;
    }
    if (lane < (kScanThreads / 32)) smem_warp[lane] = wi - w;
    if (lane == (kScanThreads / 32) - 1) smem_warp[kScanThreads / 32] = wi;
  }
  __syncthreads();
  T res = inc - v + smem_warp[wid];
  total = smem_warp[kScanThreads / 32];
  __syncthreads();
  return res;
}

template <class T>
__global__ void k_scan_reduce(const T* __restrict__ in, int64_t n, T* __restrict__ part) {
  __shared__ T sw[kScanThreads / 32 + 1];
  int64_t base = (int64_t)blockIdx.x * kScanChunk;
  T s = 0;
  for (int k = 0; k < kScanItems; ++k) {
    int64_t i = base + (int64_t)threadIdx.x * kScanItems + k;
    if (i < n) s += in[i];
  }
  T tot;
  block_exclusive_scan<T>(s, sw, tot);
  if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

// single block: exclusive scan of the per-chunk partials in place
template <class T>
__global__ void k_scan_partials(T* __restrict__ part, int64_t np, T* __restrict__ total_out) {
  __shared__ T sw[kScanThreads / 32 + 1];
  T carry = 0;
  for (int64_t base = 0; base < np; base += kScanThreads) {
    int64_t i = base + threadIdx.x;
    T v = i < np ? part[i] : T(0);
    T tot;
    T ex = block_exclusive_scan<T>(v, sw, tot);
    if (i < np) part[i] = ex + carry;
    carry += tot;
  }
  if (threadIdx.x == 0 && total_out) *total_out = carry;
}

template <class T>
__global__ void k_scan_apply(const T* __restrict__ in, int64_t n, const T* __restrict__ part,
                             T* __restrict__ out) {
  __shared__ T sw[kScanThreads / 32 + 1];
  int64_t base = (int64_t)blockIdx.x * kScanChunk + (int64_t)threadIdx.x * kScanItems;
  T loc[kScanItems];
  T s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    int64_t i = base + k;
    loc[k] = i < n ? in[i] : T(0);
    s += loc[k];
  }
  T tot;
  T ex = block_exclusive_scan<T>(s, sw, tot) + part[blockIdx.x];
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    int64_t i = base + k;
    if (i < n) out[i] = ex;
    ex += loc[k];
  }
}

int scan_launches(int64_t n) { return n <= 0 ? 0 : 3; }

size_t scan_tmp_bytes(int64_t n) {
  int64_t np = (n + kScanChunk - 1) / kScanChunk + 1;
  return (size_t)np * sizeof(int64_t) + 256;
}

// out[i] = sum_{k<i} in[k] for i < n, and (if total_out) the grand total.
template <class T>
void exclusive_scan(const T* in, T* out, int64_t n, void* tmp, T* total_out, cudaStream_t st) {
  int64_t np = (n + kScanChunk - 1) / kScanChunk;
  T* part = reinterpret_cast<T*>(tmp);
  if (np == 0) {
    if (total_out) cudaMemsetAsync(total_out, 0, sizeof(T), st);
    return;
  }
  k_scan_reduce<T><<<(unsigned)np, kScanThreads, 0, st>>>(in, n, part);
  k_scan_partials<T><<<1, kScanThreads, 0, st>>>(part, np, total_out);
  k_scan_apply<T><<<(unsigned)np, kScanThreads, 0, st>>>(in, n, part, out);
}
template void exclusive_scan<int64_t>(const int64_t*, int64_t*, int64_t, void*, int64_t*, cudaStream_t);
template void exclusive_scan<uint32_t>(const uint32_t*, uint32_t*, int64_t, void*, uint32_t*, cudaStream_t);

// ---------------------------------------------------------------------------
// stable LSD radix sort of (64-bit key, 32-bit value), 8 bits per pass
// ---------------------------------------------------------------------------
__global__ void k_rsort_hist(const uint64_t* __restrict__ kin, int64_t n, int shift, int ntiles,
                             uint32_t* __restrict__ hist) {
  __shared__ uint32_t cnt[256];
  cnt[threadIdx.x] = 0;
  __syncthreads();
  int64_t base = (int64_t)blockIdx.x * kSortTile;
  for (int r = 0; r < kSortTile / kSortThreads; ++r) {
    int64_t i = base + r * kSortThreads + threadIdx.x;
    if (i < n) atomicAdd(&cnt[(kin[i] >> shift) & 0xff], 1u);
  }
  __syncthreads();
  hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];
}

__global__ void k_rsort_scatter(const uint64_t* __restrict__ kin, const int32_t* __restrict__ vin,
                                uint64_t* __restrict__ kout, int32_t* __restrict__ vout,
                                const uint32_t* __restrict__ offs, int64_t n, int shift,
                                int ntiles) {
  __shared__ uint32_t base[256];
  __shared__ uint32_t wcnt[kSortThreads / 32][256];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  base[tid] = offs[(int64_t)tid * ntiles + blockIdx.x];
  const uint32_t lt = (1u << lane) - 1u;
  int64_t tile = (int64_t)blockIdx.x * kSortTile;
  for (int r = 0; r < kSortTile / kSortThreads; ++r) {
    int64_t i = tile + r * kSortThreads + tid;
    bool valid = i < n;
    uint64_t key = valid ? kin[i] : 0ull;
    int d = valid ? (int)((key >> shift) & 0xff) : 256;
#pragma unroll
    for (int w = 0; w < kSortThreads / 32; ++w) wcnt[w][tid] = 0;
    __syncthreads();
    unsigned peers = __match_any_sync(kFull, d);
    int rank = __popc(peers & lt);
    if (valid && rank == 0) wcnt[wid][d] = __popc(peers);
    __syncthreads();
    {
      uint32_t run = base[tid];
#pragma unroll
      for (int w = 0; w < kSortThreads / 32; ++w) {
        uint32_t c = wcnt[w][tid];
        wcnt[w][tid] = run;
        run += c;
      }
      base[tid] = run;
    }
    __syncthreads();
    if (valid) {
      uint32_t pos = wcnt[wid][d] + rank;
      kout[pos] = key;
      vout[pos] = vin[i];
    }
    __syncthreads();
  }
}

// One pass of the short sort (up to kShortTiles tiles, one block each): a launch
// per digit instead of five.  The block adds up the tiles' digit counts itself
// -- where its own tile's keys of each digit go, given the tiles before it -- and
// counts the next digit of every key at the tile it lands in.  Counts arrive
// zeroed.  Sort phase (keys included) against a histogram, a three-kernel scan and
// a scatter per digit: 30,011 particles 0.126 -> 0.048 ms, 262,144 0.157 -> 0.070
// (256 tiles of half the size 0.091).
constexpr int kShortThreads = 1024;
constexpr int kShortTiles = 152;
__global__ void __launch_bounds__(kShortThreads)
    k_short_sort(const uint64_t* __restrict__ kin, const int32_t* __restrict__ vin,
                 uint64_t* __restrict__ kout, int32_t* __restrict__ vout,
                 const uint32_t* __restrict__ cnt, uint32_t* __restrict__ cnt_next, int64_t n,
                 int shift, int shift_next, int ntiles, int tile_log2) {
  constexpr int NWARP = kShortThreads / 32;
  __shared__ uint32_t wcnt[NWARP][256];
  __shared__ uint32_t part[2][4][256];
  __shared__ uint32_t base[256];
  __shared__ uint32_t wsum[8];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  // keys of digit d = tid % 256 in all tiles and in the tiles before this one; a
  // quarter of the tiles per group of 256 threads
  {
    const int d = tid & 255, g = tid >> 8;
    uint32_t tot = 0, pre = 0;
#pragma unroll 8
    for (int b = g; b < ntiles; b += 4) {
      const uint32_t c = cnt[b * 256 + d];
      tot += c;
      if (b < (int)blockIdx.x) pre += c;
    }
    part[0][g][d] = tot;
    part[1][g][d] = pre;
  }
  __syncthreads();
  uint32_t tot = 0, inc = 0;
  if (tid < 256) {
    tot = part[0][0][tid] + part[0][1][tid] + part[0][2][tid] + part[0][3][tid];
    inc = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) wsum[wid] = inc;
  }
  __syncthreads();
  if (tid < 256) {
    uint32_t before = 0;
    for (int w = 0; w < wid; ++w) before += wsum[w];
    base[tid] = before + inc - tot + part[1][0][tid] + part[1][1][tid] + part[1][2][tid] +
                part[1][3][tid];
  }
  const int64_t first = (int64_t)blockIdx.x << tile_log2;
  const int rounds = 1 << (tile_log2 - 10);
  for (int r = 0; r < rounds; ++r) {
    const int64_t i = first + r * kShortThreads + tid;
    if (first + r * kShortThreads >= n) break;  // whole block
    const bool valid = i < n;
    const uint64_t key = valid ? kin[i] : 0ull;
    const int32_t val = valid ? vin[i] : 0;
    const int d = valid ? (int)((key >> shift) & 0xff) : 256;
    for (int k = tid; k < NWARP * 256; k += kShortThreads) (&wcnt[0][0])[k] = 0;
    __syncthreads();
    const unsigned peers = __match_any_sync(kFull, d);
    const int rank = __popc(peers & lt);
    if (valid && rank == 0) wcnt[wid][d] = __popc(peers);
    __syncthreads();
    if (tid < 256) {
      uint32_t run = base[tid];
#pragma unroll
      for (int w = 0; w < NWARP; ++w) {
        const uint32_t c = wcnt[w][tid];
        wcnt[w][tid] = run;
        run += c;
      }
      base[tid] = run;
    }
    __syncthreads();
    if (valid) {
      const uint32_t pos = wcnt[wid][d] + rank;
      kout[pos] = key;
      vout[pos] = val;
      if (shift_next >= 0)
        atomicAdd(cnt_next + ((pos >> tile_log2) << 8) + ((key >> shift_next) & 0xff), 1u);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// sorted particle arrays
// ---------------------------------------------------------------------------
__device__ __forceinline__ void put_x(float* xs, int64_t n, int64_t s, const double* xd) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float hi = __double2float_rn(xd[a]);
    float lo = __double2float_rn(xd[a] - (double)hi);
    xs[a * n + s] = hi;
    xs[(3 + a) * n + s] = lo;
  }
}
__device__ __forceinline__ void put_x(double* xs, int64_t n, int64_t s, const double* xd) {
#pragma unroll
  for (int a = 0; a < 3; ++a) xs[a * n + s] = xd[a];
}

// ---------------------------------------------------------------------------
// bucket tree (linear BVH over buckets of kBucket sorted particles)
// node index: internal nodes [0, ni), bucket b is node ni + b; one 64-byte record
// per node: lo[3], hi[3], h_max, box range, the two children (-1 for a bucket).
//
// A node of a radix tree over sorted keys covers a range of consecutive
// buckets, so its bounds need no bottom-up pass over the tree (one atomic and a
// fence per level and node: 0.077 ms of a 0.118 ms phase on 262,144
// particles, nearly all of it waiting).  A segment tree over the buckets -- level
// k, entry i bounding buckets [i 2^k, (i+1) 2^k) -- is reduced in shared memory,
// and the kernel that finds a node's range unites the few entries that tile it.
// The minimum and maximum of the same floats come out the same either way.
// ---------------------------------------------------------------------------
constexpr int kSegW = 8;          // words per segment entry: lo[3], hi[3], h_max, padding
constexpr int kSegLeafLevels = 5;  // levels reduced by the block that makes the buckets
constexpr int kSegUpLevels = 10;   // levels reduced per further pass
constexpr int kSegMax = 31;

struct SegTree {
  float* base;
  int64_t off[kSegMax + 1];  // first entry of each level
  int64_t cnt[kSegMax + 1];
  int levels;  // levels with entries (the last has one)
};

// 32-byte read-only load (one 256-bit access)
__device__ __forceinline__ void ld8(const float* p, float* o) {
  asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3]), "=f"(o[4]), "=f"(o[5]), "=f"(o[6]),
        "=f"(o[7])
      : "l"(p));
}

// word f of the union of two entries
__device__ __forceinline__ float seg_join(int f, float a, float b) {
  return f < 3 ? fminf(a, b) : fmaxf(a, b);
}

__device__ __forceinline__ void store_node(float* nrec, int64_t node, const float* box, int32_t b0,
                                           int32_t b1, int32_t c0, int32_t c1) {
  float4* o = reinterpret_cast<float4*>(nrec + node * kNodeRec);
  o[0] = make_float4(box[0], box[1], box[2], box[3]);
  o[1] = make_float4(box[4], box[5], box[6], __int_as_float(b0));
  o[2] = make_float4(__int_as_float(b1), __int_as_float(c0), __int_as_float(c1), 0.f);
}

// Reduces `levels` levels above the 2^levels entries e (shared memory, entry k at
// e + k * kSegW) of level `lev`, the block's first being entry `first`.
__device__ __forceinline__ void seg_reduce(float* e, const SegTree& t, int lev, int levels,
                                           int64_t first) {
  for (int l = 1; l <= levels && lev + l < t.levels; ++l) {
    const int cnt = (1 << levels) >> l;
    const int64_t f0 = first >> l;
    __syncthreads();
    float v[4];
    int q = 0;
    for (int k = threadIdx.x; k < cnt * kSegW; k += blockDim.x, ++q) {
      const int i = k / kSegW, f = k % kSegW;
      v[q] = seg_join(f, e[2 * i * kSegW + f], e[(2 * i + 1) * kSegW + f]);
    }
    __syncthreads();
    q = 0;
    for (int k = threadIdx.x; k < cnt * kSegW; k += blockDim.x, ++q) {
      e[k] = v[q];
      const int64_t at = f0 + k / kSegW;
      if (at < t.cnt[lev + l]) t.base[(t.off[lev + l] + at) * kSegW + k % kSegW] = v[q];
    }
  }
}

// Sorted particle arrays, the buckets' bounds and node records, the buckets'
// keys and the first levels of the segment tree; 256 particles (32 buckets) a
// block.
template <class R>
__global__ void __launch_bounds__(256)
    k_gather_sorted(const uint64_t* __restrict__ keys, const int32_t* __restrict__ idx,
                    const double* __restrict__ x, const R* __restrict__ h, int64_t n, int64_t nbk,
                    int64_t ni, int32_t* __restrict__ perm, int32_t* __restrict__ boxid,
                    R* __restrict__ xs, R* __restrict__ hs, float4* __restrict__ p4,
                    uint64_t* __restrict__ bkey, float* __restrict__ nrec, const SegTree seg) {
  static_assert(256 / kBucket == 1 << kSegLeafLevels, "a block's buckets fill the first levels");
  __shared__ float e[(256 / kBucket) * kSegW];
  const int64_t s = (int64_t)blockIdx.x * 256 + threadIdx.x;
  float box[7] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY, 0.f};
  int32_t bx = 0;
  uint64_t key = 0;
  if (s < n) {
    const int32_t p = idx[s];
    key = keys[s];
    perm[s] = p;
    bx = (int32_t)(key >> 48);
    boxid[s] = bx;
    double xd[3] = {x[p], x[n + p], x[2 * n + p]};
    put_x(xs, n, s, xd);
    const R hp = h[p];
    hs[s] = hp;
    // float position (round to nearest, the high part of the split position)
    // and h for the list build's float candidate test
    const float f[3] = {__double2float_rn(xd[0]), __double2float_rn(xd[1]),
                        __double2float_rn(xd[2])};
    p4[s] = make_float4(f[0], f[1], f[2], (float)hp);
    // bounds that contain the position: the float one float step to each side
    // in the mixed form (no FP64 arithmetic), rounded down and up in the other
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if constexpr (sizeof(R) == 4) {
        box[a] = nextafterf(f[a], -INFINITY);
        box[3 + a] = nextafterf(f[a], INFINITY);
      } else {
        box[a] = __double2float_rd(xd[a]);
        box[3 + a] = __double2float_ru(xd[a]);
      }
    }
    box[6] = sizeof(R) == 4 ? (float)hp : __double2float_ru((double)hp);
  }
  const int32_t b0 = __shfl_sync(kFull, bx, (threadIdx.x & 31) & ~(kBucket - 1));
  int32_t b1 = bx;  // box of the bucket's last particle: the largest (boxes are sorted)
#pragma unroll
  for (int o = 1; o < kBucket; o <<= 1) {
#pragma unroll
    for (int f = 0; f < 7; ++f) box[f] = seg_join(f, box[f], __shfl_xor_sync(kFull, box[f], o));
    b1 = max(b1, __shfl_xor_sync(kFull, b1, o));
  }
  const int64_t bk = s / kBucket;
  if ((threadIdx.x & (kBucket - 1)) == 0) {
    float* o = e + (threadIdx.x / kBucket) * kSegW;
#pragma unroll
    for (int f = 0; f < 7; ++f) o[f] = box[f];
    o[7] = 0.f;
    if (bk < nbk) {
      bkey[bk] = key;
      store_node(nrec, ni + bk, box, b0, b1, -1, -1);
      float4* g = reinterpret_cast<float4*>(seg.base + bk * kSegW);
      g[0] = make_float4(box[0], box[1], box[2], box[3]);
      g[1] = make_float4(box[4], box[5], box[6], 0.f);
    }
  }
  seg_reduce(e, seg, 0, kSegLeafLevels, (int64_t)blockIdx.x << kSegLeafLevels);
}

// kSegUpLevels further levels above level `lev`; 1024 entries a block.
__global__ void __launch_bounds__(1024) k_seg_up(const SegTree seg, int lev) {
  __shared__ float e[(1 << kSegUpLevels) * kSegW];
  const int64_t first = (int64_t)blockIdx.x << kSegUpLevels;
  const int64_t at = first + threadIdx.x;
  float box[8] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY, 0.f, 0.f};
  if (at < seg.cnt[lev]) ld8(seg.base + (seg.off[lev] + at) * kSegW, box);
#pragma unroll
  for (int f = 0; f < 8; ++f) e[threadIdx.x * kSegW + f] = box[f];
  seg_reduce(e, seg, lev, kSegUpLevels, first);
}

__device__ __forceinline__ int lbvh_delta(const uint64_t* __restrict__ bkey, int64_t nbk, int64_t i,
                                          int64_t j) {
  if (j < 0 || j >= nbk) return -1;
  const uint64_t a = bkey[i], b = bkey[j];
  if (a == b) return 64 + __clz((uint32_t)(i ^ j));
  return __clzll(a ^ b);
}

// Karras (2012) radix-tree construction, one thread per internal node; its
// bounds from the segment entries that tile its range of buckets.
__global__ void k_lbvh(const uint64_t* __restrict__ bkey, const int32_t* __restrict__ boxid,
                       int64_t n, int64_t nbk, int64_t ni, const SegTree seg,
                       float* __restrict__ nrec) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ni) return;
  int d = (lbvh_delta(bkey, nbk, i, i + 1) - lbvh_delta(bkey, nbk, i, i - 1)) >= 0 ? 1 : -1;
  int dmin = lbvh_delta(bkey, nbk, i, i - d);
  int64_t lmax = 2;
  while (lbvh_delta(bkey, nbk, i, i + lmax * d) > dmin) lmax <<= 1;
  int64_t l = 0;
  for (int64_t t = lmax >> 1; t >= 1; t >>= 1)
    if (lbvh_delta(bkey, nbk, i, i + (l + t) * d) > dmin) l += t;
  int64_t j = i + l * d;
  int dnode = lbvh_delta(bkey, nbk, i, j);
  int64_t s = 0, t = l;
  do {
    t = (t + 1) >> 1;
    if (lbvh_delta(bkey, nbk, i, i + (s + t) * d) > dnode) s += t;
  } while (t > 1);
  int64_t gamma = i + s * d + (d < 0 ? -1 : 0);
  const int64_t lo = min(i, j), hi = max(i, j);
  const int32_t left = (lo == gamma) ? (int32_t)(ni + gamma) : (int32_t)gamma;
  const int32_t right = (hi == gamma + 1) ? (int32_t)(ni + gamma + 1) : (int32_t)(gamma + 1);
  float box[8] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY, 0.f, 0.f};
  auto join = [&](int lev, int64_t at) {
    float q[8];
    ld8(seg.base + (seg.off[lev] + at) * kSegW, q);
#pragma unroll
    for (int f = 0; f < 7; ++f) box[f] = seg_join(f, box[f], q[f]);
  };
  int64_t a = lo, b = hi + 1;
  for (int lev = 0; a < b; ++lev, a >>= 1, b >>= 1) {
    if (a & 1) join(lev, a++);
    if (b & 1) join(lev, --b);
  }
  store_node(nrec, i, box, boxid[lo * kBucket], boxid[min(n, (hi + 1) * kBucket) - 1], left,
             right);
}

// ---------------------------------------------------------------------------
// neighbor lists: one warp per 32 sorted particles traverses the tree
// ---------------------------------------------------------------------------
// r^2 as the definition forms it (no contraction)
__device__ __forceinline__ double norm2(const double* d) {
  return __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
}
__device__ __forceinline__ double sq(double a) { return __dmul_rn(a, a); }

// Exact pair predicate.  The float candidate test of both forms works on
// positions rounded to float (and shifted by a float L to an image), so r^2
// carries an error of at most 2^-24 (10 sqrt(3) L r + 6 r^2) against the double
// r^2 of the caller's positions (each coordinate within 5 * 2^-24 L of its exact
// image difference, three roundings in the sum of squares), and a float h^2 of
// at most 3 * 2^-24 h^2 (one rounding, and in the FP64 form h rounded to
// float).  A decision r^2 < h^2 is therefore certain outside the band
// |r^2 - h^2| <= tol(h) below (wider by a third in the L term and more in the
// h^2 term, and by 2^-123 for what the five operations on the way flush to 0, each
// less than 2^-126: it is never 0, so equality of two flushed values is uncertain);
// inside it the pair is decided again in double exactly as the definition states --
// minimum image decided and formed in double, r^2 summed without contraction, compared
// with the squared smoothing lengths -- so the lists of both forms are those of the
// double predicate.  (Testing every candidate of the FP64 form in double took 2.89 ms
// of its build on 13,824 particles: GB300 runs FP64 at 1/64 of the FP32 rate.)
__device__ __forceinline__ float list_band(float h, float L) {
  return 0x1p-24f * fmaf(16.f * h, h, fmaf(24.f * L, h, 0x1p-99f));
}
__device__ __forceinline__ double exact_r2(const double* __restrict__ xd, int64_t n, int64_t pi,
                                           int64_t pj, double L) {
  const double a[3] = {xd[pi], xd[n + pi], xd[2 * n + pi]};
  const double b[3] = {xd[pj], xd[n + pj], xd[2 * n + pj]};
  double d[3];
  separation(a, b, L, 0.5 * L, d);
  return norm2(d);
}
// One warp per 32 consecutive sorted particles walks the tree once for the
// whole group (separately for each box present in the group): nodes are
// tested 32 at a time against the group's bounding box grown by
// max(h over the group, h_max of the node); overlapping buckets are staged
// 4 or 8 at a time (32 or 64 particles) in shared memory and every lane tests its own
// particle against all 32.  Traversal order is
// fixed, so the counting and the filling pass see the same entries.
// Center, half extent and largest h of the lanes with `in` set (all lanes
// take part in the shuffles).
__device__ __forceinline__ void group_bounds(bool in, const float* p, float h, float* gc, float* ge,
                                             float& hg) {
  float lo[3], hi[3];
  hg = in ? h : 0.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = in ? p[a] : 3.0e38f;
    hi[a] = in ? p[a] : -3.0e38f;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      lo[a] = fminf(lo[a], __shfl_xor_sync(kFull, lo[a], o));
      hi[a] = fmaxf(hi[a], __shfl_xor_sync(kFull, hi[a], o));
    }
    hg = fmaxf(hg, __shfl_xor_sync(kFull, hg, o));
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    gc[a] = 0.5f * (lo[a] + hi[a]);
    ge[a] = 0.5f * (hi[a] - lo[a]);
  }
}

// Resident blocks per SM, of one warp each (80 registers a thread, 5 KB of shared
// memory a block).  The walks of neighboring groups differ by a factor of two and
// more in length, so a block of four warps held its place until the slowest of them
// ended.  The build is bound by issue: of a warp's time a quarter each is the tree
// walk, the staging of candidates and the emission of hits, a sixth the
// 32-candidate tests.  Lists of 30,011 / 262,144 / 2.1 M particles: 0.215 / 0.685 /
// 4.5 ms with distances and bands evaluated again per hit, 0.201 / 0.556 / 3.63 with
// the masks, 0.186 / 0.537 / 3.58 with eight buckets staged at once and box numbers
// read only where a bucket holds two boxes, 0.164 / 0.470 / 3.08 with blocks of one
// warp (20 a SM 0.174 / 0.519 / 3.52, 28 a SM 0.178 / 0.476 / 3.05; two warps a block
// 0.188 / 0.535 / 3.48).
constexpr int kNbrBlocks = 24;
// Node stack of a warp.  Taking 32 nodes a step adds at most 32 to it; from
// three quarters on the walk takes one node a step, which adds at most one per
// level of the tree (94 at most: 64 key bits and 30 index bits), so it cannot
// overflow.  (The deepest seen with 32 a step: 268, the clumpy 128^3 box.)
constexpr int kNodeStack = 512;
// Staged candidates: a ring of three stages of 32, since up to 64 are appended to
// at most 31 that wait.
constexpr int kStage = 96;

template <class R>
__global__ void __launch_bounds__(32, kNbrBlocks) k_nbr(
    const uint64_t* __restrict__ keys, const R* __restrict__ hs, const int32_t* __restrict__ boxid,
    const double* __restrict__ box_L, int64_t n, int64_t ni, const float* __restrict__ nrec,
    const float4* __restrict__ p4, int32_t* __restrict__ cnt_g, int32_t* __restrict__ cnt_s,
    int32_t* __restrict__ wlen_g, int32_t* __restrict__ wlen_s, uint32_t* __restrict__ ell,
    int64_t cap_pp, DevHeader* hdr, const double* __restrict__ xd,
    const int32_t* __restrict__ perm, const float* __restrict__ hbox) {
  __shared__ int32_t stk[kNodeStack];
  // candidate buckets; the top bit marks one that may hold particles of two boxes
  __shared__ int32_t cand[64];
  // staged candidates, one array per component so that four (a 128-bit load)
  // arrive at once: float position (of the nearest image, where one serves the
  // whole group), h^2, its rounding band, index; and the slot of each lane's own
  // particle (-kStage: not staged)
  __shared__ float4 stage[5][kStage / 4];
  __shared__ int32_t sj[kStage];
  __shared__ int32_t self_at[32];
  const int lane = threadIdx.x;
  const int64_t w = blockIdx.x;
  const uint32_t lt = (1u << lane) - 1u;
  const int64_t s = w * 32 + lane;
  const bool live = s < n;
  float hi = 0.f;
  int32_t bi = -1;
  float p[3] = {0.f, 0.f, 0.f};
  if (live) {
    const float4 own = p4[s];
    p[0] = own.x;
    p[1] = own.y;
    p[2] = own.z;
    hi = own.w;
    bi = boxid[s];
  }
  // gather entries fill this lane's column from the front, scatter-only
  // entries from the back (moved up at the end); kg + ks > cap_pp means the
  // column overflowed
  int kg = 0, ks = 0;
  uint32_t* col = ell + w * cap_pp * 32 + lane;
  bool overflow = false;
  unsigned long long cnt_nodes = 0, cnt_buckets = 0;
  // Lane groups to traverse: one per box present in the warp, each split at
  // its highest differing Morton bit when that shrinks the searched volume
  // (32 consecutive keys can straddle a coarse octree boundary and then span
  // much of the box).
  const uint64_t mykey = live ? keys[s] : 0ull;
  unsigned todo[8];
  int ntodo = 0;
  unsigned remaining = __ballot_sync(kFull, live);
  while (remaining || ntodo) {
    unsigned m;
    if (ntodo == 0) {
      const int l0 = __ffs(remaining) - 1;
      const int32_t b0 = __shfl_sync(kFull, bi, l0);
      m = __ballot_sync(kFull, live && bi == b0);
      remaining &= ~m;
    } else {
      m = todo[--ntodo];
    }
    const bool act = (m >> lane) & 1u;
    const int lead = __ffs(m) - 1;
    const int32_t b = __shfl_sync(kFull, bi, lead);
    const double Ld = box_L[b];
    const float Lf = (float)Ld, halfLf = (float)(0.5 * Ld);
    float gc[3], ge[3], hg;
    group_bounds(act, p, hi, gc, ge, hg);
    // one image of a candidate, the one nearest the group's center, serves
    // every pair in reach when the group extent plus the largest search radius
    // stays below half the box; otherwise every pair wraps on its own
    const float reach = fmaxf(hg, __ldg(hbox + b));  // the largest h of the box
    const bool one_image = 2.f * fmaxf(ge[0], fmaxf(ge[1], ge[2])) + reach < 0.49f * Lf;
    if (__popc(m) > 2 && ntodo <= 6) {
      const uint64_t lk = __shfl_sync(kFull, mykey, lead);
      uint64_t kx = act ? (mykey ^ lk) : 0ull;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) kx |= __shfl_xor_sync(kFull, kx, o);
      if (kx != 0ull) {
        const int P = 63 - __clzll(kx);
        const unsigned m1 = __ballot_sync(kFull, act && ((mykey >> P) & 1ull));
        const unsigned m0 = m & ~m1;
        float c0[3], e0[3], h0, c1[3], e1[3], h1;
        group_bounds((m0 >> lane) & 1u, p, hi, c0, e0, h0);
        group_bounds((m1 >> lane) & 1u, p, hi, c1, e1, h1);
        const float V = (2.f * ge[0] + 2.f * hg) * (2.f * ge[1] + 2.f * hg) * (2.f * ge[2] + 2.f * hg);
        const float V0 = (2.f * e0[0] + 2.f * h0) * (2.f * e0[1] + 2.f * h0) * (2.f * e0[2] + 2.f * h0);
        const float V1 = (2.f * e1[0] + 2.f * h1) * (2.f * e1[1] + 2.f * h1) * (2.f * e1[2] + 2.f * h1);
        if (m0 && m1 && V > 1.5f * (V0 + V1)) {
          todo[ntodo++] = m1;
          todo[ntodo++] = m0;
          continue;
        }
      }
    }
    int sp = 0, nc = 0;
    int base = 0;  // first slot of the stage that is tested next
    int ns = 0;    // candidates waiting from there on
    const float hi2f = hi * hi;
    const float tol_i = list_band(hi, Lf);
    const float iLf = 1.f / Lf;
    // outside this range of box sides float squares could leave the float range:
    // every pair is then decided exactly
    const bool in_range = Lf > 1e-6f && Lf < 1e15f;
    float* sx = reinterpret_cast<float*>(stage);  // component c, slot k: sx[kStage c + k]
    self_at[lane] = -kStage;
    // Tests the first 32 staged candidates (`filled` of them valid) against the
    // lane's particle and appends the hits to its column.  Branch-free into
    // three bit masks, two candidates per packed operation: gather
    // (r^2 < h_i^2), scatter (r^2 < h_j^2) and, within the rounding band of
    // either, uncertain; the sign bit of a difference is shifted into its mask.
    // The few uncertain pairs are decided exactly; then only the hits are
    // walked, each an index load and a store.  That walk diverges (a warp runs it
    // as often as its busiest lane has hits), so nothing is evaluated in it: with
    // the distance and both bands recomputed per hit it took two thirds of the
    // build's instructions (442 million on 262,144 particles).  WRAP: minimum image
    // per coordinate (the box length times the rounded quotient, subtracted).
    auto test_stage = [&](int filled, auto wrap) {
      using D2 = F2;
      const D2 px = dup2(p[0]), py = dup2(p[1]), pz = dup2(p[2]);
      const D2 minus = dup2(-1.f), nhi2 = dup2(-hi2f);
      const D2 iL2 = dup2(iLf), nL2 = dup2(-Lf), mg = dup2(12582912.f), nmg = dup2(-12582912.f);
      uint32_t G = 0u, S = 0u, X = 0u;
      const int b4 = base >> 2;
      auto image = [&](D2 d) {
        if constexpr (decltype(wrap)::value)
          d = fma2(add2(fma2(d, iL2, mg), nmg), nL2, d);
        return d;
      };
#pragma unroll
      for (int q = 7; q >= 0; --q) {
        const float4 tx = stage[0][b4 + q], ty = stage[1][b4 + q], tz = stage[2][b4 + q];
        const float4 th = stage[3][b4 + q], tt = stage[4][b4 + q];
        const float* vx = &tx.x;
        const float* vy = &ty.x;
        const float* vz = &tz.x;
        const float* vh = &th.x;
        const float* vt = &tt.x;
#pragma unroll
        for (int u = 1; u >= 0; --u) {
          const D2 dx = image(fma2(mk2(vx[2 * u], vx[2 * u + 1]), minus, px));
          const D2 dy = image(fma2(mk2(vy[2 * u], vy[2 * u + 1]), minus, py));
          const D2 dz = image(fma2(mk2(vz[2 * u], vz[2 * u + 1]), minus, pz));
          const D2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
          float a[2], c[2];
          get2(add2(r2, nhi2), a[0], a[1]);
          get2(fma2(mk2(vh[2 * u], vh[2 * u + 1]), minus, r2), c[0], c[1]);
#pragma unroll
          for (int v = 1; v >= 0; --v) {
            G = __funnelshift_l(__float_as_uint(a[v]), G, 1);
            S = __funnelshift_l(__float_as_uint(c[v]), S, 1);
            const float m = fminf(fabsf(a[v]) - tol_i, fabsf(c[v]) - vt[2 * u + v]);
            X = __funnelshift_l(__float_as_uint(m), X, 1);
          }
        }
      }
      uint32_t valid = filled < 32 ? (1u << filled) - 1u : kFull;
      const unsigned own = (unsigned)(self_at[lane] - base);
      if (own < 32u) {
        valid &= ~(1u << own);
        self_at[lane] = -kStage;
      }
      X = in_range ? X & valid : valid;
      while (X) {
        const int k = __ffs(X) - 1;
        X &= X - 1u;
        const int32_t j = sj[base + k];
        const double r2d = exact_r2(xd, n, perm[s], perm[j], Ld);
        const uint32_t bit = 1u << k;
        G = r2d < sq((double)hs[s]) ? G | bit : G & ~bit;
        S = r2d < sq((double)hs[j]) ? S | bit : S & ~bit;
      }
      G &= valid;
      S &= valid;
      uint32_t U = G | S;
      while (U) {
        const int k = __ffs(U) - 1;
        U &= U - 1u;
        const uint32_t g = (G >> k) & 1u;
        const uint32_t e = (uint32_t)sj[base + k] | g << 31 | ((S >> k) & 1u) << 30;
        const int at = g ? kg : (int)cap_pp - 1 - ks;
        if (kg + ks < (int)cap_pp) col[at * 32] = e;
        kg += (int)g;
        ks += 1 - (int)g;
      }
    };
    auto flush = [&](int filled) {
      if (act) {
        if (one_image) test_stage(filled, std::false_type{});
        else test_stage(filled, std::true_type{});
      }
    };
    if (lane == 0) stk[0] = (ni > 0) ? 0 : (int32_t)ni;
    sp = 1;
    __syncwarp();
    while (sp > 0 || nc > 0) {
      if (sp > 0) {
        // one node at a time (depth first) once the stack is three quarters full
        const int take = sp > kNodeStack * 3 / 4 ? 1 : (sp < 32 ? sp : 32);
        const int32_t node = lane < take ? stk[sp - take + lane] : -1;
        sp -= take;
        cnt_nodes += take;
        __syncwarp();
        bool ov = false, one_box = false;
        int2 ch = make_int2(0, 0);
        if (node >= 0) {
          // the whole node record (bounds, h_max, box range, children) in
          // two 256-bit loads
          float nr[16];
          ld8(nrec + (int64_t)node * kNodeRec, nr);
          ld8(nrec + (int64_t)node * kNodeRec + 8, nr + 8);
          const int32_t b0 = __float_as_int(nr[7]), b1 = __float_as_int(nr[8]);
          const float hm = nr[6];
          const float* lo = nr;
          const float* hi_ = nr + 3;
          ch = make_int2(__float_as_int(nr[9]), __float_as_int(nr[10]));
          one_box = b0 == b1;
          if (b >= b0 && b <= b1) {
            // rounded as written (fma_, rmul): which nodes overlap sets the order of
            // the lists, and with it the sums' rounding
            const float R_ = fma_(1e-6f, Lf, rmul(fmaxf(hg, hm), 1.00001f));
            float g2 = 0.f;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              float dd = gc[a] - 0.5f * (lo[a] + hi_[a]);
              if (dd > halfLf) dd -= Lf;
              else if (dd < -halfLf) dd += Lf;
              dd = fabsf(dd) - ge[a] - 0.5f * (hi_[a] - lo[a]);
              if (dd > 0.f) g2 = fma_(dd, dd, g2);
            }
            ov = g2 <= R_ * R_;
          }
        }
        const bool leaf = node >= ni;
        const unsigned ml = __ballot_sync(kFull, ov && leaf);
        const unsigned mi = __ballot_sync(kFull, ov && !leaf);
        if (ov && leaf)
          cand[nc + __popc(ml & lt)] = (node - (int32_t)ni) | (one_box ? 0 : (int32_t)0x80000000);
        nc += __popc(ml);
        const int npush = 2 * __popc(mi);
        if (sp + npush > kNodeStack) {
          overflow = true;
          break;
        }
        if (ov && !leaf) {
          const int at = sp + 2 * __popc(mi & lt);
          stk[at] = ch.x;
          stk[at + 1] = ch.y;
        }
        sp += npush;
        __syncwarp();
      }
      while (nc >= 4 || (sp == 0 && nc > 0)) {
        // stage the particles of the last four candidate buckets, or of the last
        // two fours: the loads of both are in flight together
        const int take = nc < 4 ? nc : 4;
        const bool two = nc >= 8;
        cnt_buckets += two ? 8 : take;
        const int kb = lane >> 3;
        int64_t jj[2];
        float4 pj[2];
        int32_t bj[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const bool has = t == 0 ? kb < take : two;
          const int32_t c = has ? cand[(t == 0 ? nc - take : nc - 8) + kb] : 0;
          jj[t] = (int64_t)(c & 0x7fffffff) * kBucket + (lane & 7);
          pj[t] = make_float4(0.f, 0.f, 0.f, 0.f);
          bj[t] = -1;
          if (has && jj[t] < n) {
            pj[t] = __ldg(p4 + jj[t]);
            bj[t] = c < 0 ? __ldg(boxid + jj[t]) : b;
          }
        }
        nc -= two ? 8 : take;
        // A particle that lies farther from the group's box than
        // max(h_group, h_j) cannot be a union neighbor of any lane and is
        // dropped here; the others are appended to the stage, which is tested
        // once it holds 32.  Dropping preserves the order of the survivors, so
        // every list comes out exactly as without the filter.
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          float q[3] = {pj[t].x, pj[t].y, pj[t].z};
          const float hj = pj[t].w;
          float g2 = 0.f;
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const float dd = gc[a] - q[a];
            const float qn = q[a] + (dd > halfLf ? Lf : (dd < -halfLf ? -Lf : 0.f));
            const float o = fabsf(qn - gc[a]) - ge[a];
            if (o > 0.f) g2 += o * o;
            if (one_image) q[a] = qn;
          }
          const float Rj = fmaxf(hg, hj) * 1.00001f + 1e-6f * Lf;
          const bool pass = bj[t] == b && g2 <= Rj * Rj;
          const unsigned mp = __ballot_sync(kFull, pass);
          if (pass) {
            int at = base + ns + __popc(mp & lt);
            at -= at >= kStage ? kStage : 0;
#pragma unroll
            for (int a = 0; a < 3; ++a) sx[kStage * a + at] = q[a];
            sx[kStage * 3 + at] = hj * hj;
            sx[kStage * 4 + at] = list_band(hj, Lf);
            sj[at] = (int32_t)jj[t];
            if ((jj[t] >> 5) == w) self_at[jj[t] & 31] = at;
          }
          ns += __popc(mp);
        }
        __syncwarp();
        while (ns >= 32) {
          flush(32);
          base = base == kStage - 32 ? 0 : base + 32;
          ns -= 32;
        }
        __syncwarp();
      }
    }
    if (ns > 0) {
      flush(ns);  // the last partial stage
      __syncwarp();
      ns = 0;
    }
    if (overflow) break;
  }
  if (overflow && lane == 0) set_status(hdr, CRK_ENOMEM);
  const int need = kg + ks;
  if (need > cap_pp) set_status(hdr, CRK_ENOMEM);
  // a column that overflowed is left empty: its later slots were not written
  const int cg = need <= cap_pp ? kg : 0;
  const int cs = need <= cap_pp ? ks : 0;
  // close the gap: scatter-only entry t moves from slot cap_pp - 1 - t to
  // cg + t, so that a union list is slots 0 .. cg + cs - 1 in the order found
  {
    const int gap = (int)cap_pp - cg - cs;
    uint32_t* c0 = col;
    if (cs <= gap) {
      for (int t = 0; t < cs; t += 4) {
        uint32_t e[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          e[q] = t + q < cs ? c0[(cap_pp - 1 - t - q) * 32] : 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (t + q < cs) c0[(int64_t)(cg + t + q) * 32] = e[q];
      }
    } else if (cs > 0) {
      // a nearly full column: the two ranges overlap; reverse, then shift down
      uint32_t* r0 = c0 + (cap_pp - cs) * 32;
      for (int t = 0; t < cs / 2; ++t) {
        const uint32_t x = r0[(int64_t)t * 32], y = r0[(int64_t)(cs - 1 - t) * 32];
        r0[(int64_t)t * 32] = y;
        r0[(int64_t)(cs - 1 - t) * 32] = x;
      }
      for (int t = 0; gap > 0 && t < cs; ++t) c0[(int64_t)(cg + t) * 32] = r0[(int64_t)t * 32];
    }
  }
  if (live) {
    cnt_g[s] = cg;
    cnt_s[s] = cs;
  }
  int mg = cg, ms = cs, mneed = need;
  unsigned long long sg = (unsigned long long)kg, su = (unsigned long long)(kg + ks);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mg = max(mg, __shfl_xor_sync(kFull, mg, o));
    ms = max(ms, __shfl_xor_sync(kFull, ms, o));
    mneed = max(mneed, __shfl_xor_sync(kFull, mneed, o));
    sg += __shfl_xor_sync(kFull, sg, o);
    su += __shfl_xor_sync(kFull, su, o);
  }
  if (lane == 0) {
    wlen_g[w] = mg;
    wlen_s[w] = ms;
    atomicAdd(&hdr->gather_pairs, sg);
    atomicAdd(&hdr->union_pairs, su);
    atomicMax(&hdr->max_list, (unsigned long long)mneed);
    atomicAdd(&hdr->nbr_nodes, cnt_nodes);
    atomicAdd(&hdr->nbr_buckets, cnt_buckets);
  }
}

// ---------------------------------------------------------------------------
// neighbor sets as CSR in caller order (inspection / tests)
// ---------------------------------------------------------------------------
__global__ void k_csr_counts(const int32_t* __restrict__ perm, const int32_t* __restrict__ cg,
                             const int32_t* __restrict__ cs, int mode, int64_t n,
                             int64_t* __restrict__ rowcnt) {
  int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s < n) rowcnt[perm[s]] = cg[s] + (mode ? cs[s] : 0);
}

__global__ void k_csr_fill(const int32_t* __restrict__ perm, const int32_t* __restrict__ cg,
                           const int32_t* __restrict__ cs, int mode, int64_t cap_pp,
                           const uint32_t* __restrict__ ell, int64_t n,
                           const int64_t* __restrict__ row_ptr, int32_t* __restrict__ col,
                           int64_t cap) {
  int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const int64_t p = perm[s];
  const int64_t r0 = row_ptr[p];
  const int ng = cg[s], ns = mode ? cs[s] : 0;
  const int64_t base = (s >> 5) * cap_pp * 32 + (s & 31);
  for (int k = 0; k < ng + ns; ++k) {
    const uint32_t e = ell[base + (int64_t)k * 32];
    const int32_t j = perm[e & kIdxMask];
    // insertion into the sorted prefix of this row
    int64_t pos = r0 + k;
    if (pos >= cap) return;
    while (pos > r0 && col[pos - 1] > j) { col[pos] = col[pos - 1]; --pos; }
    col[pos] = j;
  }
}

// Work list for the union sweeps: within each run of kBalance consecutive
// sorted particles, the particles ordered by union-list length (longest
// first, ties by index).  A warp then takes 32 particles of similar length, so
// fewer of its lanes idle at the end of the walk; every particle still sums
// its own list in list order, so results are the same bit for bit.
constexpr int kBalance = 256;
__global__ void __launch_bounds__(kBalance)
    k_balance(const int32_t* __restrict__ cnt_g, const int32_t* __restrict__ cnt_s, int64_t n,
              int32_t* __restrict__ items_u, int32_t* __restrict__ cost,
              int32_t* __restrict__ seq_cost, DevHeader* hdr) {
  __shared__ int32_t lu[kBalance];
  const int64_t base = (int64_t)blockIdx.x * kBalance;
  const int t = threadIdx.x;
  const int64_t s = base + t;
  const int m = (int)(n - base < kBalance ? n - base : kBalance);
  const bool live = t < m;
  const int u = live ? cnt_g[s] + cnt_s[s] : -1;
  lu[t] = u;
  // cost of the item of 32 consecutive particles this warp covers (-1 when partial)
  {
    int um = u;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) um = max(um, __shfl_xor_sync(kFull, um, o));
    const int64_t q = s >> 5;
    if ((t & 31) == 0 && q * 32 < n) seq_cost[q] = (q * 32 + 32 <= n) ? um : -1;
  }
  if (blockIdx.x == 0 && t == 0) hdr->n_all = (int32_t)n;
  // bitonic sort of (length + 1, 255 - index) in decreasing order: longest
  // first, ties by index; the slots past the run's end sort last
  uint32_t* key = reinterpret_cast<uint32_t*>(lu);
  key[t] = ((uint32_t)(u + 1) << 8) | (uint32_t)(kBalance - 1 - t);
  __syncthreads();
#pragma unroll
  for (int k = 2; k <= kBalance; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      const int tx = t ^ j;
      if (tx > t) {
        const uint32_t a = key[t], b = key[tx];
        if ((a < b) == ((t & k) == 0)) {
          key[t] = b;
          key[tx] = a;
        }
      }
      __syncthreads();
    }
  }
  // slot r now holds the particle of rank r
  if (t >= m) return;
  const uint32_t kr = key[t];
  const int ur = (int)(kr >> 8) - 1;
  items_u[base + t] = (int32_t)(base + (kBalance - 1 - (int)(kr & 255u)));
  // the first (longest) particle of each 32-particle item gives the item's
  // cost; a partial item (the last one) gets -1
  if ((t & 31) == 0) {
    const int64_t q = (base + t) >> 5;
    cost[q] = (base + t + 32 <= n) ? ur : -1;
  }
}

// Longest items first.  A persistent sweep ends when its slowest warp finishes
// its last item, so passes with LPT take the balanced list's items (32
// particles each) in decreasing order of their longest union list: the last
// items are the shortest and the warps finish close together.  The order
// within equal costs does not matter (each particle still sums its own list),
// and a partial last item stays last.
constexpr int kLptBins = 1024;
constexpr int kLptThreads = 1024;
__global__ void __launch_bounds__(kLptThreads)
    k_item_sort(const int32_t* __restrict__ cost_bal, int32_t* __restrict__ order_bal,
                const int32_t* __restrict__ cost_seq, int32_t* __restrict__ order_seq,
                int64_t nitems) {
  // one block sorts the balanced items, the other the items of consecutive particles
  const int32_t* cost = blockIdx.x ? cost_seq : cost_bal;
  int32_t* order = blockIdx.x ? order_seq : order_bal;
  __shared__ int32_t cnt[kLptBins];
  for (int b = threadIdx.x; b < kLptBins; b += kLptThreads) cnt[b] = 0;
  __syncthreads();
  // bin 0 holds the most expensive items, bin kLptBins-1 the partial one
  auto bin = [](int32_t c) {
    const int32_t k = c < 0 ? kLptBins - 1 : (kLptBins - 2) - (c < kLptBins - 2 ? c : kLptBins - 2);
    return k;
  };
  for (int64_t q = threadIdx.x; q < nitems; q += kLptThreads) atomicAdd(&cnt[bin(cost[q])], 1);
  __syncthreads();
  // exclusive scan of the bin counts (one bin per thread)
  static_assert(kLptBins == kLptThreads, "one bin per thread");
  __shared__ int32_t wsum[kLptThreads / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int32_t v = cnt[threadIdx.x];
  int32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t t = __shfl_up_sync(kFull, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) wsum[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    const int32_t w0 = wsum[lane];
    int32_t winc = w0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t t = __shfl_up_sync(kFull, winc, o);
      if (lane >= o) winc += t;
    }
    wsum[lane] = winc - w0;
  }
  __syncthreads();
  cnt[threadIdx.x] = wsum[wid] + inc - v;
  __syncthreads();
  for (int64_t q = threadIdx.x; q < nitems; q += kLptThreads)
    order[atomicAdd(&cnt[bin(cost[q])], 1)] = (int32_t)q;
}

// ---------------------------------------------------------------------------
// host driver
// ---------------------------------------------------------------------------
template <class R>
crk_status cell_build_impl(Plan* plan, cudaStream_t st, char* ws, int64_t n, int32_t nb,
                           const int64_t* box_off, const double* box_L, const double* x,
                           const R* h) {
  const Layout& Ly = plan->ly;
  DevHeader* hdr = reinterpret_cast<DevHeader*>(ws + Ly.hdr);
  // a build starts a new session: clear the status word, counters and queues
  cudaMemsetAsync(hdr, 0, sizeof(DevHeader), st);
  double* wbox = reinterpret_cast<double*>(ws + Ly.box_L);
  BoxScale* scale = reinterpret_cast<BoxScale*>(ws + Ly.box_scale);
  unsigned int* hbox = reinterpret_cast<unsigned int*>(ws + Ly.hbox);
  int box_bits = 0;
  while ((1ll << box_bits) < nb) ++box_bits;
  // Morton resolution per axis: six bits finer than the mean spacing of the
  // largest possible box (n particles), at most 16.  Finer keys only order
  // particles that share a cell more finely; the lists do not depend on it.
  int bits = 6;
  while (bits < 16 && (double)(1ll << (3 * (bits - 6))) < (double)n) ++bits;
  {
    Phase ph(plan, st, "build.check", 1);
    k_check_boxes<<<(nb + 1 + 127) / 128, 128, 0, st>>>(box_off, box_L, nb, n, bits, wbox, scale,
                                                        hbox, hdr);
  }
  if (n == 0) return CRK_OK;
  const unsigned g256 = (unsigned)((n + 255) / 256);
  uint64_t* k0 = reinterpret_cast<uint64_t*>(ws + Ly.key0);
  uint64_t* k1 = reinterpret_cast<uint64_t*>(ws + Ly.key1);
  int32_t* v0 = reinterpret_cast<int32_t*>(ws + Ly.val0);
  int32_t* v1 = reinterpret_cast<int32_t*>(ws + Ly.val1);
  // 8-bit digits over the Morton bits [0, 3 bits) and the box bits [48, ...)
  int shifts[8], passes = 0;
  for (int b = 0; b < 3 * bits; b += 8) shifts[passes++] = b;
  for (int b = 48; b < 48 + box_bits; b += 8) shifts[passes++] = b;
  // The short sort while kShortTiles tiles (one a multiprocessor) of at most 4096
  // keys hold all keys: every block reads every tile's counts, and larger tiles
  // leave the chip idle (2.1 M particles in tiles of 16384: 0.314 ms against
  // 0.293 for the long sort).
  int tile_log2 = 10;
  while (tile_log2 < 12 && (n + (1ll << tile_log2) - 1) >> tile_log2 > kShortTiles) ++tile_log2;
  const int64_t short_tiles = (n + (1ll << tile_log2) - 1) >> tile_log2;
  const bool short_sort = short_tiles <= kShortTiles;
  uint32_t* hist = reinterpret_cast<uint32_t*>(ws + Ly.hist);
  const int ntiles = short_sort ? (int)short_tiles : (int)Ly.ntiles;
  Phase ph_sort(plan, st, "build.keys_sort",
                1 + passes * (short_sort ? 1 : 2 + scan_launches((int64_t)256 * Ly.ntiles)));
  if (short_sort) cudaMemsetAsync(hist, 0, sizeof(uint32_t) * 256 * (size_t)ntiles * passes, st);
  k_keys<R><<<g256, 256, 0, st>>>(x, h, box_off, wbox, scale, nb, n, bits, k0, v0, hbox,
                                  short_sort ? hist : nullptr, tile_log2, hdr);
  // radix sort over the used key bits
  for (int p = 0; p < passes; ++p) {
    if (short_sort) {
      uint32_t* cnt = hist + (size_t)p * ntiles * 256;
      k_short_sort<<<ntiles, kShortThreads, 0, st>>>(
          k0, v0, k1, v1, cnt, cnt + (size_t)ntiles * 256, n, shifts[p],
          p + 1 < passes ? shifts[p + 1] : -1, ntiles, tile_log2);
    } else {
      k_rsort_hist<<<ntiles, kSortThreads, 0, st>>>(k0, n, shifts[p], ntiles, hist);
      exclusive_scan<uint32_t>(hist, hist, (int64_t)256 * ntiles, ws + Ly.scan_tmp, nullptr, st);
      k_rsort_scatter<<<ntiles, kSortThreads, 0, st>>>(k0, v0, k1, v1, hist, n, shifts[p], ntiles);
    }
    std::swap(k0, k1);
    std::swap(v0, v1);
  }
  plan->sorted_keys_in_key0 = (k0 == reinterpret_cast<uint64_t*>(ws + Ly.key0));
  int32_t* perm = reinterpret_cast<int32_t*>(ws + Ly.perm);
  int32_t* boxid = reinterpret_cast<int32_t*>(ws + Ly.boxid);
  R* xs = reinterpret_cast<R*>(ws + Ly.xs);
  R* hs = reinterpret_cast<R*>(ws + Ly.hs);
  ph_sort.end();
  const int64_t nbk = Ly.nbk, ni = Ly.ni;
  // the segment tree lives in the region of the rate records, which hold nothing
  // between a build's start and the sweeps that write them
  SegTree seg{};
  seg.base = reinterpret_cast<float*>(ws + Ly.rec_c2);
  for (int64_t c = nbk, o = 0;; c = (c + 1) / 2) {
    seg.off[seg.levels] = o;
    seg.cnt[seg.levels++] = c;
    o += c;
    if (c <= 1) break;
  }
  int up = 0;
  for (int lev = kSegLeafLevels; lev + 1 < seg.levels; lev += kSegUpLevels) ++up;
  Phase ph_tree(plan, st, "build.tree", 1 + up + (ni > 0 ? 1 : 0));
  float4* p4 = reinterpret_cast<float4*>(ws + Ly.p4);
  float* nrec = reinterpret_cast<float*>(ws + Ly.nrec);
  uint64_t* bkey = reinterpret_cast<uint64_t*>(ws + Ly.bkey);
  k_gather_sorted<R><<<g256, 256, 0, st>>>(k0, v0, x, h, n, nbk, ni, perm, boxid, xs, hs, p4, bkey,
                                           nrec, seg);
  for (int lev = kSegLeafLevels; lev + 1 < seg.levels; lev += kSegUpLevels)
    k_seg_up<<<(unsigned)((seg.cnt[lev] + 1023) / 1024), 1024, 0, st>>>(seg, lev);
  if (ni > 0)
    k_lbvh<<<(unsigned)((ni + 127) / 128), 128, 0, st>>>(bkey, boxid, n, nbk, ni, seg, nrec);
  ph_tree.end();
  Phase ph_lists(plan, st, "build.lists",
                 lpt_worthwhile(Ly.nw, (int64_t)plan->num_sms * 64) ? 3 : 2);
  // neighbor lists (one pass; fixed column of cap_pp slots per particle)
  int32_t* cnt_g = reinterpret_cast<int32_t*>(ws + Ly.cnt_g);
  int32_t* cnt_s = reinterpret_cast<int32_t*>(ws + Ly.cnt_s);
  int32_t* wlen_g = reinterpret_cast<int32_t*>(ws + Ly.wlen_g);
  int32_t* wlen_s = reinterpret_cast<int32_t*>(ws + Ly.wlen_s);
  uint32_t* ell = reinterpret_cast<uint32_t*>(ws + Ly.ell);
  k_nbr<R><<<(unsigned)Ly.nw, 32, 0, st>>>(k0, hs, boxid, wbox, n, ni, nrec, p4, cnt_g, cnt_s,
                                           wlen_g, wlen_s, ell, Ly.cap_pp, hdr, x, perm,
                                           reinterpret_cast<const float*>(hbox));
  int32_t* cost = reinterpret_cast<int32_t*>(ws + Ly.item_cost);
  int32_t* seq_cost = reinterpret_cast<int32_t*>(ws + Ly.seq_cost);
  k_balance<<<(unsigned)((n + kBalance - 1) / kBalance), kBalance, 0, st>>>(
      cnt_g, cnt_s, n, reinterpret_cast<int32_t*>(ws + Ly.items_bu), cost, seq_cost, hdr);
  if (lpt_worthwhile(Ly.nw, (int64_t)plan->num_sms * 64)) {
    k_item_sort<<<2, kLptThreads, 0, st>>>(cost, reinterpret_cast<int32_t*>(ws + Ly.item_order),
                                           seq_cost, reinterpret_cast<int32_t*>(ws + Ly.seq_order),
                                           Ly.nw);
  }
  return cudaGetLastError() == cudaSuccess ? CRK_OK : CRK_ECUDA;
}

template crk_status cell_build_impl<float>(Plan*, cudaStream_t, char*, int64_t, int32_t,
                                           const int64_t*, const double*, const double*,
                                           const float*);
template crk_status cell_build_impl<double>(Plan*, cudaStream_t, char*, int64_t, int32_t,
                                            const int64_t*, const double*, const double*,
                                            const double*);

crk_status neighbors_csr_impl(Plan* plan, cudaStream_t st, char* ws, int32_t mode,
                              int64_t* row_ptr, int32_t* col, int64_t cap, int64_t* nnz) {
  const Layout& Ly = plan->ly;
  const int64_t n = Ly.n;
  const int32_t* perm = reinterpret_cast<const int32_t*>(ws + Ly.perm);
  const int32_t* cg = reinterpret_cast<const int32_t*>(ws + Ly.cnt_g);
  const int32_t* cs = reinterpret_cast<const int32_t*>(ws + Ly.cnt_s);
  const uint32_t* ell = reinterpret_cast<const uint32_t*>(ws + Ly.ell);
  const unsigned g = (unsigned)((n + 255) / 256);
  {
    DevHeader h;
    if (cudaMemcpyAsync(&h, ws + Ly.hdr, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return CRK_ECUDA;
    if ((int64_t)h.max_list > Ly.cap_pp) return CRK_ENOMEM;
  }
  if (n > 0) k_csr_counts<<<g, 256, 0, st>>>(perm, cg, cs, mode, n, row_ptr);
  exclusive_scan<int64_t>(row_ptr, row_ptr, n, ws + Ly.scan_tmp, row_ptr + n, st);
  if (cudaMemcpyAsync(nnz, row_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return CRK_ECUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return CRK_ECUDA;
  if (*nnz > cap) return CRK_ENOMEM;
  if (n > 0) k_csr_fill<<<g, 256, 0, st>>>(perm, cg, cs, mode, Ly.cap_pp, ell, n, row_ptr, col, cap);
  if (cudaStreamSynchronize(st) != cudaSuccess) return CRK_ECUDA;
  return CRK_OK;
}

}  // namespace crk

// octgrav_build.cu -- the octree build of Sec. 2.1 on the GPU: Morton keys,
// a stable LSD radix sort, the level-by-level split of key ranges, the
// bottom-up cell properties, the groups and the work items, written straight
// into the device arrays the walk kernel reads.
//
// The result equals the host build (octgrav_host.cpp) byte for byte: the same
// FP64 operations in the same order (this file is compiled with -fmad=false,
// the host with -ffp-contract=off), the same stable sort, and the same array
// layout (cells of each system in breadth-first order, systems one after the
// other). Every kernel reads its sizes from device memory, so the whole build
// is enqueued without a host round trip; the host reads one result block at
// the end (cell capacity overflow there means: enlarge and build again).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "octgrav_grid.h"
#include "octgrav_internal.h"

namespace og {
namespace {

constexpr int MAXD = 21;          // depth limit (Morton keys of 3 x 21 bits)
constexpr int NLEV = MAXD + 1;    // levels 0..21
constexpr int TB = 256;           // threads per block
constexpr int IPT = 16;           // elements per thread in the chunked kernels
constexpr int TILE = TB * IPT;    // particles per chunk (sort)
constexpr int SUB = 8;            // blocks per chunk in the key pass
constexpr int BSUB = 2;           // blocks per chunk in the box pass
constexpr int LT = 512;           // threads of the level kernel (16 warps) ...
constexpr int LBMAX = 1024;       // ... and the most blocks it may have
constexpr int LROUNDS = 16;       // most rounds in which its warps take a level ...
constexpr int64_t LROUNDS_N = 4000000;  // ... of a tree of at least so many particles
constexpr int NT = 128;           // threads of the node kernel
constexpr unsigned FULL = 0xffffffffu;
constexpr int LBINS = 32;  // leaf size bins of the moment pass (32 = "32 or more")
constexpr int SORT_CHUNKS4 = 8, SORT_CHUNKS2 = 64;  // most chunks that k_sort takes with four and two blocks each
constexpr int IBMAX = 608;  // blocks of the group and item kernel
constexpr int IBINS = 256; // work-item size bins of the default processing order (item_max <= 256)

struct SysGeo {  // root cube of a system: lower corner, side, 2^21 * fl(1 / side)
  double lo[3], side, rscale;
};

struct Chunk {  // TILE particles (or fewer) of one system
  int sys, first, count, cs;  // system, first particle, count, first chunk of the system
  int nbs, pad0, pad1, pad2;  // chunks of the system
};

// misc[] slots (int), zeroed before a build: counts, status bits, arrivals at
// the grid barriers of the sort, the level and the node kernel, nodes per level
enum { M_NGROUPS = 0, M_NITEMS, M_NLEAVES, M_MAXGROUP, M_STATUS, M_BAR_SORT, M_BAR_LEVELS, M_BAR_NODES, M_BAR_ITEMS, M_NODES };
constexpr int MISC = M_NODES + NLEV;

// Scratch layout (byte offsets into one allocation).
struct Layout {
  size_t keyA, keyB, valA, valB, cnt, dtot, part, sg, xs, ms, chunks, offs, chunk0;
  size_t ckey, cpar, cpf, cpc, csys, cfc, cnc, spl, lpre, nlist, bsum, lvl, misc;
  size_t sstart, send, lofs, ni, lorder, lhist, ihist, gmark, gcell, ioff, isum;
  size_t total;
};

inline size_t al(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

Layout layout(int64_t n, int n_sys, int64_t n_chunks, int64_t cap) {
  Layout L{};
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o += al(bytes);
    return at;
  };
  L.keyA = take(8 * n);
  L.keyB = take(8 * n);
  L.valA = take(4 * n);
  L.valB = take(4 * n);
  L.cnt = take(4 * 256 * std::max<int64_t>(n_chunks, 2 * SORT_CHUNKS2));
  L.dtot = take(4 * 256 * static_cast<size_t>(n_sys));
  L.part = take(8 * 6 * BSUB * n_chunks);
  L.sg = take(sizeof(SysGeo) * n_sys);
  L.xs = take(24 * n);
  L.ms = take(8 * n);
  L.chunks = take(sizeof(Chunk) * n_chunks);
  L.offs = take(8 * (n_sys + 1));
  L.chunk0 = take(4 * (n_sys + 1));
  L.ckey = take(8 * cap);
  L.cpar = take(4 * cap);
  L.cpf = take(4 * cap);
  L.cpc = take(4 * cap);
  L.csys = take(4 * cap);
  L.cfc = take(4 * cap);
  L.cnc = take(4 * cap);
  L.spl = take(4 * 9 * std::min<int64_t>(n, cap));
  L.lpre = take(4 * std::min<int64_t>(n, cap));
  L.nlist = take(4 * cap);
  L.bsum = take(4 * LBMAX * LROUNDS);
  L.lvl = take(4 * (NLEV + 2));
  L.misc = take(4 * MISC);
  L.sstart = take(4 * static_cast<size_t>(n_sys) * NLEV);
  L.send = take(4 * static_cast<size_t>(n_sys) * NLEV);
  L.lofs = take(4 * static_cast<size_t>(n_sys) * NLEV);
  L.ni = take(n_sys > 1 ? 4 * cap : 0);
  L.lorder = take(4 * cap);
  L.lhist = take(4 * 2 * LBINS);
  L.ihist = take(4 * 2 * IBINS);
  L.gmark = take(4 * n);
  L.gcell = take(4 * n);
  L.ioff = take(4 * n);
  L.isum = take(4 * 2 * IBMAX);
  L.total = o;
  return L;
}


template <class T>
T* at(void* base, size_t off) {
  return reinterpret_cast<T*>(static_cast<char*>(base) + off);
}

__device__ __forceinline__ uint64_t spread21(uint64_t v) {
  v &= 0x1fffffull;
  v = (v | v << 32) & 0x1f00000000ffffull;
  v = (v | v << 16) & 0x1f0000ff0000ffull;
  v = (v | v << 8) & 0x100f00f00f00f00full;
  v = (v | v << 4) & 0x10c30c30c30c30c3ull;
  v = (v | v << 2) & 0x1249249249249249ull;
  return v;
}

// Integer key with the order of `<` on non-NaN doubles (the two zeros equal),
// so that min / max run on the integer pipe (FP64 is slow on this part).
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return b >= 0 ? b : (b == (-0x7fffffffffffffffLL - 1) ? 0 : b ^ 0x7fffffffffffffffLL);
}
// min / max with the tie rule of std::min / std::max (the first argument
// wins ties, so signed zeros come out as on the host)
__device__ __forceinline__ double lesser(double a, double b) { return order_key(b) < order_key(a) ? b : a; }
__device__ __forceinline__ double greater(double a, double b) { return order_key(a) < order_key(b) ? b : a; }

// Exclusive block-wide scan of one int per thread (TB threads); returns the
// exclusive prefix and writes the block total to *total.
__device__ int block_scan_excl(int v, int* total) {
  __shared__ int warp_tot[TB / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(FULL, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) warp_tot[w] = x;
  __syncthreads();
  if (w == 0) {
    int t = lane < TB / 32 ? warp_tot[lane] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(FULL, t, d);
      if (lane >= d) t += y;
    }
    if (lane < TB / 32) warp_tot[lane] = t;  // inclusive
  }
  __syncthreads();
  const int before = w ? warp_tot[w - 1] : 0;
  *total = warp_tot[TB / 32 - 1];
  __syncthreads();  // warp_tot is reused by the next call
  return before + x - v;
}

// ---------------------------------------------------------------- keys and sort

// Bounding box per half of a chunk; flags non-finite coordinates or masses and
// negative masses.
__global__ void __launch_bounds__(TB) k_bbox(const double* __restrict__ pos, const double* __restrict__ mass,
                                             const Chunk* __restrict__ ch, double* __restrict__ part,
                                             int* __restrict__ misc) {
  const Chunk c = ch[blockIdx.x / BSUB];
  double mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
  bool bad = false;
  const int k0 = static_cast<int>(blockIdx.x % BSUB) * (TILE / BSUB), k1 = min(c.count, k0 + TILE / BSUB);
  for (int k = k0 + threadIdx.x; k < k1; k += TB) {
    const int64_t i = c.first + k;
    for (int d = 0; d < 3; ++d) {
      const double v = pos[3 * i + d];
      bad |= !isfinite(v);
      mn[d] = lesser(mn[d], v);
      mx[d] = greater(mx[d], v);
    }
    const double m = mass[i];
    bad |= !isfinite(m) || m < 0;
  }
  __shared__ double red[6][TB / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int d = 0; d < 3; ++d) {
    for (int s = 16; s; s >>= 1) {
      mn[d] = lesser(mn[d], __shfl_xor_sync(FULL, mn[d], s));
      mx[d] = greater(mx[d], __shfl_xor_sync(FULL, mx[d], s));
    }
    if (lane == 0) {
      red[d][w] = mn[d];
      red[3 + d][w] = mx[d];
    }
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&misc[M_STATUS], GPU_BUILD_BADINPUT);
  if (threadIdx.x < 6) {
    double v = red[threadIdx.x][0];
    for (int k = 1; k < TB / 32; ++k) v = threadIdx.x < 3 ? lesser(v, red[threadIdx.x][k]) : greater(v, red[threadIdx.x][k]);
    part[6 * blockIdx.x + threadIdx.x] = v;
  }
}

// Root cube per system (the host build's arithmetic, operation for operation).
// One block per system.
__global__ void __launch_bounds__(TB) k_root(const double* __restrict__ part, const int* __restrict__ chunk0,
                                             SysGeo* __restrict__ sg) {
  const int s = blockIdx.x;
  double mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int b = BSUB * chunk0[s] + threadIdx.x; b < BSUB * chunk0[s + 1]; b += TB)
    for (int d = 0; d < 3; ++d) {
      mn[d] = lesser(mn[d], part[6 * b + d]);
      mx[d] = greater(mx[d], part[6 * b + 3 + d]);
    }
  __shared__ double red[6][TB / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int d = 0; d < 3; ++d) {
    for (int o = 16; o; o >>= 1) {
      mn[d] = lesser(mn[d], __shfl_xor_sync(FULL, mn[d], o));
      mx[d] = greater(mx[d], __shfl_xor_sync(FULL, mx[d], o));
    }
    if (lane == 0) {
      red[d][w] = mn[d];
      red[3 + d][w] = mx[d];
    }
  }
  __syncthreads();
  if (threadIdx.x) return;
  for (int k = 1; k < TB / 32; ++k)
    for (int d = 0; d < 3; ++d) {
      red[d][0] = lesser(red[d][0], red[d][k]);
      red[3 + d][0] = greater(red[3 + d][0], red[3 + d][k]);
    }
  for (int d = 0; d < 3; ++d) {
    mn[d] = red[d][0];
    mx[d] = red[3 + d][0];
  }
  double ext = mx[0] - mn[0];
  if (mx[1] - mn[1] > ext) ext = mx[1] - mn[1];
  if (mx[2] - mn[2] > ext) ext = mx[2] - mn[2];
  if (!(ext > 0)) ext = 1.0;
  const double side = ext * (1.0 + 1.0 / 1048576.0);
  for (int d = 0; d < 3; ++d) sg[s].lo[d] = (mn[d] + mx[d]) * 0.5 - side * 0.5;
  sg[s].side = side;
  sg[s].rscale = (1.0 / side) * 2097152.0;
}

__global__ void __launch_bounds__(TB) k_morton(const double* __restrict__ pos, const Chunk* __restrict__ ch,
                                               const SysGeo* __restrict__ sg, uint64_t* __restrict__ key,
                                               uint32_t* __restrict__ val) {
  const Chunk c = ch[blockIdx.x / SUB];
  const SysGeo g = sg[c.sys];
  const double* lo = g.lo;
  const double side = g.side;
  const double scale = 2097152.0;  // 2^21
  const uint64_t qmax = (1ull << MAXD) - 1;
  const int k0 = static_cast<int>(blockIdx.x % SUB) * (TILE / SUB), k1 = min(c.count, k0 + TILE / SUB);
  for (int k = k0 + threadIdx.x; k < k1; k += TB) {
    const int64_t i = c.first + k;
    uint64_t q[3];
    for (int d = 0; d < 3; ++d) {
      // The quantised coordinate is floor(fl(fl(x - lo) / side) * 2^21) =
      // floor(fl(fl(x - lo) * 2^21 / side)). a = fl(x - lo) * g.rscale is
      // within 4 ulp (< 2^-29 for a <= 2^21) of fl(fl(x - lo) * 2^21 / side).
      // Adding 1.5 * 2^22 rounds a to a multiple of 2^-30 (half a unit more)
      // and leaves it in the low mantissa bits, so whenever its fraction is 4
      // units or more from an integer the floors agree; the rare remaining
      // cases take the division. Three FP64 operations per coordinate, the
      // rest on the integer pipe: FP64 issue bounds this pass (72 us at 1M
      // particles with floor() of both ends of the interval, 22 us now).
      const double dx = pos[3 * i + d] - lo[d];
      const double a = dx * g.rscale;
      const double magic = 6291456.0;
      const long long u = __double_as_longlong(a + magic) - __double_as_longlong(magic);
      const int frac = static_cast<int>(u) & ((1 << 30) - 1);
      long long v = u >> 30;
      if (frac < 4 || frac > (1 << 30) - 5) v = static_cast<long long>(floor((dx / side) * scale));
      q[d] = v <= 0 ? 0 : (v >= static_cast<long long>(qmax) ? qmax : static_cast<uint64_t>(v));
    }
    key[i] = spread21(q[0]) | (spread21(q[1]) << 1) | (spread21(q[2]) << 2);
    val[i] = static_cast<uint32_t>(i);
  }
}

// Digit histogram of one chunk, stored at (system, digit, chunk within the
// system): the scan over a (system, digit) row is then contiguous.
__global__ void __launch_bounds__(TB) k_upsweep(const uint64_t* __restrict__ key, const Chunk* __restrict__ ch,
                                                int shift, int* __restrict__ cnt) {
  __shared__ int h[256];
  const Chunk c = ch[blockIdx.x];
  h[threadIdx.x] = 0;
  __syncthreads();
  for (int k = threadIdx.x; k < c.count; k += TB)
    atomicAdd(&h[(key[c.first + k] >> shift) & 255], 1);
  __syncthreads();
  cnt[256 * c.cs + threadIdx.x * c.nbs + (blockIdx.x - c.cs)] = h[threadIdx.x];
}

// Per (system, digit): exclusive scan over the system's chunks in place, and
// the digit's total. One warp per (system, digit).
__global__ void __launch_bounds__(TB) k_scan_digits(int* __restrict__ cnt, const int* __restrict__ chunk0, int n_sys,
                                                    int* __restrict__ dtot) {
  const int seg = static_cast<int>((blockIdx.x * static_cast<int64_t>(TB) + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (seg >= 256 * n_sys) return;
  const int s = seg >> 8, d = seg & 255;
  const int cs = chunk0[s], nbs = chunk0[s + 1] - cs;
  int* a = cnt + 256 * static_cast<int64_t>(cs) + static_cast<int64_t>(d) * nbs;
  int run = 0;
  for (int base = 0; base < nbs; base += 32) {
    const int v = base + lane < nbs ? a[base + lane] : 0;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, x, o);
      if (lane >= o) x += y;
    }
    if (base + lane < nbs) a[base + lane] = run + x - v;
    run += __shfl_sync(FULL, x, 31);
  }
  if (lane == 0) dtot[seg] = run;
}

// Stable ranks of one chunk's keys by the digit at `shift`: warp w ranks its
// 32 K elements round by round (32 at a time, in order); afterwards wc[w][d] is
// the number of elements of digit d in the warps before, and an element's place
// among its chunk's digit is wc[w][d] + rk. Returns the chunk's count of digit
// threadIdx.x.
template <int K>
__device__ __forceinline__ int chunk_ranks(const uint64_t* kin, const uint32_t* vin, const Chunk& c, int shift,
                                           int (*wc)[257], uint64_t* kk, uint32_t* vv, int* rk) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < K; ++r) {
    const int e = w * (32 * K) + r * 32 + lane;
    const bool ok = e < c.count;
    kk[r] = ok ? __ldcg(kin + c.first + e) : 0ull;
    vv[r] = ok ? __ldcg(vin + c.first + e) : 0u;
  }
#pragma unroll
  for (int r = 0; r < K; ++r) {
    const int e = w * (32 * K) + r * 32 + lane;
    const int d = e < c.count ? static_cast<int>((kk[r] >> shift) & 255) : 256;
    const unsigned peers = __match_any_sync(FULL, d);
    const int before = wc[w][d];
    rk[r] = before + __popc(peers & lt);
    __syncwarp();
    if (lane == __ffs(peers) - 1) wc[w][d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  int run = 0;  // warp offsets per digit
  for (int q = 0; q < TB / 32; ++q) {
    const int t = wc[q][threadIdx.x];
    wc[q][threadIdx.x] = run;
    run += t;
  }
  __syncthreads();
  return run;
}

// Stable scatter of one chunk by the digit at `shift`; the chunk's offsets come
// from the scan.
__global__ void __launch_bounds__(TB) k_downsweep(const uint64_t* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                  uint64_t* __restrict__ kout, uint32_t* __restrict__ vout,
                                                  const Chunk* __restrict__ ch, int shift,
                                                  const int* __restrict__ cnt, const int* __restrict__ dtot) {
  __shared__ int wc[TB / 32][257];  // per-warp digit counters (+ one for empty slots)
  __shared__ int goff[256];
  const Chunk c = ch[blockIdx.x];
  for (int k = threadIdx.x; k < (TB / 32) * 257; k += TB) (&wc[0][0])[k] = 0;
  {  // destination of this chunk's first element of each digit
    int unused;
    const int dbase = block_scan_excl(dtot[256 * c.sys + threadIdx.x], &unused);
    goff[threadIdx.x] = ch[c.cs].first + dbase + cnt[256 * c.cs + threadIdx.x * c.nbs + (blockIdx.x - c.cs)];
  }
  __syncthreads();
  uint64_t kk[IPT];
  uint32_t vv[IPT];
  int rk[IPT];
  chunk_ranks<IPT>(kin, vin, c, shift, wc, kk, vv, rk);
#pragma unroll
  for (int r = 0; r < IPT; ++r) {
    const int e = (threadIdx.x >> 5) * (32 * IPT) + r * 32 + (threadIdx.x & 31);
    if (e < c.count) {
      const int d = static_cast<int>((kk[r] >> shift) & 255);
      const int dst = goff[d] + wc[threadIdx.x >> 5][d] + rk[r];
      kout[dst] = kk[r];
      vout[dst] = vv[r];
    }
  }
}

// All eight passes in one cooperative launch, W blocks per chunk: ranks, the
// blocks' digit counts, a grid barrier, offsets (every block adds the counts of
// its system's blocks itself, a thread per digit), scatter, a second barrier.
// The same order as the passes by three launches each, whose gaps and short
// grids made up most of the time of a small sort: from the keys to the gather
// 157 us at 5000 particles, 48 us so. The rest is latency: a warp ranks its 16 /
// W rounds one after the other, and the sums grow with the blocks. Times of W =
// 1 / 2 / 4 / 8 (us): 5000 particles 83 / 79 / 48 / 54, 16,384 87 / 62 / 50 / 69,
// 32,768 85 / 67 / 57 / 97, 65,536 87 / 67 / 71 / 146, 262,144 100 / 98 / 176
// (159 by three launches a pass). Hence four blocks a chunk up to 8 chunks, two
// up to 64.
template <int W>
__global__ void __launch_bounds__(TB) k_sort(uint64_t* keyA, uint32_t* valA, uint64_t* keyB, uint32_t* valB,
                                             const Chunk* __restrict__ ch, int* cnt, int* misc) {
  __shared__ int wc[TB / 32][257];
  __shared__ int goff[256];
  constexpr int K = IPT / W;
  Chunk c = ch[blockIdx.x / W];
  c.first += static_cast<int>(blockIdx.x % W) * (K * TB);
  c.count = min(max(c.count - static_cast<int>(blockIdx.x % W) * (K * TB), 0), K * TB);
  const int first = ch[c.cs].first, grid = gridDim.x, mine = blockIdx.x;
  int bars = 0;
  for (int pass = 0; pass < 8; ++pass) {
    const int shift = 8 * pass;
    const bool even = (pass & 1) == 0;
    for (int k = threadIdx.x; k < (TB / 32) * 257; k += TB) (&wc[0][0])[k] = 0;
    __syncthreads();
    uint64_t kk[K];
    uint32_t vv[K];
    int rk[K];
    cnt[256 * mine + threadIdx.x] =
        chunk_ranks<K>(even ? keyA : keyB, even ? valA : valB, c, shift, wc, kk, vv, rk);
    if (!grid_barrier(&misc[M_BAR_SORT], ++bars * grid, &misc[M_STATUS], GPU_BUILD_STUCK)) return;
    int before = 0, total = 0;
#pragma unroll 8
    for (int j = W * c.cs; j < W * (c.cs + c.nbs); ++j) {
      const int v = __ldcg(&cnt[256 * j + threadIdx.x]);
      total += v;
      before += j < mine ? v : 0;
    }
    int unused;
    goff[threadIdx.x] = first + block_scan_excl(total, &unused) + before;
    __syncthreads();
    uint64_t* kout = even ? keyB : keyA;
    uint32_t* vout = even ? valB : valA;
#pragma unroll
    for (int r = 0; r < K; ++r) {
      const int e = (threadIdx.x >> 5) * (32 * K) + r * 32 + (threadIdx.x & 31);
      if (e < c.count) {
        const int d = static_cast<int>((kk[r] >> shift) & 255);
        const int dst = goff[d] + wc[threadIdx.x >> 5][d] + rk[r];
        kout[dst] = kk[r];
        vout[dst] = vv[r];
      }
    }
    if (pass < 7 && !grid_barrier(&misc[M_BAR_SORT], ++bars * grid, &misc[M_STATUS], GPU_BUILD_STUCK)) return;
  }
}

// Particles in tree order: FP64 copies for the moments, hi/lo FP32 records
// for the walk kernel, and the permutation; a build's group marks are cleared
// on the way.
__global__ void k_gather(const uint32_t* __restrict__ val, const double* __restrict__ pos,
                         const double* __restrict__ mass, int64_t n, double* __restrict__ xs,
                         double* __restrict__ ms, float4* __restrict__ parts, int* __restrict__ perm,
                         int* __restrict__ gmark) {
  for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < n;
       t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    if (gmark) gmark[t] = 0;
    const int64_t i = val[t];
    const double x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2], m = mass[i];
    xs[3 * t] = x;
    xs[3 * t + 1] = y;
    xs[3 * t + 2] = z;
    ms[t] = m;
    const float hx = static_cast<float>(x), hy = static_cast<float>(y), hz = static_cast<float>(z);
    parts[2 * t] = make_float4(hx, hy, hz, static_cast<float>(m));
    parts[2 * t + 1] = make_float4(static_cast<float>(x - static_cast<double>(hx)),
                                   static_cast<float>(y - static_cast<double>(hy)),
                                   static_cast<float>(z - static_cast<double>(hz)), 0.f);
    perm[t] = static_cast<int>(i);
  }
}

// ---------------------------------------------------------------- levels

struct Cells {
  uint64_t* key;
  int *par, *pf, *pc, *sys, *fc, *nc;
};

__global__ void k_roots(int n_sys, const int64_t* __restrict__ offs, Cells C, int* __restrict__ lvl,
                        int* __restrict__ lhist) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < n_sys) {
    C.key[s] = 1;
    C.par[s] = -1;
    C.pf[s] = static_cast<int>(offs[s]);
    C.pc[s] = static_cast<int>(offs[s + 1] - offs[s]);
    C.sys[s] = s;
    C.fc[s] = -1;
    C.nc[s] = 0;
  }
  if (s <= NLEV + 1) lvl[s] = s == 0 ? 0 : n_sys;
  if (s < 2 * LBINS) lhist[s] = 0;
}

// Split points of a cell holding particles [f, f + cnt): sp[o] = the first
// position whose child octant at depth D is >= o, sp[0] = f, sp[8] = f + cnt
// (octants ascend inside a cell). One warp; every lane returns the same sp.
// A cell of at most 128 particles has all its keys loaded at once, four a lane,
// and the particles of the octants below o are counted.
__device__ __forceinline__ void load_keys(const uint64_t* __restrict__ code, int f, int cnt, int lane, uint64_t* v) {
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = lane + 32 * j < cnt ? code[f + lane + 32 * j] : 0;
}
__device__ __forceinline__ void small_split(const uint64_t* v, int f, int cnt, int D, int lane, int* sp) {
  const int bit = 3 * (MAXD - D);
  sp[0] = f;
  sp[8] = f + cnt;
#pragma unroll
  for (int o = 1; o < 8; ++o) sp[o] = f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (32 * j >= cnt) break;
    const int oc = lane + 32 * j < cnt ? static_cast<int>(v[j] >> bit) & 7 : 8;
#pragma unroll
    for (int o = 1; o < 8; ++o) sp[o] += __popc(__ballot_sync(FULL, oc < o));
  }
}

// The same for a larger cell. The seven boundaries are searched together: a round
// probes 32 positions a power of two apart of each one's interval, seven
// independent loads per lane, so a cell of a million particles takes four rounds
// of load latency and one of at most 1024 two. (One boundary after the other took
// seven times as many rounds; probes at 33rds of the intervals spent 10 us of a
// level on their 64-bit divisions.)
__device__ void warp_split(const uint64_t* __restrict__ code, int f, int cnt, int D, int lane, int* sp) {
  const int bit = 3 * (MAXD - D);
  sp[0] = f;
  sp[8] = f + cnt;
  // invariant: boundary o lies in [a[o], b[o]], and b[o] is the end or a known hit
  int a[8], b[8];
#pragma unroll
  for (int o = 1; o < 8; ++o) {
    a[o] = f;
    b[o] = f + cnt;
  }
  int sh = max(0, 32 - __clz(cnt - 1) - 5);  // 32 probes 2^sh apart cover the interval
  for (;;) {
    const int off = lane << sh;
    int oc[8];
#pragma unroll
    for (int o = 1; o < 8; ++o)
      oc[o] = off < b[o] - a[o] ? static_cast<int>(code[a[o] + off] >> bit) & 7 : 8;
#pragma unroll
    for (int o = 1; o < 8; ++o) {
      const unsigned m = __ballot_sync(FULL, oc[o] >= o);  // a probe beyond the end is a hit
      const int k = m ? __ffs(m) - 1 : 32;
      const int hi = k == 32 ? b[o] : min(b[o], a[o] + (k << sh));
      a[o] = k == 0 ? a[o] : min(b[o], a[o] + ((k - 1) << sh) + 1);
      b[o] = hi;
    }
    if (sh == 0) break;
    sh = max(0, sh - 5);
  }
#pragma unroll
  for (int o = 1; o < 8; ++o) sp[o] = b[o];
}

// After a barrier that ran out: a tree without cells, which the rest of the
// build passes through without touching anything (the host reports the status).
__device__ void no_cells(int* lvl) {
  if (threadIdx.x <= NLEV + 1) lvl[threadIdx.x] = 0;
}

// Split points of the cells [c0, c1) of the level from lb on that hold more than
// n_leaf particles, a warp per cell; the keys of the next cell are loaded while one is
// worked on. Returns the children of all of them.
__device__ __forceinline__ int split_cells(int c0, int c1, int lb, int L, const uint64_t* __restrict__ code, const Cells& C,
                                           int n_leaf, int* spl, int* lpre, int* nlist, int* misc) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int mine = 0;
  for (int base = c0; base < c1; base += 32) {
    const int c = base + lane;
    const int cnt = c < c1 ? C.pc[c] : 0;
    const int f = c < c1 ? C.pf[c] : 0;
    unsigned todo = __ballot_sync(FULL, cnt > n_leaf);
    const unsigned nodes = todo;
    int nch = 0;
    int kf = 0, kc = 0;  // the cell that is split next: its first particle and their number ...
    uint64_t v[4];       // ... and its keys, where there are at most 128
    const auto next = [&]() {
      const int k = todo ? __ffs(todo) - 1 : 0;
      kf = __shfl_sync(FULL, f, k);
      kc = todo ? __shfl_sync(FULL, cnt, k) : 0;
      if (kc <= 128) load_keys(code, kf, kc, lane, v);
    };
    next();
    while (todo) {
      const int k = __ffs(todo) - 1, f0 = kf, n0 = kc;
      todo &= todo - 1;
      uint64_t u[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) u[j] = v[j];
      next();
      int sp[9];
      if (n0 <= 128) small_split(u, f0, n0, L + 1, lane, sp);
      else warp_split(code, f0, n0, L + 1, lane, sp);
      int n = 0, own = sp[0];
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        n += sp[o + 1] > sp[o];
        own = lane == o + 1 ? sp[o + 1] : own;
      }
      if (lane < 9) spl[9 * static_cast<int64_t>(base + k - lb) + lane] = own;
      if (lane == k) nch = n;
    }
    int x = nch;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(FULL, x, d);
      if (lane >= d) x += y;
    }
    int at = 0;
    if (lane == 0 && nodes) at = atomicAdd(&misc[M_NODES + L], __popc(nodes));
    at = __shfl_sync(FULL, at, 0);
    if (nch) {
      C.nc[c] = nch;
      lpre[c - lb] = mine + x - nch;
      nlist[lb + at + __popc(nodes & lt)] = c;
    }
    mine += __shfl_sync(FULL, x, 31);
  }
  return mine;
}

// Their children, numbered from `first` on: of the cells that were split four at a
// time, lane (k, o) writing child o of the k-th.
__device__ __forceinline__ void emit_cells(int c0, int c1, int lb, int first, const Cells& C, const int* spl, const int* lpre) {
  const int lane = threadIdx.x & 31, o = lane & 7, sub = lane >> 3;
  for (int base = c0; base < c1; base += 32) {
    unsigned nodes = __ballot_sync(FULL, base + lane < c1 && C.nc[base + lane] > 0);
    while (nodes) {
      int c = -1;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (nodes && sub == k) c = base + __ffs(nodes) - 1;
        nodes &= nodes - 1;
      }
      int f = 0, e = 0;
      if (c >= 0) {
        f = spl[9 * static_cast<int64_t>(c - lb) + o];
        e = spl[9 * static_cast<int64_t>(c - lb) + o + 1];
      }
      const unsigned m = __ballot_sync(FULL, e > f) >> (8 * sub) & 255u;
      if (e > f) {
        const int k0 = first + lpre[c - lb], k = k0 + __popc(m & ((1u << o) - 1u));
        if ((m & ((1u << o) - 1u)) == 0) C.fc[c] = k0;
        C.key[k] = (C.key[c] << 3) | static_cast<uint64_t>(o);
        C.par[k] = c;
        C.pf[k] = f;
        C.pc[k] = e - f;
        C.sys[k] = C.sys[c];
        C.fc[k] = -1;
        C.nc[k] = 0;
      }
    }
  }
}

// All levels of the tree in one cooperative launch. Per level: every block
// takes contiguous ranges of the level's cells and finds the split points of
// those that hold more than n_leaf particles (a warp per cell); after a
// barrier every block adds the blocks' children counts up to its own, which
// places its children in the host's breadth-first order, and writes them;
// after a second barrier they are the next level. The loop ends with the first
// level without children. The cells that were split are also listed per level
// (nlist, M_NODES) for the moment pass.
//
// Latency bounds it: a level is a few dependent rounds of loads and two
// barriers (5 us; the levels with tens of thousands of cells up to 20 us, where
// a warp's cells are all split). As three launches per level for 21 levels (4096
// blocks each, most of them empty) the levels took 412 us at 1M particles and
// 229 us at 5000 (sum of the launches); 301 us and 79 us now.
//
// The cells that are split lie together, so with one range a block a large level
// waits for the blocks in the dense part. From LROUNDS_N particles on a warp takes
// up to 16 ranges of at least 32 cells, spread over the level: 4.2M particles 627 ->
// 590 us, 16M 2100 -> 1210 us, where the three launches a level took 636 and 1460;
// at 3M 503 us with one range, 540 with several.
template <int ROUNDS>
__global__ void __launch_bounds__(LT, 2) k_levels(const uint64_t* __restrict__ code, Cells C, int n_leaf, int* lvl,
                                                  int* spl, int* lpre, int* nlist, int* bsum, int cap, int* misc) {
  constexpr int W = LT / 32;
  static_assert(W >= ROUNDS, "a warp per round");
  __shared__ int wsum[ROUNDS * W];
  __shared__ int before[ROUNDS], all[ROUNDS];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, grid = gridDim.x;
  int lb = lvl[0], le = lvl[1], bars = 0;
  if (__ldcg(&misc[M_STATUS]) & GPU_BUILD_STUCK) {  // the sort did not finish
    no_cells(lvl);
    return;
  }
  for (int L = 0; L < MAXD; ++L) {
    const int nl = le - lb;
    // a round gives every warp `per` consecutive cells, a block's warps one after the other
    const int rounds = ROUNDS == 1 || nl <= 32 * grid * W ? 1 : min(ROUNDS, (nl + grid * W * 32 - 1) / (grid * W * 32));
    const int per = (nl + grid * W * rounds - 1) / (grid * W * rounds);
    const auto range = [&](int r) {  // this warp's cells of round r
      const int c0 = lb + min(((r * grid + static_cast<int>(blockIdx.x)) * W + w) * per, nl);
      return make_int2(c0, min(le, c0 + per));
    };
    const int2 first_range = range(0);
    for (int r = 0; r < rounds; ++r) {
      const int2 cells = ROUNDS == 1 ? first_range : range(r);
      const int c0 = cells.x, c1 = cells.y;
      const int mine = split_cells(c0, c1, lb, L, code, C, n_leaf, spl, lpre, nlist, misc);
      if (lane == 0) wsum[r * W + w] = mine;
    }
    __syncthreads();
    if (w < rounds) {  // children before each warp, and the block's, in round w
      const int v = lane < W ? wsum[w * W + lane] : 0;
      int x = v;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(FULL, x, d);
        if (lane >= d) x += y;
      }
      if (lane < W) wsum[w * W + lane] = x - v;
      if (lane == 31) bsum[w * grid + blockIdx.x] = x;
      if (lane == 0) before[w] = all[w] = 0;
    }
    if (!grid_barrier(&misc[M_BAR_LEVELS], ++bars * grid, &misc[M_STATUS], GPU_BUILD_STUCK)) {
      no_cells(lvl);
      return;
    }
    {  // per round: children of the blocks before this one, and of all
      const int warps = rounds == 1 ? W : W / rounds, r = rounds == 1 ? 0 : w / warps;
      if (r < rounds) {
        int bef = 0, sum = 0;
        for (int b = 32 * (w - r * warps) + lane; b < grid; b += 32 * warps) {
          const int v = __ldcg(&bsum[r * grid + b]);
          sum += v;
          bef += b < static_cast<int>(blockIdx.x) ? v : 0;
        }
#pragma unroll
        for (int d = 16; d; d >>= 1) {
          bef += __shfl_xor_sync(FULL, bef, d);
          sum += __shfl_xor_sync(FULL, sum, d);
        }
        if (lane == 0) {
          atomicAdd(&before[r], bef);
          atomicAdd(&all[r], sum);
        }
      }
    }
    __syncthreads();
    int total = 0;
    for (int r = 0; r < rounds; ++r) total += all[r];
    const int64_t next = static_cast<int64_t>(le) + total;
    if (total == 0 || next > cap) {  // the same in every block
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        for (int k = L + 2; k <= NLEV; ++k) lvl[k] = le;
        if (next > cap) {
          atomicOr(&misc[M_STATUS], GPU_BUILD_OVERFLOW);
          misc[M_NODES + L] = 0;
        }
      }
      if (next > cap)  // the unsplit cells are no nodes
        for (int r = 0; r < rounds; ++r) {
          const int2 cells = ROUNDS == 1 ? first_range : range(r);
          for (int c = cells.x + lane; c < cells.y; c += 32) C.nc[c] = 0;
        }
      return;
    }
    int done = le;  // the rounds before
    for (int r = 0; r < rounds; done += all[r], ++r) {
      const int2 cells = ROUNDS == 1 ? first_range : range(r);
      const int c0 = cells.x, c1 = cells.y;
      const int first = done + before[r] + wsum[r * W + w];
      emit_cells(c0, c1, lb, first, C, spl, lpre);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) lvl[L + 2] = static_cast<int>(next);
    if (!grid_barrier(&misc[M_BAR_LEVELS], ++bars * grid, &misc[M_STATUS], GPU_BUILD_STUCK)) {
      no_cells(lvl);
      return;
    }
    lb = le;
    le = static_cast<int>(next);
  }
}

// Level of cell c: the last L with lvl[L] <= c.
__device__ __forceinline__ int level_of(const int* lvl, int c) {
  int L = 0;
  while (L + 1 < NLEV && lvl[L + 1] <= c) ++L;
  return L;
}

// ---------------------------------------------------------------- system-major order (batches)

__global__ void k_sys_bounds(const int* __restrict__ lvl, const int* __restrict__ csys, int* __restrict__ sstart,
                             int* __restrict__ send) {
  const int nc = lvl[NLEV];
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
    const int L = level_of(lvl, c), s = csys[c];
    if (c == lvl[L] || csys[c - 1] != s) sstart[s * NLEV + L] = c;
    if (c == lvl[L + 1] - 1 || csys[c + 1] != s) send[s * NLEV + L] = c + 1;
  }
}

// Per system: its first cell in the final order and the final position of
// its first cell of every level.
__global__ void __launch_bounds__(1024) k_sys_offsets(int n_sys, const int* __restrict__ sstart,
                                                      const int* __restrict__ send, int* __restrict__ lofs,
                                                      int64_t* __restrict__ cell_off) {
  __shared__ int ws[32];
  const int per = (n_sys + 1023) / 1024;
  const int lo = min(n_sys, static_cast<int>(threadIdx.x) * per), hi = min(n_sys, lo + per);
  int sum = 0;
  for (int s = lo; s < hi; ++s)
    for (int L = 0; L < NLEV; ++L) sum += send[s * NLEV + L] - sstart[s * NLEV + L];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = sum;
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(FULL, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  if (w == 0) {
    int t = ws[lane];
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(FULL, t, d);
      if (lane >= d) t += y;
    }
    ws[lane] = t;
  }
  __syncthreads();
  int run = (w ? ws[w - 1] : 0) + x - sum;
  for (int s = lo; s < hi; ++s) {
    cell_off[s] = run;
    for (int L = 0; L < NLEV; ++L) {
      lofs[s * NLEV + L] = run;
      run += send[s * NLEV + L] - sstart[s * NLEV + L];
    }
  }
  if (threadIdx.x == 1023) cell_off[n_sys] = ws[31];
}

__global__ void k_new_index(const int* __restrict__ lvl, const int* __restrict__ csys, const int* __restrict__ sstart,
                            const int* __restrict__ lofs, int* __restrict__ ni) {
  const int nc = lvl[NLEV];
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
    const int L = level_of(lvl, c), k = csys[c] * NLEV + L;
    ni[c] = lofs[k] + (c - sstart[k]);
  }
}

// ---------------------------------------------------------------- cell properties

struct Props {  // final-order FP64 arrays and records
  double *bmin, *bmax, *cube, *M, *com, *S;
  uint64_t* key;
  float4* geo;
  int2* link;
  float4* mp;
  int *pcount, *cfirst;
};

__device__ __forceinline__ int final_index(const int* ni, int c) { return ni ? ni[c] : c; }

// Tight box, boundary cube, mass, centre of mass and second moments of a
// cell: sums over its members in the host build's operation order.
struct Moments {
  double bn[3], bx[3];  // tight box
  double M, sx, sy, sz; // mass, mass-weighted positions
  double cu[4], cm[3];  // boundary cube (centre, half side), centre of mass
  double s6[6];         // second moments about cm

  __device__ __forceinline__ void clear() {
    for (int d = 0; d < 3; ++d) {
      bn[d] = INFINITY;
      bx[d] = -INFINITY;
    }
    M = sx = sy = sz = 0;
    for (int k = 0; k < 6; ++k) s6[k] = 0;
  }
  __device__ __forceinline__ void add_mass(double m, double x, double y, double z) {
    M += m;
    sx = fma(m, x, sx);
    sy = fma(m, y, sy);
    sz = fma(m, z, sz);
  }
  __device__ __forceinline__ void centre() {
    for (int d = 0; d < 3; ++d) cu[d] = (bn[d] + bx[d]) * 0.5;
    double e = bx[0] - bn[0];
    if (bx[1] - bn[1] > e) e = bx[1] - bn[1];
    if (bx[2] - bn[2] > e) e = bx[2] - bn[2];
    cu[3] = 0.5 * e;
    if (M > 0) {
      cm[0] = sx / M;
      cm[1] = sy / M;
      cm[2] = sz / M;
    } else {
      cm[0] = cu[0];
      cm[1] = cu[1];
      cm[2] = cu[2];
    }
  }
  __device__ __forceinline__ void add_outer(double wt, double y0, double y1, double y2) {
    const double w0 = wt * y0, w1 = wt * y1, w2 = wt * y2;
    s6[0] = fma(w0, y0, s6[0]);
    s6[1] = fma(w1, y1, s6[1]);
    s6[2] = fma(w2, y2, s6[2]);
    s6[3] = fma(w0, y1, s6[3]);
    s6[4] = fma(w0, y2, s6[4]);
    s6[5] = fma(w1, y2, s6[5]);
  }
  // FP64 arrays and the walk kernel's records of cell j (final order).
  __device__ __forceinline__ void store(int j, uint64_t key, int f, int cnt, int2 link, const Props& P) const {
    for (int d = 0; d < 3; ++d) {
      P.bmin[3 * j + d] = bn[d];
      P.bmax[3 * j + d] = bx[d];
      P.com[3 * j + d] = cm[d];
    }
    for (int d = 0; d < 4; ++d) P.cube[4 * j + d] = cu[d];
    for (int k = 0; k < 6; ++k) P.S[6 * j + k] = s6[k];
    P.M[j] = M;
    P.key[j] = key;
    P.geo[j] = make_float4(static_cast<float>(cu[0]), static_cast<float>(cu[1]), static_cast<float>(cu[2]),
                           static_cast<float>(cu[3]));
    P.link[j] = link;
    float chi[3], clo[3];
    for (int d = 0; d < 3; ++d) {
      chi[d] = static_cast<float>(cm[d]);
      clo[d] = static_cast<float>(cm[d] - static_cast<double>(chi[d]));
    }
    const double tr = s6[0] + s6[1] + s6[2];
    P.mp[4 * j] = make_float4(chi[0], chi[1], chi[2], static_cast<float>(M));
    P.mp[4 * j + 1] = make_float4(clo[0], clo[1], clo[2], static_cast<float>(cnt));
    P.mp[4 * j + 2] = make_float4(static_cast<float>(3.0 * s6[0]), static_cast<float>(3.0 * s6[1]),
                                  static_cast<float>(3.0 * s6[2]), static_cast<float>(3.0 * s6[3]));
    P.mp[4 * j + 3] = make_float4(static_cast<float>(3.0 * s6[4]), static_cast<float>(3.0 * s6[5]),
                                  static_cast<float>(1.5 * tr), static_cast<float>(0.5 * tr));
    P.pcount[j] = cnt;
    P.cfirst[j] = f;
  }
};

// A leaf, from its particles.
__device__ __forceinline__ void leaf_props(int c, Cells C, const int* __restrict__ ni, const double* __restrict__ xs,
                                           const double* __restrict__ ms, const Props& P) {
  Moments A;
  A.clear();
  const int f = C.pf[c], cnt = C.pc[c];
  for (int t = f; t < f + cnt; ++t) {
    const double* xp = &xs[3 * static_cast<int64_t>(t)];
    for (int d = 0; d < 3; ++d) {
      A.bn[d] = lesser(A.bn[d], xp[d]);
      A.bx[d] = greater(A.bx[d], xp[d]);
    }
    A.add_mass(ms[t], xp[0], xp[1], xp[2]);
  }
  A.centre();
  for (int t = f; t < f + cnt; ++t) {
    const double* xp = &xs[3 * static_cast<int64_t>(t)];
    A.add_outer(ms[t], xp[0] - A.cm[0], xp[1] - A.cm[1], xp[2] - A.cm[2]);
  }
  A.store(final_index(ni, c), C.key[c], f, cnt, make_int2(f, -cnt), P);
}

// A node, from its children (contiguous in both orders) with the
// parallel-axis shift. The children's records are loaded ahead of the sums,
// four at a time, so that a node waits for a few rounds of loads and not for
// one per child and pass.
__device__ __forceinline__ void node_props(int c, Cells C, const int* __restrict__ ni, const Props& P) {
  Moments A;
  A.clear();
  const int nch = C.nc[c], jc = final_index(ni, C.fc[c]);
  double m[8], x[8], y[8], z[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int j = jc + min(q, nch - 1);
    m[q] = P.M[j];
    x[q] = P.com[3 * j];
    y[q] = P.com[3 * j + 1];
    z[q] = P.com[3 * j + 2];
  }
#pragma unroll
  for (int h = 0; h < 8; h += 4) {
    double v[4][6];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = jc + min(h + q, nch - 1);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        v[q][d] = P.bmin[3 * j + d];
        v[q][3 + d] = P.bmax[3 * j + d];
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (h + q < nch) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          A.bn[d] = lesser(A.bn[d], v[q][d]);
          A.bx[d] = greater(A.bx[d], v[q][3 + d]);
        }
      }
  }
#pragma unroll
  for (int q = 0; q < 8; ++q)
    if (q < nch) A.add_mass(m[q], x[q], y[q], z[q]);
  A.centre();
#pragma unroll
  for (int h = 0; h < 8; h += 4) {
    double v[4][6];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = jc + min(h + q, nch - 1);
#pragma unroll
      for (int k = 0; k < 6; ++k) v[q][k] = P.S[6 * j + k];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (h + q < nch) {
#pragma unroll
        for (int k = 0; k < 6; ++k) A.s6[k] += v[q][k];
        A.add_outer(m[h + q], x[h + q] - A.cm[0], y[h + q] - A.cm[1], z[h + q] - A.cm[2]);
      }
  }
  A.store(final_index(ni, c), C.key[c], C.pf[c], C.pc[c], make_int2(jc, nch), P);
}

// Leaves (of every level) bucketed by particle count, largest first, so that
// the lanes of a warp loop over equally many particles: histogram, then
// scatter of the cell indices into lorder.
__device__ __forceinline__ int leaf_bin(int cnt) { return LBINS - min(cnt, LBINS); }  // 32+ -> bin 0

__global__ void __launch_bounds__(TB) k_leaf_hist(Cells C, const int* __restrict__ lvl, int* __restrict__ lhist,
                                                  int* __restrict__ misc, int64_t* __restrict__ cell_off) {
  __shared__ int h[LBINS];
  if (threadIdx.x < LBINS) h[threadIdx.x] = 0;
  __syncthreads();
  const int nc = lvl[NLEV];
  if (cell_off && blockIdx.x == 0 && threadIdx.x < 2) cell_off[threadIdx.x] = threadIdx.x ? nc : 0;
  int leaves = 0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x)
    if (C.nc[c] == 0) {
      atomicAdd(&h[leaf_bin(C.pc[c])], 1);
      ++leaves;
    }
  for (int s = 16; s; s >>= 1) leaves += __shfl_xor_sync(FULL, leaves, s);
  if ((threadIdx.x & 31) == 0 && leaves) atomicAdd(&misc[M_NLEAVES], leaves);
  __syncthreads();
  if (threadIdx.x < LBINS && h[threadIdx.x]) atomicAdd(&lhist[threadIdx.x], h[threadIdx.x]);
}

__global__ void __launch_bounds__(TB) k_leaf_scatter(Cells C, const int* __restrict__ lvl,
                                                     const int* __restrict__ lhist, int* __restrict__ lfill,
                                                     int* __restrict__ lorder) {
  __shared__ int base[LBINS], h[LBINS];
  if (threadIdx.x < 32) {
    const int v = lhist[threadIdx.x];
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, x, o);
      if (threadIdx.x >= o) x += y;
    }
    base[threadIdx.x] = x - v;
  }
  const int nc = lvl[NLEV];
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t c0 = static_cast<int64_t>(blockIdx.x) * blockDim.x; c0 < nc; c0 += stride) {
    if (threadIdx.x < LBINS) h[threadIdx.x] = 0;
    __syncthreads();
    const int c = static_cast<int>(c0) + threadIdx.x;
    const bool leaf = c < nc && C.nc[c] == 0;
    const int b = leaf ? leaf_bin(C.pc[c]) : 0;
    const int r = leaf ? atomicAdd(&h[b], 1) : 0;  // rank within the block's bin
    __syncthreads();
    if (threadIdx.x < LBINS && h[threadIdx.x]) h[threadIdx.x] = atomicAdd(&lfill[threadIdx.x], h[threadIdx.x]);
    __syncthreads();
    if (leaf) lorder[base[b] + h[b] + r] = c;
    __syncthreads();
  }
}

// Bound by the FP64 instructions of a warp (see k_nodes), a lane per leaf. Four
// warps a block, one per scheduler of an SM: with eight, trees of up to a few
// hundred thousand particles left most SMs idle. 27 -> 22 us at 5000 particles,
// 31 -> 22 at 65,536, 39 -> 31 at 262,144; 82 at 1M either way.
constexpr int LT_LEAF = 128;

__global__ void __launch_bounds__(LT_LEAF) k_leaf_props(Cells C, const int* __restrict__ lorder,
                                                   const int* __restrict__ misc, const int* __restrict__ ni,
                                                   const double* __restrict__ xs, const double* __restrict__ ms,
                                                   Props P) {
  const int nl = misc[M_NLEAVES];
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nl; k += gridDim.x * blockDim.x)
    leaf_props(lorder[k], C, ni, xs, ms, P);
}

// The double of another lane.
__device__ __forceinline__ double from_lane(double v, int src) {
  return __shfl_sync(FULL, v, src);
}

// node_props by eight lanes (l = 0..7, base = the first one's lane): every
// FP64 instruction works on up to six components at once, each component's
// operations in the same order. `live` lanes hold a node, the others only
// take part in the shuffles.
__device__ __forceinline__ void node_props8(int c, bool live, int l, int base, Cells C, const int* __restrict__ ni,
                                            const Props& P) {
  const int nch = live ? C.nc[c] : 0, jc = live ? final_index(ni, C.fc[c]) : 0;
  const int last = max(nch - 1, 0);
  // lanes 0..2 hold component l of vectors, lanes 0..5 component l of boxes and second moments
  const int d = l < 3 ? l : (l < 6 ? l - 3 : 0), k6 = l < 6 ? l : 5;
  double m[8], v[8], bb[8], ss[8];
  if (live) {
    const double* box = l < 3 ? P.bmin : P.bmax;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int j = jc + min(q, last);
      m[q] = P.M[j];
      v[q] = P.com[3 * j + d];
      bb[q] = box[3 * j + d];
      ss[q] = P.S[6 * j + k6];
    }
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) m[q] = v[q] = bb[q] = ss[q] = 0;
  }
  double b = l < 3 ? INFINITY : -INFINITY;  // lanes 0..2: lower, 3..5: upper corner
  double M = 0, s = 0;                      // lane 3 sums the mass: fma(m, 1, M) rounds as M + m
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    if (q < nch) {
      b = l < 3 ? lesser(b, bb[q]) : greater(b, bb[q]);
      s = fma(m[q], l == 3 ? 1.0 : v[q], s);
    }
  }
  M = from_lane(s, base + 3);
  const double up = from_lane(b, base + min(l + 3, 7));
  // centre of the cube and longest side (order-key comparisons: sides are >= 0)
  const double cu = (b + up) * 0.5;
  const double side = up - b;
  double e = from_lane(side, base);
  const double e1 = from_lane(side, base + 1), e2 = from_lane(side, base + 2);
  if (order_key(e1) > order_key(e)) e = e1;
  if (order_key(e2) > order_key(e)) e = e2;
  const double half = 0.5 * e;
  const double cm = M > 0 ? s / M : cu;  // lanes 0..2
  // second moments: lane k takes w_a y_b of its pair (a, b)
  const int pa = k6 < 3 ? k6 : (k6 == 5 ? 1 : 0), pb = k6 < 3 ? k6 : (k6 == 3 ? 1 : 2);
  double s6 = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const double y = v[q] - cm, w = m[q] * y;
    const double wa = from_lane(w, base + pa), yb = from_lane(y, base + pb);
    if (q < nch) s6 = fma(wa, yb, s6 + ss[q]);
  }
  const double s0 = from_lane(s6, base), s1 = from_lane(s6, base + 1), s2 = from_lane(s6, base + 2);
  const double tr = s0 + s1 + s2;
  const float ch = static_cast<float>(cm), cl = static_cast<float>(cm - static_cast<double>(ch));
  const float cuf = static_cast<float>(cu), t3 = static_cast<float>(3.0 * s6), Mf = static_cast<float>(M);
  // a lane's float of the walk's records: (com_hi, M), (com_lo, count), 3S, 3 tr / 2, tr / 2; (cube centre, half side)
  const float trf = static_cast<float>((l & 1 ? 0.5 : 1.5) * tr), hf = static_cast<float>(half);
  if (!live) return;
  const int j = final_index(ni, c), cnt = C.pc[c];
  float* mp = reinterpret_cast<float*>(P.mp + 4 * static_cast<int64_t>(j));
  float* geo = reinterpret_cast<float*>(P.geo + j);
  if (l < 3) {
    P.bmin[3 * j + l] = b;
    P.bmax[3 * j + l] = up;
    P.com[3 * j + l] = cm;
    P.cube[4 * j + l] = cu;
    mp[l] = ch;
    mp[4 + l] = cl;
    geo[l] = cuf;
  }
  if (l < 6) {
    P.S[6 * j + l] = s6;
    mp[8 + l] = t3;
  } else {
    mp[8 + l] = trf;  // lane 6: 3 tr / 2, lane 7: tr / 2
  }
  if (l == 3) {
    P.M[j] = M;
    mp[3] = Mf;
    mp[7] = static_cast<float>(cnt);
  }
  if (l == 4) {
    P.cube[4 * j + 3] = half;
    geo[3] = hf;
    P.key[j] = C.key[c];
  }
  if (l == 5) {
    P.link[j] = make_int2(jc, nch);
    P.pcount[j] = cnt;
    P.cfirst[j] = C.pf[c];
  }
}

// Nodes of all levels, deepest first, in one cooperative launch with a
// barrier between levels; the nodes come from the level kernel's lists.
//
// Each of an SM's four schedulers issues an FP64 warp instruction every 82
// clocks, however many lanes it has, so the number of FP64 instructions a
// warp goes through is what counts: about 300 for 32 nodes, a lane each, or 80
// for 4 nodes, eight lanes each. With NODE_WIDE nodes (four rounds of eight-lane warps
// over the 608 schedulers) both take the same time; levels below it, nearly
// all of them up to a few million particles, take eight lanes. As a launch per
// level over all of its cells (one in eight a node), a lane per cell, the
// nodes took 372 us at 1M particles and 170 us at 5000; 120 us and 58 us now.
constexpr int NODE_WIDE = 4 * 4 * 608;

__global__ void __launch_bounds__(NT) k_nodes(Cells C, int* lvl, const int* __restrict__ nlist,
                                              const int* __restrict__ ni, Props P, int* misc) {
  const int grid = gridDim.x, lane = threadIdx.x & 31;
  const int warp = (threadIdx.x >> 5) * grid + static_cast<int>(blockIdx.x);  // consecutive warps on different SMs
  const int warps = grid * (NT / 32);
  int bars = 0;
  if (__ldcg(&misc[M_STATUS]) & GPU_BUILD_STUCK) return;
  for (int L = MAXD - 1; L >= 0; --L) {
    const int nn = __ldcg(&misc[M_NODES + L]);
    if (nn == 0) continue;
    const int* nodes = nlist + lvl[L];
    if (nn > NODE_WIDE) {
      for (int k = 32 * warp + lane; k < nn; k += 32 * warps) node_props(nodes[k], C, ni, P);
    } else {
      for (int k0 = 4 * warp; k0 < nn; k0 += 4 * warps) {  // warp-uniform
        const int k = k0 + (lane >> 3);
        const bool live = k < nn;
        node_props8(live ? nodes[k] : 0, live, lane & 7, lane & 24, C, ni, P);
      }
    }
    if (L > 0 && !grid_barrier(&misc[M_BAR_NODES], ++bars * grid, &misc[M_STATUS], GPU_BUILD_STUCK)) {
      no_cells(lvl);
      return;
    }
  }
}

// ---------------------------------------------------------------- groups and items

struct Items {
  const int64_t* cell_off;
  int item_max, split;
  int4* items;
  float4* ibox;
  uint64_t* item_key;
  int* group_item;
};

// Work items of group g in cell c (final order) of system s, from item k on, cut
// by next_item_size (at most item_max particles each), all with the group's
// box, centre (hi/lo) and particle range. `item(k, size)` sees each of them.
template <class F>
__device__ __forceinline__ void group_items(int g, int c, int s, int k, const Props& P, const Items& I, F item) {
  const int pf = P.cfirst[c], cnt = P.pcount[c];
  float chi[3], clo[3];
  for (int d = 0; d < 3; ++d) {
    const double C0 = P.cube[4 * c + d];
    chi[d] = static_cast<float>(C0);
    clo[d] = static_cast<float>(C0 - static_cast<double>(chi[d]));
  }
  const float4 b0 = make_float4(static_cast<float>(P.bmin[3 * c]), static_cast<float>(P.bmin[3 * c + 1]),
                                static_cast<float>(P.bmin[3 * c + 2]), chi[0]);
  const float4 b1 = make_float4(static_cast<float>(P.bmax[3 * c]), static_cast<float>(P.bmax[3 * c + 1]),
                                static_cast<float>(P.bmax[3 * c + 2]), chi[1]);
  const float4 b2 = make_float4(clo[0], clo[1], clo[2], chi[2]);
  const float4 b3 = make_float4(__int_as_float(pf), __int_as_float(cnt), 0.f, 0.f);
  const int root = static_cast<int>(I.cell_off[s]);
  I.group_item[g] = k;
  for (int off = 0, sz; off < cnt; off += sz, ++k) {
    sz = next_item_size(cnt - off, I.item_max, I.split != 0);
    I.items[k] = make_int4(root, pf + off, sz, s);
    I.ibox[4 * static_cast<int64_t>(k)] = b0;
    I.ibox[4 * static_cast<int64_t>(k) + 1] = b1;
    I.ibox[4 * static_cast<int64_t>(k) + 2] = b2;
    I.ibox[4 * static_cast<int64_t>(k) + 3] = b3;
    I.item_key[k] = P.key[c];
    item(sz);
  }
}

// The items again from the same groups (a refit: boxes and centres change).
__global__ void k_items(const int* __restrict__ n_groups, const int* __restrict__ group_cell,
                        const int* __restrict__ group_sys, const int* __restrict__ ioff, Props P, Items I) {
  const int ng = *n_groups;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += gridDim.x * blockDim.x)
    group_items(g, group_cell[g], group_sys[g], ioff[g], P, I, [](int) {});
}

__device__ void finish(const int* lvl, const int* misc, int64_t* res) {
  int depth = 0;
  for (int L = 0; L < NLEV; ++L)
    if (__ldcg(&lvl[L + 1]) > __ldcg(&lvl[L])) depth = L;
  res[GB_NCELLS] = __ldcg(&lvl[NLEV]);
  res[GB_NGROUPS] = __ldcg(&misc[M_NGROUPS]);
  res[GB_NITEMS] = __ldcg(&misc[M_NITEMS]);
  res[GB_DEPTH] = depth;
  res[GB_NLEAVES] = __ldcg(&misc[M_NLEAVES]);
  res[GB_MAXGROUP] = __ldcg(&misc[M_MAXGROUP]);
  res[GB_STATUS] = __ldcg(&misc[M_STATUS]);
}

__global__ void k_finish(const int* __restrict__ lvl, const int* __restrict__ misc, int64_t* __restrict__ res) {
  finish(lvl, misc, res);
}

// Groups (ordered by first particle), their work items, the items' default
// processing order and the build's result, in one cooperative launch:
//   marks: a group is a cell that is a leaf or holds <= n_group particles while
//     its parent does not (the property is inherited by descendants, so "the
//     first such cell from the root" is exactly this), marked at its first
//     particle;
//   sums: every block counts the groups and items of its range of particles;
//   group numbers and first items from the sums of the blocks before;
//   items, a thread per group;
//   order: most particles first, a counting sort on the item size (the order
//     inside a size is arbitrary and does not affect any result).
// Latency-bound: each phase is a few dependent loads. 17 us at 5000 particles
// and 45 us at 1M, with four barriers of about 2 us; as twelve launches, with
// two scans of three launches each, the build's end took 56 and 97 us more.
struct Groups {
  int n, n_group;
  int mark;  // 0: the marks of the build are there
  const int* ni;
  int *gmark, *gcell;
  int *group_cell, *group_sys;
  int *ioff, *isum, *ihist;
  int* order;
  int64_t* result;
};

__global__ void __launch_bounds__(TB) k_groups(Cells C, Props P, Items I, Groups G, int* lvl, int* misc) {
  static_assert(IBINS == TB, "a thread per size bin");
  __shared__ int hist[IBINS], base[IBINS];
  const int grid = gridDim.x, first = blockIdx.x * TB + threadIdx.x, stride = grid * TB;
  int bars = 0;
  // all blocks see the same bit of an earlier kernel; a barrier that runs out stops this one
  const auto sync = [&]() {
    if (grid_barrier(&misc[M_BAR_ITEMS], ++bars * grid, &misc[M_STATUS], GPU_BUILD_STUCK)) return true;
    no_cells(lvl);
    if (threadIdx.x == 0) finish(lvl, misc, G.result);
    return false;
  };
  if (__ldcg(&misc[M_STATUS]) & GPU_BUILD_STUCK) {
    if (threadIdx.x == 0) finish(lvl, misc, G.result);
    return;
  }
  if (blockIdx.x == 0)
    for (int k = threadIdx.x; k < 2 * IBINS; k += TB) G.ihist[k] = 0;
  if (G.mark) {
    const int nc = lvl[NLEV];
    for (int c = first; c < nc; c += stride) {
      const bool elig = C.nc[c] == 0 || C.pc[c] <= G.n_group;
      const int p = C.par[c];
      const bool pelig = p >= 0 && C.pc[p] <= G.n_group;  // a parent is never a leaf
      if (elig && !pelig) {
        G.gmark[C.pf[c]] = 1;
        G.gcell[C.pf[c]] = c;
      }
    }
  }
  if (!sync()) return;

  const int64_t per = (static_cast<int64_t>(G.n) + stride - 1) / stride * TB;
  const int64_t lo = blockIdx.x * per, hi = min(static_cast<int64_t>(G.n), lo + per);
  const auto marked = [&](int64_t t, int* c) {
    if (t >= hi || !__ldcg(&G.gmark[t])) return false;
    *c = __ldcg(&G.gcell[t]);
    return true;
  };
  {
    int ng = 0, nk = 0, mg = 0, c, tot;
    for (int64_t t = lo + threadIdx.x; t < hi; t += TB)
      if (marked(t, &c)) {
        const int pc = C.pc[c];
        ++ng;
        nk += item_count(pc, I.item_max, I.split != 0);
        mg = max(mg, pc);
      }
    block_scan_excl(ng, &tot);
    if (threadIdx.x == 0) G.isum[2 * blockIdx.x] = tot;
    block_scan_excl(nk, &tot);
    if (threadIdx.x == 0) G.isum[2 * blockIdx.x + 1] = tot;
    for (int s = 16; s; s >>= 1) mg = max(mg, __shfl_xor_sync(FULL, mg, s));
    if ((threadIdx.x & 31) == 0 && mg) atomicMax(&misc[M_MAXGROUP], mg);
  }
  if (!sync()) return;

  int ng = 0, nk = 0;  // of all blocks
  {
    int bg = 0, bk = 0;
    for (int j = threadIdx.x; j < grid; j += TB) {
      const int2 v = __ldcg(reinterpret_cast<const int2*>(G.isum) + j);
      ng += v.x;
      nk += v.y;
      if (j < static_cast<int>(blockIdx.x)) {
        bg += v.x;
        bk += v.y;
      }
    }
    block_scan_excl(ng, &ng);
    block_scan_excl(nk, &nk);
    block_scan_excl(bg, &bg);
    block_scan_excl(bk, &bk);
    for (int64_t t0 = lo; t0 < hi; t0 += TB) {
      int c = 0, tot;
      const bool m = marked(t0 + threadIdx.x, &c);
      const int g = bg + block_scan_excl(m ? 1 : 0, &tot);
      bg += tot;
      const int k = bk + block_scan_excl(m ? item_count(C.pc[c], I.item_max, I.split != 0) : 0, &tot);
      bk += tot;
      if (m) {
        G.group_cell[g] = final_index(G.ni, c);
        G.group_sys[g] = C.sys[c];
        G.ioff[g] = k;
      }
    }
  }
  if (!sync()) return;

  hist[threadIdx.x] = 0;
  __syncthreads();
  for (int g = first; g < ng; g += stride)
    group_items(g, __ldcg(&G.group_cell[g]), __ldcg(&G.group_sys[g]), __ldcg(&G.ioff[g]), P, I,
                [&](int sz) { atomicAdd(&hist[IBINS - min(sz, IBINS)], 1); });
  __syncthreads();
  if (hist[threadIdx.x]) atomicAdd(&G.ihist[threadIdx.x], hist[threadIdx.x]);
  if (!sync()) return;

  int tot;
  base[threadIdx.x] = block_scan_excl(__ldcg(&G.ihist[threadIdx.x]), &tot);
  int* fill = G.ihist + IBINS;
  for (int64_t k0 = static_cast<int64_t>(blockIdx.x) * TB; k0 < nk; k0 += stride) {
    hist[threadIdx.x] = 0;
    __syncthreads();
    const int k = static_cast<int>(k0) + threadIdx.x;
    const bool live = k < nk;
    const int b = live ? IBINS - min(__ldcg(&I.items[k].z), IBINS) : 0;
    const int r = live ? atomicAdd(&hist[b], 1) : 0;
    __syncthreads();
    if (hist[threadIdx.x]) hist[threadIdx.x] = atomicAdd(&fill[threadIdx.x], hist[threadIdx.x]);
    __syncthreads();
    if (live) G.order[base[b] + hist[b] + r] = k;
    __syncthreads();
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    misc[M_NGROUPS] = ng;
    misc[M_NITEMS] = nk;
    finish(lvl, misc, G.result);
  }
}

// Before a refit: the counts of the build stay.
__global__ void k_clear_status(int* __restrict__ misc) {
  misc[M_STATUS] = 0;
  misc[M_BAR_NODES] = 0;
}

__global__ void k_unpermute(const float4* __restrict__ out, const int* __restrict__ perm, int64_t n,
                            double* __restrict__ acc, double* __restrict__ pot) {
  for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < n;
       t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const float4 a = out[t];
    const int64_t i = perm[t];
    acc[3 * i] = a.x;
    acc[3 * i + 1] = a.y;
    acc[3 * i + 2] = a.z;
    if (pot) pot[i] = a.w;
  }
}

int grid_for(int64_t n, int per_block) {
  const int64_t b = (n + per_block - 1) / per_block;
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16)));
}


// The node kernel: a warp per 4 nodes of a level (a level holds at most n /
// (n_leaf + 1) nodes) and at most one block per SM: its four warps have a
// scheduler each, and fewer blocks make cheaper barriers.
cudaError_t enqueue_nodes(const GpuBuild& a, const Layout& Lo, Cells C, const int* ni, Props P, cudaStream_t st) {
  const int64_t blocks = std::max<int64_t>(1, (a.n / (a.n_leaf + 1) + 15) / 16);
  const int most = static_cast<int>(std::min<int64_t>(blocks, 152));
  return launch_cooperative(k_nodes, resident_blocks(k_nodes, NT, most), NT, 0, st, C,
                            at<int>(a.scratch, Lo.lvl),
                            static_cast<const int*>(at<int>(a.scratch, Lo.nlist)), ni, P, at<int>(a.scratch, Lo.misc));
}

Items item_args(const GpuBuild& a) {
  return {a.cell_off, a.item_max, a.item_split, a.items, a.ibox, a.item_key, a.group_item};
}

// Groups and items; with mark = false of the groups that a build has marked.
cudaError_t enqueue_groups(const GpuBuild& a, const Layout& Lo, bool mark, cudaStream_t st) {
  void* S = a.scratch;
  Cells C{at<uint64_t>(S, Lo.ckey), at<int>(S, Lo.cpar), at<int>(S, Lo.cpf), at<int>(S, Lo.cpc),
          at<int>(S, Lo.csys),      at<int>(S, Lo.cfc),  at<int>(S, Lo.cnc)};
  Props P{a.bmin, a.bmax, a.cube, a.M, a.com, a.S, a.key, a.geo, a.link, a.mp, a.pcount, a.cfirst};
  const Groups G{static_cast<int>(a.n), a.n_group, mark, a.n_sys > 1 ? at<int>(S, Lo.ni) : nullptr,
                 at<int>(S, Lo.gmark), at<int>(S, Lo.gcell), a.group_cell, a.group_sys, at<int>(S, Lo.ioff),
                 at<int>(S, Lo.isum), at<int>(S, Lo.ihist), a.order, a.result};
  const int most = static_cast<int>(std::min<int64_t>((a.n + TB - 1) / TB, IBMAX));
  return launch_cooperative(k_groups, resident_blocks(k_groups, TB, most), TB, 0, st, C, P, item_args(a), G,
                            at<int>(S, Lo.lvl), at<int>(S, Lo.misc));
}

std::vector<Chunk> make_chunks(const int64_t* offsets, int n_sys, std::vector<int>& chunk0) {
  std::vector<Chunk> ch;
  chunk0.assign(n_sys + 1, 0);
  for (int s = 0; s < n_sys; ++s) {
    chunk0[s] = static_cast<int>(ch.size());
    const int64_t p0 = offsets[s], ns = offsets[s + 1] - p0;
    const int nbs = static_cast<int>((ns + TILE - 1) / TILE);
    for (int k = 0; k < nbs; ++k) {
      Chunk c{};
      c.sys = s;
      c.first = static_cast<int>(p0 + static_cast<int64_t>(k) * TILE);
      c.count = static_cast<int>(std::min<int64_t>(TILE, ns - static_cast<int64_t>(k) * TILE));
      c.cs = chunk0[s];
      c.nbs = nbs;
      ch.push_back(c);
    }
  }
  chunk0[n_sys] = static_cast<int>(ch.size());
  return ch;
}

}  // namespace

size_t gpu_build_scratch_bytes(int64_t n, int n_sys, int64_t cap) {
  const int64_t chunks = (n + TILE - 1) / TILE + n_sys;
  return layout(n, n_sys, chunks, cap).total;
}

cudaError_t gpu_build_tables(const GpuBuild& a, cudaStream_t st) {
  std::vector<int> chunk0;
  const std::vector<Chunk> ch = make_chunks(a.offsets, a.n_sys, chunk0);
  const Layout Lo = layout(a.n, a.n_sys, (a.n + TILE - 1) / TILE + a.n_sys, a.cap);
  if (Lo.total > a.scratch_bytes) return cudaErrorInvalidValue;
  // chunks, offsets and first chunks lie side by side: one copy
  std::vector<char> host(Lo.chunk0 + 4 * static_cast<size_t>(a.n_sys + 1) - Lo.chunks);
  std::memcpy(host.data(), ch.data(), sizeof(Chunk) * ch.size());
  std::memcpy(host.data() + (Lo.offs - Lo.chunks), a.offsets, 8 * static_cast<size_t>(a.n_sys + 1));
  std::memcpy(host.data() + (Lo.chunk0 - Lo.chunks), chunk0.data(), 4 * static_cast<size_t>(a.n_sys + 1));
  return cudaMemcpyAsync(at<char>(a.scratch, Lo.chunks), host.data(), host.size(), cudaMemcpyHostToDevice, st);
}

cudaError_t gpu_build(const GpuBuild& a, cudaStream_t st) {
  cudaError_t e = gpu_build_tables(a, st);
  return e != cudaSuccess ? e : gpu_build_kernels(a, st);
}

cudaError_t gpu_build_kernels(const GpuBuild& a, cudaStream_t st) {
  int nch = 0;
  for (int s = 0; s < a.n_sys; ++s) nch += static_cast<int>((a.offsets[s + 1] - a.offsets[s] + TILE - 1) / TILE);
  const Layout Lo = layout(a.n, a.n_sys, (a.n + TILE - 1) / TILE + a.n_sys, a.cap);
  if (Lo.total > a.scratch_bytes) return cudaErrorInvalidValue;
  void* S = a.scratch;
  uint64_t* keyA = at<uint64_t>(S, Lo.keyA);
  uint64_t* keyB = at<uint64_t>(S, Lo.keyB);
  uint32_t* valA = at<uint32_t>(S, Lo.valA);
  uint32_t* valB = at<uint32_t>(S, Lo.valB);
  int* cnt = at<int>(S, Lo.cnt);
  double* part = at<double>(S, Lo.part);
  SysGeo* sg = at<SysGeo>(S, Lo.sg);
  double* xs = at<double>(S, Lo.xs);
  double* ms = at<double>(S, Lo.ms);
  Chunk* dch = at<Chunk>(S, Lo.chunks);
  int64_t* doffs = at<int64_t>(S, Lo.offs);
  int* dchunk0 = at<int>(S, Lo.chunk0);
  int* lvl = at<int>(S, Lo.lvl);
  int* misc = at<int>(S, Lo.misc);
  int* spl = at<int>(S, Lo.spl);
  int* lpre = at<int>(S, Lo.lpre);
  int* bsum = at<int>(S, Lo.bsum);
  Cells C{at<uint64_t>(S, Lo.ckey), at<int>(S, Lo.cpar), at<int>(S, Lo.cpf), at<int>(S, Lo.cpc),
          at<int>(S, Lo.csys),      at<int>(S, Lo.cfc),  at<int>(S, Lo.cnc)};
  Props P{a.bmin, a.bmax, a.cube, a.M, a.com, a.S, a.key, a.geo, a.link, a.mp, a.pcount, a.cfirst};
  cudaError_t e;
#define OG_TRY(x)                       \
  do {                                  \
    if ((e = (x)) != cudaSuccess) return e; \
  } while (0)
  OG_TRY(cudaMemsetAsync(misc, 0, 4 * MISC, st));

  // ---- keys and the stable sort (8 passes of 8 bits over the 63-bit keys)
  k_bbox<<<BSUB * nch, TB, 0, st>>>(a.pos, a.mass, dch, part, misc);
  k_root<<<a.n_sys, TB, 0, st>>>(part, dchunk0, sg);
  k_morton<<<SUB * nch, TB, 0, st>>>(a.pos, dch, sg, keyA, valA);
  const Chunk* chunks = dch;
  if (nch <= SORT_CHUNKS4 && resident_blocks(k_sort<4>, TB, 4 * nch) == 4 * nch) {
    OG_TRY(launch_cooperative(k_sort<4>, 4 * nch, TB, 0, st, keyA, valA, keyB, valB, chunks, cnt, misc));
  } else if (nch <= SORT_CHUNKS2 && resident_blocks(k_sort<2>, TB, 2 * nch) == 2 * nch) {
    OG_TRY(launch_cooperative(k_sort<2>, 2 * nch, TB, 0, st, keyA, valA, keyB, valB, chunks, cnt, misc));
  } else {
    int* dtot = at<int>(S, Lo.dtot);
    const int segblocks = (256 * a.n_sys + TB / 32 - 1) / (TB / 32);
    for (int pass = 0; pass < 8; ++pass) {
      const int sh = 8 * pass;
      const bool even = (pass & 1) == 0;
      k_upsweep<<<nch, TB, 0, st>>>(even ? keyA : keyB, dch, sh, cnt);
      k_scan_digits<<<segblocks, TB, 0, st>>>(cnt, dchunk0, a.n_sys, dtot);
      k_downsweep<<<nch, TB, 0, st>>>(even ? keyA : keyB, even ? valA : valB, even ? keyB : keyA,
                                      even ? valB : valA, dch, sh, cnt, dtot);
    }
  }
  OG_TRY(cudaGetLastError());
  k_gather<<<grid_for(a.n, TB), TB, 0, st>>>(valA, a.pos, a.mass, a.n, xs, ms, a.parts, a.perm,
                                             at<int>(S, Lo.gmark));

  // ---- cells, level by level (sizes live in lvl[] on the device)
  k_roots<<<(std::max({a.n_sys, NLEV + 2, 2 * LBINS}) + 127) / 128, 128, 0, st>>>(a.n_sys, doffs, C, lvl,
                                                                                 at<int>(S, Lo.lhist));
  {
    // about a warp per cell that is split on the widest level; a small tree gets
    // few blocks, whose barriers are cheaper; up to 200,000 particles one an SM, half
    // of the places (65,536 particles 115 us, 119 with two; 131,072 130 and 134; 262,144
    // 164 and 155)
    const int64_t want = std::max<int64_t>(1, a.n / (16 * (LT / 32)));
    const int most = static_cast<int>(std::min<int64_t>(want, a.n <= 200000 ? 152 : LBMAX));
    const auto kernel = a.n < LROUNDS_N ? k_levels<1> : k_levels<LROUNDS>;
    OG_TRY(launch_cooperative(kernel, resident_blocks(kernel, LT, most), LT, 0, st, static_cast<const uint64_t*>(keyA), C,
                              a.n_leaf, lvl, spl, lpre, at<int>(S, Lo.nlist), bsum, static_cast<int>(a.cap), misc));
  }

  // ---- final (system-major) cell order
  const int gc = grid_for(a.cap, TB);
  int* ni = nullptr;
  if (a.n_sys > 1) {
    int* sstart = at<int>(S, Lo.sstart);
    int* send = at<int>(S, Lo.send);
    int* lofs = at<int>(S, Lo.lofs);
    ni = at<int>(S, Lo.ni);
    OG_TRY(cudaMemsetAsync(sstart, 0, 4 * static_cast<size_t>(a.n_sys) * NLEV, st));
    OG_TRY(cudaMemsetAsync(send, 0, 4 * static_cast<size_t>(a.n_sys) * NLEV, st));
    k_sys_bounds<<<gc, TB, 0, st>>>(lvl, C.sys, sstart, send);
    k_sys_offsets<<<1, 1024, 0, st>>>(a.n_sys, sstart, send, lofs, a.cell_off);
    k_new_index<<<gc, TB, 0, st>>>(lvl, C.sys, sstart, lofs, ni);
  }

  // ---- properties: every leaf at once, then the nodes deepest level first
  int* lorder = at<int>(S, Lo.lorder);
  int* lhist = at<int>(S, Lo.lhist);
  k_leaf_hist<<<gc, TB, 0, st>>>(C, lvl, lhist, misc, a.n_sys > 1 ? nullptr : a.cell_off);
  k_leaf_scatter<<<gc, TB, 0, st>>>(C, lvl, lhist, lhist + LBINS, lorder);
  k_leaf_props<<<grid_for(a.cap, LT_LEAF), LT_LEAF, 0, st>>>(C, lorder, misc, ni, xs, ms, P);
  OG_TRY(cudaGetLastError());
  OG_TRY(enqueue_nodes(a, Lo, C, ni, P, st));

  // ---- groups (ordered by first particle), work items and the result
  OG_TRY(enqueue_groups(a, Lo, true, st));
#undef OG_TRY
  return cudaGetLastError();
}

cudaError_t gpu_refit(const GpuBuild& a, cudaStream_t st) {
  const Layout Lo = layout(a.n, a.n_sys, (a.n + TILE - 1) / TILE + a.n_sys, a.cap);
  if (Lo.total > a.scratch_bytes) return cudaErrorInvalidValue;
  void* S = a.scratch;
  int nch = 0;
  for (int s = 0; s < a.n_sys; ++s) nch += static_cast<int>((a.offsets[s + 1] - a.offsets[s] + TILE - 1) / TILE);
  int* misc = at<int>(S, Lo.misc);
  const int* lvl = at<int>(S, Lo.lvl);
  Cells C{at<uint64_t>(S, Lo.ckey), at<int>(S, Lo.cpar), at<int>(S, Lo.cpf), at<int>(S, Lo.cpc),
          at<int>(S, Lo.csys),      at<int>(S, Lo.cfc),  at<int>(S, Lo.cnc)};
  Props P{a.bmin, a.bmax, a.cube, a.M, a.com, a.S, a.key, a.geo, a.link, a.mp, a.pcount, a.cfirst};
  const int* ni = a.n_sys > 1 ? at<int>(S, Lo.ni) : nullptr;
  const int gc = grid_for(a.cap, TB);
  cudaError_t e;
  // the status bits only: the counts of the build stay
  k_clear_status<<<1, 1, 0, st>>>(misc);
  k_bbox<<<BSUB * nch, TB, 0, st>>>(a.pos, a.mass, at<Chunk>(S, Lo.chunks), at<double>(S, Lo.part), misc);
  k_gather<<<grid_for(a.n, TB), TB, 0, st>>>(at<uint32_t>(S, Lo.valA), a.pos, a.mass, a.n, at<double>(S, Lo.xs),
                                             at<double>(S, Lo.ms), a.parts, a.perm, nullptr);
  k_leaf_props<<<grid_for(a.cap, LT_LEAF), LT_LEAF, 0, st>>>(C, at<int>(S, Lo.lorder), misc, ni, at<double>(S, Lo.xs), at<double>(S, Lo.ms), P);
  if ((e = enqueue_nodes(a, Lo, C, ni, P, st)) != cudaSuccess) return e;
  k_items<<<grid_for(a.n, TB), TB, 0, st>>>(&misc[M_NGROUPS], a.group_cell, a.group_sys, at<int>(S, Lo.ioff), P,
                                            item_args(a));
  k_finish<<<1, 1, 0, st>>>(lvl, misc, a.result);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return cudaSuccess;
}

cudaError_t gpu_build_items(const GpuBuild& a, cudaStream_t st) {
  const Layout Lo = layout(a.n, a.n_sys, (a.n + TILE - 1) / TILE + a.n_sys, a.cap);
  if (Lo.total > a.scratch_bytes) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(at<int>(a.scratch, Lo.misc) + M_BAR_ITEMS, 0, 4, st);
  return e != cudaSuccess ? e : enqueue_groups(a, Lo, false, st);
}

__global__ void k_pull(const uint4* __restrict__ src, uint4* __restrict__ dst, int64_t n16) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n16;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    dst[i] = src[i];
}

cudaError_t pull_host(void* dst, const void* src, size_t bytes, cudaStream_t st) {
  if ((reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(src) | bytes) & 15u) return cudaErrorInvalidValue;
  const int64_t n16 = static_cast<int64_t>(bytes / 16);
  if (n16 == 0) return cudaSuccess;
  k_pull<<<grid_for(n16, TB * 4), TB, 0, st>>>(static_cast<const uint4*>(src), static_cast<uint4*>(dst), n16);
  return cudaGetLastError();
}

cudaError_t gpu_unpermute(const float4* out, const int* perm, int64_t n, double* acc, double* pot, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_unpermute<<<grid_for(n, TB), TB, 0, st>>>(out, perm, n, acc, pot);
  return cudaGetLastError();
}

}  // namespace og

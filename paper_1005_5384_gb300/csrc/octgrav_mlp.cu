// octgrav_mlp.cu -- learned opening criterion: training samples (features and
// FP64 error labels) and training (FP32 forward/backward of the 12-64-64-1
// network, Adam), all on the GPU.
//
// A label is the error of accepting cell c for group g: the largest, over the
// group's particles i, of |a_multipole(c, i) - a_direct(members of c, i)| /
// |a_ref(i)|, with a_ref a tight reference of the particle's total
// acceleration. The network learns log10 of it from the inputs defined in
// octgrav_mlp.h; the walk then accepts a cell when the prediction is below a
// threshold.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "octgrav_grid.h"
#include "octgrav_internal.h"
#include "octgrav_mlp.h"

namespace og {
namespace {

// ---------------------------------------------------------------- samples

__global__ void feature_kernel(MlpSampleArgs a) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= a.n) return;
  const int item = a.item[s], c = a.cell[s];
  const int4 it = a.items[item];
  const float4 b0 = a.ibox[4 * item], b1 = a.ibox[4 * item + 1], b2 = a.ibox[4 * item + 2];
  const float4 b3 = a.ibox[4 * item + 3];
  const float3 gmin = make_float3(b0.x, b0.y, b0.z), gmax = make_float3(b1.x, b1.y, b1.z);
  const float3 chi = make_float3(b0.w, b1.w, b2.w), clo = make_float3(b2.x, b2.y, b2.z);
  const float4 r0 = a.mp[4 * it.x], r1 = a.mp[4 * it.x + 1];  // root centre of mass (hi, lo)
  const float ox = (chi.x - r0.x) + (clo.x - r1.x), oy = (chi.y - r0.y) + (clo.y - r1.y),
              oz = (chi.z - r0.z) + (clo.z - r1.z);
  const float f10 = static_cast<float>(__float_as_int(b3.y)) / static_cast<float>(a.n_group);
  const float f11 = mlp_lg2(sqrtf(ox * ox + oy * oy + oz * oz));
  float f[MLP_NF];
  mlp_features(a.geo[c], a.mp[4 * c], a.mp[4 * c + 1], a.mp[4 * c + 2], a.mp[4 * c + 3], gmin, gmax, chi, clo, f10,
               f11, f);
  for (int k = 0; k < MLP_NF; ++k) a.feat[MLP_NF * s + k] = f[k];
}

// One warp per (sample, chunk of 32 group particles): lane = particle.
__global__ void label_kernel(MlpSampleArgs a) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const int s = warp / a.chunks, chunk = warp % a.chunks;
  if (s >= a.n) return;
  const int item = a.item[s], c = a.cell[s];
  const float4 b3 = a.ibox[4 * item + 3];
  const int gfirst = __float_as_int(b3.x), gcount = __float_as_int(b3.y);
  const int k = chunk * 32 + lane;
  double e = 0.0;
  if (k < gcount) {
    const int i = gfirst + k;
    const float4 hi = a.parts[2 * i], lo = a.parts[2 * i + 1];
    const double xi = (double)hi.x + lo.x, yi = (double)hi.y + lo.y, zi = (double)hi.z + lo.z;
    // multipole (monopole + quadrupole, FP64 moments)
    const double* cm = a.com64 + 3 * c;
    const double* S = a.S64 + 6 * c;
    const double M = a.M64[c];
    const double y0 = xi - cm[0], y1 = yi - cm[1], y2 = zi - cm[2];
    const double r2 = y0 * y0 + y1 * y1 + y2 * y2 + a.eps2;
    const double r = sqrt(r2), r3 = r2 * r, r5 = r3 * r2, r7 = r5 * r2;
    const double s0 = S[0] * y0 + S[3] * y1 + S[4] * y2;
    const double s1 = S[3] * y0 + S[1] * y1 + S[5] * y2;
    const double s2 = S[4] * y0 + S[5] * y1 + S[2] * y2;
    const double ySy = y0 * s0 + y1 * s1 + y2 * s2, tr = S[0] + S[1] + S[2];
    const double cy = -M / r3 - 7.5 * ySy / r7 + 1.5 * tr / r5;
    const double am0 = cy * y0 + 3.0 * s0 / r5, am1 = cy * y1 + 3.0 * s1 / r5, am2 = cy * y2 + 3.0 * s2 / r5;
    // direct sum over the cell's members
    const int2 lk = a.link_first_count[c];
    double ad0 = 0, ad1 = 0, ad2 = 0;
    for (int j = lk.x; j < lk.x + lk.y; ++j) {
      const float4 hj = a.parts[2 * j], lj = a.parts[2 * j + 1];
      const double dx = ((double)hj.x + lj.x) - xi, dy = ((double)hj.y + lj.y) - yi,
                   dz = ((double)hj.z + lj.z) - zi;
      const double rinv = 1.0 / sqrt(dx * dx + dy * dy + dz * dz + a.eps2);
      const double mr3 = (double)hj.w * rinv * rinv * rinv;
      ad0 += mr3 * dx;
      ad1 += mr3 * dy;
      ad2 += mr3 * dz;
    }
    const float4 ar = a.aref[i];
    const double na = sqrt((double)ar.x * ar.x + (double)ar.y * ar.y + (double)ar.z * ar.z);
    const double ea = sqrt((am0 - ad0) * (am0 - ad0) + (am1 - ad1) * (am1 - ad1) + (am2 - ad2) * (am2 - ad2));
    e = na > 0 ? ea / na : 0.0;
  }
  for (int o = 16; o > 0; o >>= 1) e = fmax(e, __shfl_xor_sync(0xffffffffu, e, o));
  if (lane == 0) atomicMax(reinterpret_cast<unsigned long long*>(a.label64 + s), __double_as_longlong(e));
}

// ---------------------------------------------------------------- training

// Standardisation of the inputs: mean and deviation per feature in FP64, then
// x = (f - mean) / deviation, the range of x, and the targets log10(label).
// Blocks of 16 rows x 12 features take rows in strides of the grid and leave
// partial results that every block of the next pass adds in the same order.
// Three passes over the features (3 MB for 65,536 samples, from L2) and a few
// FP64 operations per value, where the host's loops took 2.4 ms of a call:
// 100 training steps on 65,536 samples 4.13 ms with them, 2.28 ms with these.
constexpr int SR = 16;             // rows of a block
constexpr int ST = SR * MLP_NF;    // its threads
constexpr int SB = 152;            // blocks

struct StdPart {  // one block's partial results
  double sum[MLP_NF], sq[MLP_NF];
  float lo[MLP_NF], hi[MLP_NF];
};
static_assert(SB * sizeof(StdPart) <= 4 * MLP_STD_FLOATS, "partial results fit their place");

// Sums of the features (SQ: of their squared distances from the mean).
template <bool SQ>
__global__ void __launch_bounds__(ST) std_sum_kernel(const float* __restrict__ feat, int64_t n, StdPart* part) {
  __shared__ double red[SR][MLP_NF];
  const int f = threadIdx.x % MLP_NF, r = threadIdx.x / MLP_NF;
  double mean = 0;
  if (SQ) {
#pragma unroll 8
    for (int b = 0; b < static_cast<int>(gridDim.x); ++b) mean += part[b].sum[f];
    mean /= static_cast<double>(n);
  }
  double s = 0;
  for (int64_t k = static_cast<int64_t>(blockIdx.x) * SR + r; k < n; k += static_cast<int64_t>(gridDim.x) * SR) {
    const double d = static_cast<double>(feat[k * MLP_NF + f]) - mean;
    s += SQ ? d * d : d;
  }
  red[r][f] = s;
  __syncthreads();
  if (r == 0) {
    for (int q = 1; q < SR; ++q) s += red[q][f];
    (SQ ? part[blockIdx.x].sq : part[blockIdx.x].sum)[f] = s;
  }
}

// feat becomes x in place; record[0..24) = mean, deviation (block 0).
__global__ void __launch_bounds__(ST) std_apply_kernel(float* feat, const float* __restrict__ label, int64_t n,
                                                        StdPart* part, float* __restrict__ y, float* __restrict__ record) {
  __shared__ float lo[SR][MLP_NF], hi[SR][MLP_NF];
  const int f = threadIdx.x % MLP_NF, r = threadIdx.x / MLP_NF;
  double mean = 0, sq = 0;
#pragma unroll 8
  for (int b = 0; b < static_cast<int>(gridDim.x); ++b) {
    mean += part[b].sum[f];
    sq += part[b].sq[f];
  }
  mean /= static_cast<double>(n);
  const double dev = fmax(sqrt(sq / static_cast<double>(n)), 1e-6);
  if (blockIdx.x == 0 && r == 0) {
    record[f] = static_cast<float>(mean);
    record[MLP_NF + f] = static_cast<float>(dev);
  }
  float l = INFINITY, h = -INFINITY;
  for (int64_t k = static_cast<int64_t>(blockIdx.x) * SR + r; k < n; k += static_cast<int64_t>(gridDim.x) * SR) {
    const float x = static_cast<float>((static_cast<double>(feat[k * MLP_NF + f]) - mean) / dev);
    feat[k * MLP_NF + f] = x;
    l = x < l ? x : l;
    h = h < x ? x : h;
    if (f == 0) {
      const double v = label[k];
      y[k] = static_cast<float>(log10(v < 1e-12 ? 1e-12 : v));
    }
  }
  lo[r][f] = l;
  hi[r][f] = h;
  __syncthreads();
  if (r == 0) {
    for (int q = 1; q < SR; ++q) {
      l = lo[q][f] < l ? lo[q][f] : l;
      h = h < hi[q][f] ? hi[q][f] : h;
    }
    part[blockIdx.x].lo[f] = l;
    part[blockIdx.x].hi[f] = h;
  }
}

// record[24..48) = range of x per feature.
__global__ void std_range_kernel(const StdPart* __restrict__ part, int blocks, float* __restrict__ record) {
  const int f = threadIdx.x;
  if (f >= MLP_NF) return;
  float l = INFINITY, h = -INFINITY;
#pragma unroll 8
  for (int b = 0; b < blocks; ++b) {
    l = part[b].lo[f] < l ? part[b].lo[f] : l;
    h = h < part[b].hi[f] ? part[b].hi[f] : h;
  }
  record[2 * MLP_NF + f] = l;
  record[3 * MLP_NF + f] = h;
}

// Counter-based uniform index in [0, n): splitmix64 of (seed, step, b).
__device__ __forceinline__ int sample_index(uint64_t seed, int step, int b, int n) {
  uint64_t z = seed + 0x9E3779B97F4A7C15ull * (static_cast<uint64_t>(step) * 1000003ull + b + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return static_cast<int>(z % static_cast<uint64_t>(n));
}

constexpr int TB = 32;             // samples per tile: one per lane
constexpr int GT = 256;            // threads of the gradient kernel (8 warps, 8 hidden units each)
constexpr int RS = MLP_NH + 4;     // row stride of the activations: 16-byte rows, 8 rows on distinct banks
constexpr int XS = MLP_NF + 8;     // row stride of the inputs

struct GradSmem {
  float4 w1t[MLP_NF][MLP_NH / 4];  // W1 transposed: 8 consecutive units of one input are two 16-byte words
  float4 w2t[MLP_NH][MLP_NH / 4];  // W2 transposed (layer 2) ...
  float4 w2[MLP_NH][RS / 4];       // ... and as it is (back through layer 2)
  float4 xs[TB][XS / 4];
  float4 h1[TB][RS / 4];           // relu(z1); z1 > 0 iff h1 > 0
  float4 dz2[TB][RS / 4];
  float4 d1[TB][RS / 4];           // dz1
  float b1[MLP_NH], b2[MLP_NH], w3[MLP_NH];
  float ypart[GT / 32][TB];        // warps' shares of the output
  float ts[TB];
  float dy[2];                     // sums over the tile: dy and L
  float gw3[MLP_NH];               // and w3's gradient
  float b3;
};

__device__ __forceinline__ void fma8(float* z, const float4* w, float x) {
  const float4 a = w[0], b = w[1];
  z[0] = fmaf(a.x, x, z[0]);
  z[1] = fmaf(a.y, x, z[1]);
  z[2] = fmaf(a.z, x, z[2]);
  z[3] = fmaf(a.w, x, z[3]);
  z[4] = fmaf(b.x, x, z[4]);
  z[5] = fmaf(b.y, x, z[5]);
  z[6] = fmaf(b.z, x, z[6]);
  z[7] = fmaf(b.w, x, z[7]);
}

// One block's share of the gradient of L = sum_b (y_b - t_b)^2 / (2B), written
// to part[block] (MLP_PART floats: the parameters, then L).
//
// FP32 FMAs and shared-memory reads bound it (6 x 5057 flops a sample), so the
// layout is made for the reads. Layers: lane = sample, warp w = units 8w ..
// 8w + 7; a weight row's 8 values are the same for the whole warp (two
// broadcast 16-byte reads for 8 FMAs), a sample's activations are read 16
// bytes at a time from rows 8 of which lie on distinct banks. Weight
// gradients: a 4 x 4 tile of (unit, input) per thread, summed over the
// samples in registers and over the block's tiles, and written once: no
// atomics, so a step's result does not depend on scheduling. One output per thread with
// W2[j][i] read at a stride of 64 floats put all 32 lanes on one bank:
// 43 us a step at B = 4096, 17 us so (both with the parameter update as a second
// launch).
__device__ __forceinline__ void block_gradient(GradSmem& S, const float* w, const float* __restrict__ X,
                                               const float* __restrict__ t, int n_total, int B, int step,
                                               uint64_t seed, int use_all, float* __restrict__ part) {
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const float* b1 = w + MLP_NH * MLP_NF;
  const float* W2 = b1 + MLP_NH;
  const float* b2 = W2 + MLP_NH * MLP_NH;
  const float* w3 = b2 + MLP_NH;
  float* w1t = reinterpret_cast<float*>(S.w1t);
  float* w2t = reinterpret_cast<float*>(S.w2t);
  float* w2s = reinterpret_cast<float*>(S.w2);
  for (int k = tid; k < MLP_NH * MLP_NF; k += GT) w1t[(k % MLP_NF) * MLP_NH + k / MLP_NF] = __ldcg(w + k);
  for (int k = tid; k < MLP_NH * MLP_NH; k += GT) w2s[(k / MLP_NH) * RS + k % MLP_NH] = __ldcg(W2 + k);
  __syncthreads();
  for (int k = tid; k < MLP_NH * MLP_NH; k += GT) w2t[k] = w2s[(k % MLP_NH) * RS + k / MLP_NH];
  if (tid < MLP_NH) {
    S.b1[tid] = __ldcg(b1 + tid);
    S.b2[tid] = __ldcg(b2 + tid);
    S.w3[tid] = __ldcg(w3 + tid);
  }
  if (tid == 0) S.b3 = __ldcg(w3 + MLP_NH);
  const float invB = 1.f / static_cast<float>(B);
  const int u0 = 8 * wp;                                // this warp's units
  const int ja = 4 * (tid >> 4), ib = 4 * (tid & 15);   // this thread's 4 x 4 tile of W2's gradient
  const int jc = tid >> 2, ic = 3 * (tid & 3);          // and its three entries of W1's
  float g2[4][4] = {}, g1[3] = {0.f, 0.f, 0.f};
  float gb = 0.f;  // threads 0..63: b1; 64..127: b2; 128..191: w3; 192: b3; 193: L
  const int tiles = (B + TB - 1) / TB;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int base = tile * TB, nb = min(TB, B - base);
    __syncthreads();  // the weights are in, the last tile's activations are free
    for (int k = tid; k < TB * MLP_NF; k += GT) {
      const int r = k / MLP_NF, f = k % MLP_NF;
      float v = 0.f;
      if (r < nb) {
        const int sidx = use_all ? base + r : sample_index(seed, step, base + r, n_total);
        v = X[static_cast<size_t>(sidx) * MLP_NF + f];
        if (f == 0) S.ts[r] = t[sidx];
      }
      reinterpret_cast<float*>(S.xs[r])[f] = v;
    }
    __syncthreads();
    // layer 1
    float z[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) z[k] = S.b1[u0 + k];
#pragma unroll
    for (int q = 0; q < MLP_NF / 4; ++q) {
      const float4 x = S.xs[lane][q];
      fma8(z, &S.w1t[4 * q][u0 / 4], x.x);
      fma8(z, &S.w1t[4 * q + 1][u0 / 4], x.y);
      fma8(z, &S.w1t[4 * q + 2][u0 / 4], x.z);
      fma8(z, &S.w1t[4 * q + 3][u0 / 4], x.w);
    }
    S.h1[lane][u0 / 4] = make_float4(fmaxf(z[0], 0.f), fmaxf(z[1], 0.f), fmaxf(z[2], 0.f), fmaxf(z[3], 0.f));
    S.h1[lane][u0 / 4 + 1] = make_float4(fmaxf(z[4], 0.f), fmaxf(z[5], 0.f), fmaxf(z[6], 0.f), fmaxf(z[7], 0.f));
    __syncthreads();
    // layer 2
#pragma unroll
    for (int k = 0; k < 8; ++k) z[k] = S.b2[u0 + k];
#pragma unroll 4
    for (int q = 0; q < MLP_NH / 4; ++q) {
      const float4 h = S.h1[lane][q];
      fma8(z, &S.w2t[4 * q][u0 / 4], h.x);
      fma8(z, &S.w2t[4 * q + 1][u0 / 4], h.y);
      fma8(z, &S.w2t[4 * q + 2][u0 / 4], h.z);
      fma8(z, &S.w2t[4 * q + 3][u0 / 4], h.w);
    }
    // output, residual
    float yp = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) yp = fmaf(S.w3[u0 + k], fmaxf(z[k], 0.f), yp);
    S.ypart[wp][lane] = yp;
    __syncthreads();
    float res = 0.f;  // every warp adds the shares in the same order
    if (lane < nb) {
      float y = S.b3;
#pragma unroll
      for (int q = 0; q < GT / 32; ++q) y += S.ypart[q][lane];
      res = y - S.ts[lane];
    }
    const float dy = res * invB;
    if (wp == 0) {
      float l = 0.5f * res * res * invB, d = dy;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        l += __shfl_xor_sync(0xffffffffu, l, o);
        d += __shfl_xor_sync(0xffffffffu, d, o);
      }
      if (lane == 0) S.dy[0] = d, S.dy[1] = l;
    }
    // w3's gradient and dz2 = dy w3 [z2 > 0]
    float dz[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      float g = dy * fmaxf(z[k], 0.f);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
      if (lane == 0) S.gw3[u0 + k] = g;
      dz[k] = z[k] > 0.f ? dy * S.w3[u0 + k] : 0.f;
    }
    S.dz2[lane][u0 / 4] = make_float4(dz[0], dz[1], dz[2], dz[3]);
    S.dz2[lane][u0 / 4 + 1] = make_float4(dz[4], dz[5], dz[6], dz[7]);
    __syncthreads();
    // dz1[r][i] = (sum_j dz2[r][j] W2[j][i]) [h1 > 0]
    float e[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int q = 0; q < MLP_NH / 4; ++q) {
      const float4 d = S.dz2[lane][q];
      fma8(e, &S.w2[4 * q][u0 / 4], d.x);
      fma8(e, &S.w2[4 * q + 1][u0 / 4], d.y);
      fma8(e, &S.w2[4 * q + 2][u0 / 4], d.z);
      fma8(e, &S.w2[4 * q + 3][u0 / 4], d.w);
    }
    const float4 ha = S.h1[lane][u0 / 4], hb = S.h1[lane][u0 / 4 + 1];
    S.d1[lane][u0 / 4] = make_float4(ha.x > 0.f ? e[0] : 0.f, ha.y > 0.f ? e[1] : 0.f, ha.z > 0.f ? e[2] : 0.f,
                                     ha.w > 0.f ? e[3] : 0.f);
    S.d1[lane][u0 / 4 + 1] = make_float4(hb.x > 0.f ? e[4] : 0.f, hb.y > 0.f ? e[5] : 0.f, hb.z > 0.f ? e[6] : 0.f,
                                         hb.w > 0.f ? e[7] : 0.f);
    // W2's gradient: sum_r dz2[r][j] h1[r][i]
#pragma unroll 4
    for (int r = 0; r < TB; ++r) {
      const float4 d = S.dz2[r][ja / 4], h = S.h1[r][ib / 4];
      const float dd[4] = {d.x, d.y, d.z, d.w}, hh[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) g2[p][q] = fmaf(dd[p], hh[q], g2[p][q]);
    }
    __syncthreads();
    // W1's gradient: sum_r dz1[r][j] x[r][i]; the biases' and w3's
#pragma unroll 4
    for (int r = 0; r < TB; ++r) {
      const float d = reinterpret_cast<const float*>(S.d1[r])[jc];
      const float* x = reinterpret_cast<const float*>(S.xs[r]) + ic;
#pragma unroll
      for (int q = 0; q < 3; ++q) g1[q] = fmaf(d, x[q], g1[q]);
    }
    if (tid < 2 * MLP_NH) {
      const float* col = reinterpret_cast<const float*>(tid < MLP_NH ? S.d1[0] : S.dz2[0]) + (tid & (MLP_NH - 1));
      float g = 0.f;
#pragma unroll 8
      for (int r = 0; r < TB; ++r) g += col[r * RS];
      gb += g;
    } else if (tid < 3 * MLP_NH) {
      gb += S.gw3[tid - 2 * MLP_NH];
    } else if (tid < 3 * MLP_NH + 2) {
      gb += S.dy[tid - 3 * MLP_NH];
    }
  }
  float* out = part + static_cast<size_t>(blockIdx.x) * MLP_PART;
  float* o2 = out + MLP_NH * MLP_NF + MLP_NH;
#pragma unroll
  for (int q = 0; q < 3; ++q) out[jc * MLP_NF + ic + q] = g1[q];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) o2[(ja + p) * MLP_NH + ib + q] = g2[p][q];
  if (tid < MLP_NH) out[MLP_NH * MLP_NF + tid] = gb;
  else if (tid < 3 * MLP_NH + 2) o2[MLP_NH * MLP_NH + tid - MLP_NH] = gb;  // b2, w3, b3, L follow each other
}

__global__ void __launch_bounds__(GT) grad_kernel(const float* w, const float* __restrict__ X,
                                                   const float* __restrict__ t, int n, float* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem[];
  block_gradient(*reinterpret_cast<GradSmem*>(smem), w, X, t, n, n, 0, 0, 1, part);
}

// Sum of the blocks' shares per parameter, and of L. A block takes 32
// parameters: warp s adds the shares s, s + 8, ..., the warps' sums are added in
// order.
__global__ void __launch_bounds__(256) reduce_kernel(const float* __restrict__ part, int blocks,
                                                      float* __restrict__ grad, float* __restrict__ loss) {
  __shared__ float sum[8][32];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, k = 32 * blockIdx.x + lane;
  float s = 0.f;
  if (k <= MLP_NPARAM) {
#pragma unroll 8
    for (int b = wp; b < blocks; b += 8) s += part[static_cast<size_t>(b) * MLP_PART + k];
  }
  sum[wp][lane] = s;
  __syncthreads();
  if (wp || k > MLP_NPARAM) return;
  float g = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) g += sum[q][lane];
  if (k == MLP_NPARAM) *loss = g;
  else grad[k] = g;
}

// `steps` training steps in one cooperative launch. Per step: every block's
// share of the gradient, a grid barrier, then the blocks add the shares of
// their range of parameters (a thread per parameter and slice of the shares,
// the slices in order) and apply the Adam update, and a second barrier. coef
// holds the steps' bias corrections 1 / (1 - 0.9^k) and 1 / (1 - 0.999^k).
//
// A step is a chain of short dependent phases, so what it waits for between
// them counts: as two launches it took 17 us at B = 4096, 14 us so.
__global__ void __launch_bounds__(GT) train_kernel(float* w, float* m, float* v, const float* __restrict__ X,
                                                    const float* __restrict__ t, int n_total, int B, int step0,
                                                    int steps, uint64_t seed, float lr,
                                                    const float2* __restrict__ coef, float* part,
                                                    float* loss, int* bar) {
  extern __shared__ __align__(16) unsigned char smem[];
  GradSmem& S = *reinterpret_cast<GradSmem*>(smem);
  float* sum = reinterpret_cast<float*>(S.h1);  // free between the gradients
  const int grid = gridDim.x, tid = threadIdx.x;
  const int per = (MLP_NPARAM + 1 + grid - 1) / grid;      // parameters of a block (the last is L)
  const int k0 = min(MLP_NPARAM + 1, static_cast<int>(blockIdx.x) * per), nk = min(MLP_NPARAM + 1 - k0, per);
  const int slices = max(1, GT / per);
  int bars = 0;
  for (int k = 0; k < steps; ++k) {
    block_gradient(S, w, X, t, n_total, B, step0 + k, seed, 0, part);
    if (!grid_barrier(bar, ++bars * grid, bar + 1, 1)) return;
    const float2 c = coef[k];
    for (int e0 = 0; e0 < nk; e0 += GT) {  // one round unless the grid is tiny
      const int e = e0 + (slices > 1 ? tid % per : tid), q = slices > 1 ? tid / per : 0;
      float s = 0.f;
      if (e < nk && q < slices) {
#pragma unroll 8
        for (int b = q; b < grid; b += slices) s += __ldcg(part + static_cast<size_t>(b) * MLP_PART + k0 + e);
        if (slices > 1) sum[q * per + e] = s;
      }
      if (slices > 1) __syncthreads();
      if (e < nk && q == 0) {
        for (int r = 1; r < slices; ++r) s += sum[r * per + e];
        const int p = k0 + e;
        if (p == MLP_NPARAM) {
          *loss = s;
        } else {
          const float mk = 0.9f * m[p] + 0.1f * s;
          const float vk = 0.999f * v[p] + 0.001f * s * s;
          m[p] = mk;
          v[p] = vk;
          w[p] -= lr * (mk * c.x) / (sqrtf(vk * c.y) + 1e-8f);
        }
      }
    }
    if (!grid_barrier(bar, ++bars * grid, bar + 1, 1)) return;
  }
}

}  // namespace

cudaError_t mlp_sample_features(const MlpSampleArgs& a, cudaStream_t st) {
  if (a.n <= 0) return cudaSuccess;
  feature_kernel<<<(a.n + 127) / 128, 128, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t mlp_sample_labels(const MlpSampleArgs& a, cudaStream_t st) {
  if (a.n <= 0) return cudaSuccess;
  const long long warps = static_cast<long long>(a.n) * a.chunks;
  label_kernel<<<static_cast<unsigned>((warps * 32 + 255) / 256), 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t mlp_standardise(float* feat, const float* label, int64_t n, float* scratch, float* y, float* record,
                            cudaStream_t st) {
  const int64_t rows = (n + SR - 1) / SR;
  const int blocks = rows < SB ? static_cast<int>(rows) : SB;
  StdPart* part = reinterpret_cast<StdPart*>(scratch);
  std_sum_kernel<false><<<blocks, ST, 0, st>>>(feat, n, part);
  std_sum_kernel<true><<<blocks, ST, 0, st>>>(feat, n, part);
  std_apply_kernel<<<blocks, ST, 0, st>>>(feat, label, n, part, y, record);
  std_range_kernel<<<1, 32, 0, st>>>(part, blocks, record);
  return cudaGetLastError();
}

// Blocks of a gradient over B samples: one per tile of 32, at most two per SM.
int mlp_blocks(int B) {
  const int tiles = B / TB + (B % TB != 0);
  return tiles < 2 * 152 ? tiles : 2 * 152;
}

cudaError_t mlp_gradient(const float* w, const float* X, const float* t, int n, float* part, float* grad, float* loss,
                         cudaStream_t st) {
  const cudaError_t e = cudaFuncSetAttribute(grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(GradSmem));
  if (e != cudaSuccess) return e;
  grad_kernel<<<mlp_blocks(n), GT, sizeof(GradSmem), st>>>(w, X, t, n, part);
  reduce_kernel<<<(MLP_NPARAM + 1 + 31) / 32, 256, 0, st>>>(part, mlp_blocks(n), grad, loss);
  return cudaGetLastError();
}

cudaError_t mlp_train_steps(float* w, float* m, float* v, const float* X, const float* t, int n_total, int B, int step0,
                            int steps, uint64_t seed, float lr, const float2* coef, float* part, float* loss, int* bar,
                            cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(GradSmem));
  if (e != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(bar, 0, 8, st)) != cudaSuccess) return e;
  return launch_cooperative(train_kernel, resident_blocks(train_kernel, GT, mlp_blocks(B), sizeof(GradSmem)), GT,
                            sizeof(GradSmem), st, w, m, v, X, t, n_total, B, step0, steps, seed, lr, coef, part, loss, bar);
}

}  // namespace og

// aap.cu -- the AAP weight quantiser of Sec. 4.1 (eq. Ternary) on the GPU, as the training forward
// applies it, and the expansion of 2-bit ternary weights into the decoder's bf16 tile stream.
//
// aap_ternarize_kernel: one cluster of CTAs per weight tensor.
//   gamma = Percentile(|W|, 0.5): the median of |W| with linear interpolation between the two
//     middle order statistics (position 0.5 (len - 1)), the two order statistics found exactly by
//     a most-significant-digit radix select over the bit patterns of |W| (for non-negative
//     floats the bit patterns order like the values), the interpolation in double precision;
//   scale = gamma * delta (fp32), t = RoundClip(W / (scale + eps), -1, 1) with an IEEE fp32
//     division and round to nearest even;
//   t goes out in the 2-bit format of aecct_create (weight i at bits 2 (i % 4) of byte i / 4:
//     00 = 0, 01 = +1, 11 = -1), and optionally as the training forward's weight scale * t.
// unpack_weights_kernel: the 2-bit weights of aecct_create, expanded on the GPU into bf16 K-major
//   core-matrix chunks in WeightSchedule order (one 16-byte core-matrix row per thread).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "aecct_internal.h"

namespace cg = cooperative_groups;

namespace aecct {

namespace {

constexpr int kSelectThreads = 512;
constexpr int kSelectQuads = 4;  // groups of 4 weights that a thread keeps in registers
constexpr int kSelectSlice = 4 * kSelectThreads * kSelectQuads;  // weights of a CTA that are read once
constexpr int kSelectBins = 2048;
constexpr int kSelectMaxCluster = 8;

struct TernarizeArgs {
  const float *w[kTernarizeMaxTensors];
  int64_t off[kTernarizeMaxTensors];  // first element of tensor j in wq (and of its codes * 4)
  int64_t len[kTernarizeMaxTensors];
  float delta[kTernarizeMaxTensors];
};

// One cluster per tensor, each CTA a contiguous slice of its groups of 4 weights, the first
// kSelectQuads groups of a thread in registers for every pass (a longer slice's rest is read again).
// The median's two order statistics: a most-significant-digit radix select over the 31-bit patterns
// of |W| with digits of 11, 10 and 10 bits (11 bits take the exponent and 3 bits of the mantissa, so
// that weights of one scale spread over tens of bins: with 8-bit digits nearly all of them meet in
// a few, and the shared-memory atomics on those run one after the other), then the smallest pattern
// above the lower one where the upper is another.  CTAs count into their own histogram, add its
// non-empty bins to the first CTA's over distributed shared memory, and that CTA finds the digit.
// Bound by the latency of those rounds (two cluster barriers each): the weights are read once, the
// codes written once.  All 60 tensors of a d = 128, N = 10 model: 91 us with one CTA per tensor and two
// selects of four 8-bit digits, each reading the weights again, now 31 us.
__global__ void __launch_bounds__(kSelectThreads) aap_ternarize_kernel(const __grid_constant__ TernarizeArgs a,
                                                                       float eps, uint8_t *packed, float *scale,
                                                                       float *wq) {
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ uint32_t hist[kSelectBins];  // this CTA's counts
  __shared__ uint32_t tot[kSelectBins];   // first CTA: the cluster's counts
  __shared__ uint32_t wsum[kSelectThreads / 32];
  __shared__ uint32_t sel[3];  // digit, weights below it, weights in it
  __shared__ uint32_t above;   // first CTA: smallest pattern above the lower order statistic
  const int C = static_cast<int>(cluster.num_blocks()), rank = static_cast<int>(cluster.block_rank());
  const int j = blockIdx.x / C, tid = threadIdx.x, lane = tid & 31;
  const int64_t len = a.len[j], off = a.off[j];
  const float *__restrict__ wt = a.w[j];
  const bool vec = ((reinterpret_cast<uintptr_t>(wt) | reinterpret_cast<uintptr_t>(wq)) & 15u) == 0;  // (off is a multiple of 4)
  const int64_t nq = len / 4, per = (nq + C - 1) / C;
  const int64_t q0 = min(nq, rank * per) + tid, q1 = min(nq, (rank + 1) * per);
  auto load = [&](int64_t q) -> float4 {
    if (vec) return __ldg(reinterpret_cast<const float4 *>(wt) + q);
    return make_float4(__ldg(wt + 4 * q), __ldg(wt + 4 * q + 1), __ldg(wt + 4 * q + 2), __ldg(wt + 4 * q + 3));
  };
  float4 v[kSelectQuads];
#pragma unroll
  for (int i = 0; i < kSelectQuads; ++i)
    if (q0 + i * kSelectThreads < q1) v[i] = load(q0 + i * kSelectThreads);
  auto each_quad = [&](auto &&f) {
#pragma unroll
    for (int i = 0; i < kSelectQuads; ++i)
      if (q0 + i * kSelectThreads < q1) f(q0 + i * kSelectThreads, v[i]);
    for (int64_t q = q0 + kSelectQuads * kSelectThreads; q < q1; q += kSelectThreads) f(q, load(q));
  };
  auto each_key = [&](auto &&f) {
    each_quad([&](int64_t, const float4 &x) {
      f(__float_as_uint(x.x) & 0x7FFFFFFFu), f(__float_as_uint(x.y) & 0x7FFFFFFFu);
      f(__float_as_uint(x.z) & 0x7FFFFFFFu), f(__float_as_uint(x.w) & 0x7FFFFFFFu);
    });
  };
  uint32_t *tot0 = cluster.map_shared_rank(tot, 0), *above0 = cluster.map_shared_rank(&above, 0);
  for (int b = tid; b < kSelectBins; b += kSelectThreads) hist[b] = 0, tot[b] = 0;
  if (tid == 0) above = 0xFFFFFFFFu;
  cluster.sync();
  // Percentile(|W|, 0.5): position 0.5 (len - 1) between the order statistics lo and lo + 1
  const double pos = 0.5 * static_cast<double>(len - 1);
  const int64_t lo = static_cast<int64_t>(floor(pos));
  const double frac = pos - static_cast<double>(lo);
  uint32_t k = static_cast<uint32_t>(lo), prefix = 0, mask = 0;
#pragma unroll 1
  for (int pass = 0; pass < 3; ++pass) {
    const int shift = pass == 0 ? 20 : pass == 1 ? 10 : 0;
    const uint32_t digits = pass == 0 ? 2047u : 1023u;
    each_key([&](uint32_t key) {
      if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & digits], 1u);
    });
    __syncthreads();
    for (int b = tid; b < kSelectBins; b += kSelectThreads) {
      const uint32_t c = hist[b];
      if (c) atomicAdd(tot0 + b, c), hist[b] = 0;
    }
    cluster.sync();
    if (rank == 0) {
      // the digit whose range of ranks holds k: a scan over the bins, 4 to a thread
      const uint4 c4 = reinterpret_cast<const uint4 *>(tot)[tid];
      const uint32_t sum = c4.x + c4.y + c4.z + c4.w;
      uint32_t inc = sum;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
      }
      if (lane == 31) wsum[tid >> 5] = inc;
      __syncthreads();
      uint32_t below = inc - sum;
      for (int i = 0; i < (tid >> 5); ++i) below += wsum[i];
      if (k >= below && k - below < sum) {
        const uint32_t c[4] = {c4.x, c4.y, c4.z, c4.w};
        int b = 0;
        while (k - below >= c[b]) below += c[b], ++b;
        for (int r = 0; r < C; ++r) {
          uint32_t *s = cluster.map_shared_rank(sel, r);
          s[0] = 4u * static_cast<uint32_t>(tid) + static_cast<uint32_t>(b), s[1] = below, s[2] = c[b];
        }
      }
      reinterpret_cast<uint4 *>(tot)[tid] = make_uint4(0u, 0u, 0u, 0u);
    }
    cluster.sync();
    k -= sel[1];
    prefix |= sel[0] << shift;
    mask |= digits << shift;
  }
  const uint32_t klo = prefix;
  uint32_t khi = klo;
  if (lo + 1 < len && k + 1 >= sel[2]) {  // (the same in every CTA) no further weight of the lower pattern
    uint32_t mn = 0xFFFFFFFFu;
    each_key([&](uint32_t key) {
      if (key > klo) mn = min(mn, key);
    });
    mn = __reduce_min_sync(0xffffffffu, mn);
    if (lane == 0 && mn != 0xFFFFFFFFu) atomicMin(above0, mn);
    cluster.sync();
    khi = *above0;
  }
  const double alo = static_cast<double>(__uint_as_float(klo)), ahi = static_cast<double>(__uint_as_float(khi));
  const float gamma = static_cast<float>(alo + frac * (ahi - alo));
  const float sc = __fmul_rn(gamma, a.delta[j]), den = __fadd_rn(sc, eps);
  if (rank == 0 && tid == 0) scale[j] = sc;
  uint8_t *pk = packed + off / 4;
  each_quad([&](int64_t q, const float4 &x) {
    const float xs[4] = {x.x, x.y, x.z, x.w};
    uint32_t byte = 0;
    float t[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float r = rintf(__fdiv_rn(xs[i], den));
      // RoundClip to the integers {-1, 0, +1} (a rounded -0 is the integer 0)
      t[i] = r >= 1.0f ? 1.0f : (r <= -1.0f ? -1.0f : 0.0f);
      byte |= (t[i] > 0.0f ? 1u : (t[i] < 0.0f ? 3u : 0u)) << (2 * i);
      t[i] = __fmul_rn(sc, t[i]);
    }
    pk[q] = static_cast<uint8_t>(byte);
    if (wq) {
      float *o = wq + off + 4 * q;
      if (vec) *reinterpret_cast<float4 *>(o) = make_float4(t[0], t[1], t[2], t[3]);
      else o[0] = t[0], o[1] = t[1], o[2] = t[2], o[3] = t[3];
    }
  });
  cluster.sync();  // no CTA leaves while another reads the first one's shared memory
}

struct UnpackArgs {
  int D, n_chunks;
  uint32_t layer_bytes;
  ChunkDesc chunk[32];
};

// one thread per (layer, chunk, row, 8-column group): 8 ternary codes (2 bytes of the packed row)
// -> one 16-byte core-matrix row of bf16
__global__ void unpack_weights_kernel(const uint8_t *__restrict__ packed, int n_layers, const UnpackArgs a,
                                      uint8_t *wstream) {
  const int D = a.D, F = 4 * D;
  const size_t per_layer_packed = 3u * static_cast<size_t>(D) * D;  // 12 D^2 weights / 4
  int64_t item = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  // items per layer: sum over chunks of nrows * kcols / 8
  int64_t per_layer = 0;
  for (int c = 0; c < a.n_chunks; ++c) per_layer += static_cast<int64_t>(a.chunk[c].nrows) * a.chunk[c].kcols / 8;
  if (item >= per_layer * n_layers) return;
  const int l = static_cast<int>(item / per_layer);
  item -= static_cast<int64_t>(l) * per_layer;
  int c = 0;
  for (; c < a.n_chunks; ++c) {
    const int64_t n = static_cast<int64_t>(a.chunk[c].nrows) * a.chunk[c].kcols / 8;
    if (item < n) break;
    item -= n;
  }
  const ChunkDesc ch = a.chunk[c];
  const int rr = static_cast<int>(item / (ch.kcols / 8)), cg = static_cast<int>(item % (ch.kcols / 8));
  const int n = ch.n0 + rr, k = ch.k0 + 8 * cg;
  // the ABI tensor and row of GEMM row n: QKV rows [0, D) W_q, [D, 2D) W_k, [2D, 3D) W_v; O W_o;
  // FFN1 W_1 [F][D] (output column n holds hidden unit ffn1_unit_of_column(D, n)); FFN2 W_2 [D][F]
  size_t toff;
  int row, din;
  if (ch.gemm == 0) toff = static_cast<size_t>(n / D) * D * D / 4, row = n % D, din = D;
  else if (ch.gemm == 1) toff = 3u * static_cast<size_t>(D) * D / 4, row = n, din = D;
  else if (ch.gemm == 2) toff = static_cast<size_t>(D) * D, row = ffn1_unit_of_column(D, n), din = D;
  else toff = static_cast<size_t>(D) * D + static_cast<size_t>(F) * D / 4, row = n, din = F;
  const uint8_t *src = packed + per_layer_packed * l + toff + static_cast<size_t>(row) * (din / 4) + k / 4;
  const uint32_t bits = static_cast<uint32_t>(src[0]) | (static_cast<uint32_t>(src[1]) << 8);
  uint32_t h[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t pair = 0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const uint32_t code = (bits >> (2 * (2 * i + s))) & 3u;
      const uint32_t bf = code == 1u ? 0x3F80u : (code == 3u ? 0xBF80u : 0u);  // +1, -1, 0 in bf16
      pair |= bf << (16 * s);
    }
    h[i] = pair;
  }
  uint8_t *dst = wstream + static_cast<size_t>(l) * a.layer_bytes + ch.off + core_off(rr, 8 * cg, ch.kcols);
  *reinterpret_cast<uint4 *>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
}

}  // namespace

cudaError_t launch_aap_ternarize(const float *const *w, int n, const int64_t *len, const float *delta, float eps,
                                 uint8_t *packed, float *scale, float *wq, cudaStream_t stream) {
  int64_t off = 0;
  for (int j0 = 0; j0 < n; j0 += kTernarizeMaxTensors) {
    TernarizeArgs a = {};
    const int count = n - j0 < kTernarizeMaxTensors ? n - j0 : kTernarizeMaxTensors;
    int64_t first = off, longest = 0;
    for (int j = 0; j < count; ++j) {
      a.w[j] = w[j0 + j];
      a.off[j] = off - first;
      a.len[j] = len[j0 + j];
      a.delta[j] = delta[j0 + j];
      off += len[j0 + j];
      longest = len[j0 + j] > longest ? len[j0 + j] : longest;
    }
    // the fewest CTAs that keep the longest tensor in registers, at most the portable cluster size
    int C = 1;
    while (C < kSelectMaxCluster && static_cast<int64_t>(C) * kSelectSlice < longest) C *= 2;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C, attr[0].val.clusterDim.y = 1, attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(count * C);
    cfg.blockDim = dim3(kSelectThreads);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, aap_ternarize_kernel, a, eps, packed + first / 4,
                                             scale + j0, wq ? wq + first : nullptr);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_unpack_weights(const uint8_t *packed, int n_layers, int D, const ChunkDesc *chunks, int n_chunks,
                                  uint32_t layer_bytes, uint8_t *wstream, cudaStream_t stream) {
  UnpackArgs a = {};
  a.D = D, a.n_chunks = n_chunks, a.layer_bytes = layer_bytes;
  int64_t per_layer = 0;
  for (int c = 0; c < n_chunks; ++c) {
    a.chunk[c] = chunks[c];
    per_layer += static_cast<int64_t>(chunks[c].nrows) * chunks[c].kcols / 8;
  }
  const int64_t items = per_layer * n_layers;
  const int threads = 256;
  unpack_weights_kernel<<<static_cast<unsigned>((items + threads - 1) / threads), threads, 0, stream>>>(packed, n_layers,
                                                                                                        a, wstream);
  return cudaGetLastError();
}

}  // namespace aecct

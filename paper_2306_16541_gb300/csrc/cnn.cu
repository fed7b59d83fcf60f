// cnn.cu -- CNN_skel (Sec. 4.2): the canonical weight volume W^c generated from
// a constant latent z by a fully-connected layer and five 3D transposed
// convolutions (kernel 4, stride 2, padding 1: 1^3 -> 32^3), LeakyReLU(0.2)
// between layers and a softmax over the 25 channels (after adding log(prior)
// when one is given); and its backward from dL/dW^c to the network's weights.
//
// Parameters (float32, packed in this order): W_fc [C0][256], b_fc [C0], then
// for each transposed convolution k = 1..5: W_k [C_{k-1}][C_k][4][4][4],
// b_k [C_k] with C_5 = 25.  Everything runs on CUDA cores in float32: a forward
// is ~1 GFLOP at the default widths, small beside a training step.
//
// Transposed convolution, per axis: output u = 2 i - 1 + k (k = 0..3), so output
// u gathers input i = t (tap k = u + 1 - 2t) and i = t - 1 (tap k + 2), t = (u + 1) / 2.
#include <math.h>
#include <string.h>

#include "render.cuh"

namespace nr {

constexpr int kCnnZ = 256;
constexpr int kCnnOut = kBones + 1;   // 25 channels
constexpr int kCnnRes = 32;
constexpr float kSlope = 0.2f;

__device__ __forceinline__ float leaky(float v) { return v > 0.f ? v : kSlope * v; }
__device__ __forceinline__ float leaky_grad(float post) { return post > 0.f ? 1.f : kSlope; }

// the two (input index, tap) pairs feeding output coordinate u of an axis with r inputs
__device__ __forceinline__ void taps(int u, int r, int *i, int *k) {
  const int t = (u + 1) >> 1;
  i[0] = t;
  k[0] = u + 1 - 2 * t;
  i[1] = t - 1;
  k[1] = k[0] + 2;
  if (i[0] >= r) i[0] = -1;
  if (i[1] < 0) i[1] = -1;
}

__global__ void cnn_fc_fwd(const float *__restrict__ W, const float *__restrict__ b, const float *__restrict__ z,
                           int C0, float *__restrict__ h) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= C0) return;
  float a = b[o];
#pragma unroll 32
  for (int k = 0; k < kCnnZ; ++k) a = fmaf(W[(size_t)o * kCnnZ + k], z[k], a);
  h[o] = leaky(a);
}

// out[o][u] = b[o] + sum_i sum_taps in[i][tap] W[i][o][k(tap)]: `split` consecutive lanes per
// output (a power of two up to 32), lane j taking inputs i = j, j + split, ... and the group
// summing over shuffles, so that the first layers' few outputs still fill the GPU
__global__ void __launch_bounds__(256) cnn_convt_fwd(const float *__restrict__ in, const float *__restrict__ W,
                                                     const float *__restrict__ b, int Cin, int Cout, int r,
                                                     int act, int split, float *__restrict__ out) {
  const int R = 2 * r;
  const size_t n = (size_t)Cout * R * R * R;
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t idx = t / split;
  const int j = (int)(t % split);
  const bool valid = idx < n;
  float acc = 0.f;
  if (valid) {
    const int x = (int)(idx % R), y = (int)((idx / R) % R), zz = (int)((idx / ((size_t)R * R)) % R);
    const int o = (int)(idx / ((size_t)R * R * R));
    int iz[2], kz[2], iy[2], ky[2], ix[2], kx[2];
    taps(zz, r, iz, kz);
    taps(y, r, iy, ky);
    taps(x, r, ix, kx);
    const size_t r3 = (size_t)r * r * r;
    for (int i = j; i < Cin; i += split) {
      const float *wi = W + ((size_t)i * Cout + o) * 64;
      const float *xi = in + (size_t)i * r3;
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        if (iz[a] < 0) continue;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (iy[c] < 0) continue;
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            if (ix[e] < 0) continue;
            acc = fmaf(xi[((size_t)iz[a] * r + iy[c]) * r + ix[e]], wi[(kz[a] * 4 + ky[c]) * 4 + kx[e]], acc);
          }
        }
      }
    }
  }
  for (int off = split >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (valid && j == 0) {
    acc += b[idx / ((size_t)R * R * R)];
    out[idx] = act ? leaky(acc) : acc;
  }
}

// The same for a layer wide enough to give every thread its own sums (split 1): kFwdOut outputs at
// one position.  The eight output parities (blockIdx.z) take different taps and one class of a
// block shares them, so its weights come from shared memory as broadcasts (two 16-byte loads per
// output and input) and its inputs are read coalesced, once for the kFwdOut outputs; a thread per
// output read two values from L1 for each multiply-add.  Each sum runs over the inputs and taps in
// the order of cnn_convt_fwd, so the volume keeps its bits.  0.37 and 0.45 ms for the last two
// layers before, 0.17 for both now.  A tap outside the input is a product with zero (as in the
// gradients below): weights are finite when they are installed, and one that has become infinite
// since makes the rim NaN along with the voxels that it reaches.
constexpr int kFwdOut = 4, kFwdIn = 16, kFwdThreads = 128;
__global__ void __launch_bounds__(kFwdThreads) cnn_convt_fwd_wide(const float *__restrict__ in,
                                                                  const float *__restrict__ W,
                                                                  const float *__restrict__ b, int Cin, int Cout,
                                                                  int r, int act, float *__restrict__ out) {
  __shared__ float4 sw[kFwdIn * kFwdOut * 2];
  const int par[3] = {(int)(blockIdx.z >> 2), (int)(blockIdx.z >> 1) & 1, (int)blockIdx.z & 1};   // of z, y, x
  const int r3 = r * r * r, m = blockIdx.x * kFwdThreads + threadIdx.x, o0 = blockIdx.y * kFwdOut;
  const bool valid = m < r3;
  const int mx = m % r, my = (m / r) % r, mz = m / (r * r);
  // tap a of an axis: input m + parity - a, kernel index (parity ? 0 : 1) + 2 a
  int at[8];
  bool ok[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const int z = mz + par[0] - (t >> 2), y = my + par[1] - ((t >> 1) & 1), x = mx + par[2] - (t & 1);
    ok[t] = valid && z >= 0 && y >= 0 && x >= 0 && z < r && y < r && x < r;
    at[t] = ok[t] ? (z * r + y) * r + x : 0;
  }
  float acc[kFwdOut] = {};
  for (int i0 = 0; i0 < Cin; i0 += kFwdIn) {
    __syncthreads();
    for (int e = threadIdx.x; e < kFwdIn * kFwdOut * 8; e += kFwdThreads) {
      const int t = e & 7, oc = (e >> 3) % kFwdOut, i = i0 + e / (8 * kFwdOut);
      const int kz = (par[0] ? 0 : 1) + 2 * (t >> 2), ky = (par[1] ? 0 : 1) + 2 * ((t >> 1) & 1),
                kx = (par[2] ? 0 : 1) + 2 * (t & 1);
      reinterpret_cast<float *>(sw)[e] =
          i < Cin && o0 + oc < Cout ? __ldg(W + ((size_t)i * Cout + o0 + oc) * 64 + (kz * 4 + ky) * 4 + kx) : 0.f;
    }
    __syncthreads();
    const int ni = min(kFwdIn, Cin - i0);
#pragma unroll 2
    for (int ic = 0; ic < ni; ++ic) {
      const float *xi = in + (size_t)(i0 + ic) * r3;
      float x[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) x[t] = ok[t] ? __ldg(xi + at[t]) : 0.f;
#pragma unroll
      for (int oc = 0; oc < kFwdOut; ++oc) {
        const float4 u = sw[(ic * kFwdOut + oc) * 2], v = sw[(ic * kFwdOut + oc) * 2 + 1];
        const float w[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
        for (int t = 0; t < 8; ++t) acc[oc] = fmaf(x[t], w[t], acc[oc]);
      }
    }
  }
  if (!valid) return;
  const int R = 2 * r;
  const size_t u = ((size_t)(2 * mz + par[0]) * R + 2 * my + par[1]) * R + 2 * mx + par[2];
#pragma unroll
  for (int oc = 0; oc < kFwdOut; ++oc)
    if (o0 + oc < Cout) {
      const float v = acc[oc] + b[o0 + oc];
      out[(size_t)(o0 + oc) * R * R * R + u] = act ? leaky(v) : v;
    }
}

// W^c[c][v] = softmax_c(logit[c][v] + log_prior[c][v])
__global__ void cnn_softmax_fwd(const float *__restrict__ logit, const float *__restrict__ log_prior, int V,
                                float *__restrict__ w) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= V) return;
  float m = -INFINITY, a[kCnnOut];
#pragma unroll
  for (int c = 0; c < kCnnOut; ++c) {
    a[c] = logit[(size_t)c * V + v] + (log_prior ? log_prior[(size_t)c * V + v] : 0.f);
    m = fmaxf(m, a[c]);
  }
  float s = 0.f;
#pragma unroll
  for (int c = 0; c < kCnnOut; ++c) {
    a[c] = expf(a[c] - m);
    s += a[c];
  }
  const float inv = 1.f / s;
#pragma unroll
  for (int c = 0; c < kCnnOut; ++c) w[(size_t)c * V + v] = a[c] * inv;
}

// dlogit[c][v] = w[c][v] (g[c][v] - sum_c' w[c'][v] g[c'][v])
__global__ void cnn_softmax_bwd(const float *__restrict__ w, const float *__restrict__ g, int V,
                                float *__restrict__ dlogit) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= V) return;
  float dot = 0.f;
#pragma unroll
  for (int c = 0; c < kCnnOut; ++c) dot = fmaf(w[(size_t)c * V + v], g[(size_t)c * V + v], dot);
#pragma unroll
  for (int c = 0; c < kCnnOut; ++c) {
    const size_t e = (size_t)c * V + v;
    dlogit[e] = w[e] * (g[e] - dot);
  }
}

// din[i][q] = leaky'(in[i][q]) sum_o sum_k W[i][o][k] dout[o][2 q - 1 + k].
//
// r >= 8: a block takes 64 positions and four inputs, its four pairs of warps every fourth output;
// a thread's 64 dout values of an output serve the four inputs, whose weights come from shared
// memory as broadcasts.  (One group of lanes per input value, each reading its own weight rows and
// window, took 0.17 and 0.22 ms for the two layers; 0.17 for both now.)
constexpr int kBackIn = 4;
__global__ void __launch_bounds__(256) cnn_convt_bwd_data_wide(const float *__restrict__ in, const float *__restrict__ W,
                                                               const float *__restrict__ dout, int Cin, int Cout, int r,
                                                               float *__restrict__ din) {
  __shared__ float4 sw[4][kBackIn][16];
  __shared__ float red[4][kBackIn][64];
  const int part = threadIdx.x >> 6, p = threadIdx.x & 63, q = blockIdx.x * 64 + p, i0 = blockIdx.y * kBackIn;
  const int x = q % r, y = (q / r) % r, z = q / (r * r), R = 2 * r;
  const size_t R3 = (size_t)R * R * R;
  float acc[kBackIn] = {};
  for (int o0 = 0; o0 < Cout; o0 += 4) {
    __syncthreads();
    for (int e = threadIdx.x; e < 4 * kBackIn * 64; e += 256) {
      const int k = e & 63, i = i0 + ((e >> 6) % kBackIn), o = o0 + e / (64 * kBackIn);
      reinterpret_cast<float *>(sw)[e] = i < Cin && o < Cout ? __ldg(W + ((size_t)i * Cout + o) * 64 + k) : 0.f;
    }
    __syncthreads();
    const int o = o0 + part;
    if (o >= Cout) continue;
    const float *go = dout + (size_t)o * R3;
#pragma unroll
    for (int kz = 0; kz < 4; ++kz) {
      const int uz = 2 * z - 1 + kz;
#pragma unroll
      for (int ky = 0; ky < 4; ++ky) {
        const int uy = 2 * y - 1 + ky;
        const bool row = uz >= 0 && uz < R && uy >= 0 && uy < R;
        const float *gr = go + ((ptrdiff_t)uz * R + uy) * R;
        float g[4];
#pragma unroll
        for (int kx = 0; kx < 4; ++kx) {
          const int ux = 2 * x - 1 + kx;
          g[kx] = row && ux >= 0 && ux < R ? __ldg(gr + ux) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < kBackIn; ++i) {
          const float4 w = sw[part][i][kz * 4 + ky];
          acc[i] = fmaf(w.x, g[0], fmaf(w.y, g[1], fmaf(w.z, g[2], fmaf(w.w, g[3], acc[i]))));
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kBackIn; ++i) red[part][i][p] = acc[i];
  __syncthreads();
  const int i = i0 + part;   // pair of warps `part` finishes input i0 + part
  static_assert(kBackIn == 4, "one input per pair of warps");
  if (i < Cin) {
    const size_t at = (size_t)i * r * r * r + q;
    din[at] = ((red[0][part][p] + red[1][part][p]) + (red[2][part][p] + red[3][part][p])) * leaky_grad(in[at]);
  }
}

// r = 1: an input sees the eight outputs through the inner taps (1 and 2 of each axis); the outer
// taps reach nothing and their weights are not read.  `split` lanes per input (outputs o = j,
// j + split, ...), summed over shuffles.  0.025 ms for 1024 x 512 channels (0.053 as below).
__global__ void __launch_bounds__(256) cnn_convt_bwd_data_first(const float *__restrict__ in, const float *__restrict__ W,
                                                                const float *__restrict__ dout, int Cin, int Cout,
                                                                int split, float *__restrict__ din) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, i = t / split, j = t % split;
  float acc = 0.f;
  if (i < Cin)
    for (int o = j; o < Cout; o += split) {
      const float *wi = W + ((size_t)i * Cout + o) * 64, *go = dout + (size_t)o * 8;
#pragma unroll
      for (int u = 0; u < 8; ++u) acc = fmaf(wi[((u >> 2) + 1) * 16 + (((u >> 1) & 1) + 1) * 4 + (u & 1) + 1], go[u], acc);
    }
  for (int off = split >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (i < Cin && j == 0) din[i] = acc * leaky_grad(in[i]);
}

// r = 2, 4: a block takes one input channel with every position in its registers.  Its threads
// are the 64 taps by four outputs, so the weights, the larger operand here, are read once and
// coalesced; the outputs' gradients lie in shared memory with a rim of zeros.  r = 4: 0.39 -> 0.16 ms,
// r = 2: 0.22 -> 0.10.
template <int r>
__global__ void __launch_bounds__(256) cnn_convt_bwd_data_deep(const float *__restrict__ in, const float *__restrict__ W,
                                                               const float *__restrict__ dout, int Cout,
                                                               float *__restrict__ din) {
  constexpr int R = 2 * r, P = R + 2, R3 = R * R * R, P3 = P * P * P, r3 = r * r * r, OCH = r == 4 ? 4 : 16;
  __shared__ float pad[OCH * P3];
  __shared__ float red[8][r3];
  const int i = blockIdx.x, k = threadIdx.x & 63, kx = k & 3, ky = (k >> 2) & 3, kz = k >> 4;
  const float *Wi = W + (size_t)i * Cout * 64 + k;
  float acc[r3] = {};
  for (int o0 = 0; o0 < Cout; o0 += OCH) {
    float w[OCH / 4];
#pragma unroll
    for (int j = 0; j < OCH / 4; ++j) {
      const int o = o0 + (threadIdx.x >> 6) + 4 * j;
      w[j] = o < Cout ? __ldg(Wi + (size_t)o * 64) : 0.f;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < OCH * P3; e += 256) {
      const int o = o0 + e / P3, c = e % P3, ux = c % P - 1, uy = (c / P) % P - 1, uz = c / (P * P) - 1;
      pad[e] = o < Cout && ux >= 0 && ux < R && uy >= 0 && uy < R && uz >= 0 && uz < R
                   ? __ldg(dout + (size_t)o * R3 + (uz * R + uy) * R + ux)
                   : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < OCH / 4; ++j) {
      const float *g = pad + ((threadIdx.x >> 6) + 4 * j) * P3 + (kz * P + ky) * P + kx;
#pragma unroll
      for (int q = 0; q < r3; ++q)
        acc[q] = fmaf(w[j], g[(2 * (q / (r * r)) * P + 2 * ((q / r) % r)) * P + 2 * (q % r)], acc[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < r3; ++q) {
    float v = acc[q];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][q] = v;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < r3; q += 256) {
    float v = 0.f;
#pragma unroll
    for (int wp = 0; wp < 8; ++wp) v += red[wp][q];
    din[(size_t)i * r3 + q] = v * leaky_grad(in[(size_t)i * r3 + q]);
  }
}

// dW[i][o][k] = sum_q in[i][q] dout[o][2 q - 1 + k].
//
// r >= 4: a block takes one output and eight inputs; its threads are the 64 taps by slices of the
// planes of q.  A dout value serves the eight inputs, whose values are the same for all taps
// (16-byte broadcasts).  (A thread per weight took 0.43 ms for the last layer's 102,400 and
// 0.71 for the three; 0.34 now.)
constexpr int kWgIn = 8;
__global__ void __launch_bounds__(512) cnn_convt_bwd_weight_wide(const float *__restrict__ in,
                                                                 const float *__restrict__ dout, int Cin, int Cout,
                                                                 int r, int aligned, float *__restrict__ dW) {
  __shared__ float red[8][kWgIn][64];
  const int k = threadIdx.x & 63, slice = threadIdx.x >> 6, slices = blockDim.x >> 6;
  const int kx = k & 3, ky = (k >> 2) & 3, kz = k >> 4, o = blockIdx.x, i0 = blockIdx.y * kWgIn, R = 2 * r;
  const size_t r3 = (size_t)r * r * r;
  const float *go = dout + (size_t)o * R * R * R;
  float acc[kWgIn] = {};
  for (int z = slice; z < r; z += slices) {
    const int uz = 2 * z - 1 + kz;
    if (uz < 0 || uz >= R) continue;
    for (int y = 0; y < r; ++y) {
      const int uy = 2 * y - 1 + ky;
      const bool row = uy >= 0 && uy < R;
      const float *gr = go + ((ptrdiff_t)uz * R + uy) * R;
      for (int x = 0; x < r; x += 4) {
        float g[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int ux = 2 * (x + e) - 1 + kx;
          g[e] = row && ux >= 0 && ux < R ? __ldg(gr + ux) : 0.f;
        }
        const float *xi = in + (size_t)i0 * r3 + (z * r + y) * r + x;
#pragma unroll
        for (int i = 0; i < kWgIn; ++i) {
          if (i0 + i >= Cin) break;
          float4 v;
          if (aligned) {
            v = __ldg(reinterpret_cast<const float4 *>(xi + i * r3));
          } else {
            v = make_float4(__ldg(xi + i * r3), __ldg(xi + i * r3 + 1), __ldg(xi + i * r3 + 2), __ldg(xi + i * r3 + 3));
          }
          acc[i] = fmaf(v.x, g[0], fmaf(v.y, g[1], fmaf(v.z, g[2], fmaf(v.w, g[3], acc[i]))));
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kWgIn; ++i) red[slice][i][k] = acc[i];
  __syncthreads();
  for (int e = threadIdx.x; e < kWgIn * 64; e += blockDim.x) {
    const int i = e >> 6;
    if (i0 + i >= Cin) break;
    float v = 0.f;
    for (int sl = 0; sl < slices; ++sl) v += red[sl][i][e & 63];
    dW[((size_t)(i0 + i) * Cout + o) * 64 + (e & 63)] = v;
  }
}

// r = 1, 2: few positions and many weights, so the kernel is the store of dW: a thread per tap
// row of an output (four weights), a grid row per input, no division (0.27 ms for both, 0.07 now).
__global__ void __launch_bounds__(256) cnn_convt_bwd_weight_deep(const float *__restrict__ in,
                                                                 const float *__restrict__ dout, int Cout, int r,
                                                                 int aligned, float *__restrict__ dW) {
  const int t = blockIdx.x * 256 + threadIdx.x, o = t >> 4, ky = t & 3, kz = (t >> 2) & 3, i = blockIdx.y, R = 2 * r;
  if (o >= Cout) return;
  const float *xi = in + (size_t)i * r * r * r;
  const float *go = dout + (size_t)o * R * R * R;
  float acc[4] = {};
  for (int z = 0; z < r; ++z) {
    const int uz = 2 * z - 1 + kz;
    if (uz < 0 || uz >= R) continue;
    for (int y = 0; y < r; ++y) {
      const int uy = 2 * y - 1 + ky;
      if (uy < 0 || uy >= R) continue;
      for (int x = 0; x < r; ++x) {
        const float v = __ldg(xi + (z * r + y) * r + x);
#pragma unroll
        for (int kx = 0; kx < 4; ++kx) {
          const int ux = 2 * x - 1 + kx;
          if (ux >= 0 && ux < R) acc[kx] = fmaf(v, __ldg(go + (uz * R + uy) * R + ux), acc[kx]);
        }
      }
    }
  }
  float *d = dW + ((size_t)i * Cout + o) * 64 + (kz * 4 + ky) * 4;
  if (aligned) {
    *reinterpret_cast<float4 *>(d) = make_float4(acc[0], acc[1], acc[2], acc[3]);
  } else {
#pragma unroll
    for (int kx = 0; kx < 4; ++kx) d[kx] = acc[kx];
  }
}

// db[o] = sum_u dout[o][u]: one block per channel (up to 1024 threads)
__global__ void __launch_bounds__(1024) cnn_bias_grad(const float *__restrict__ dout, int n_per,
                                                      float *__restrict__ db) {
  __shared__ float red[1024];
  const int o = blockIdx.x;
  float a = 0.f;
  for (int u = threadIdx.x; u < n_per; u += blockDim.x) a += dout[(size_t)o * n_per + u];
  red[threadIdx.x] = a;
  __syncthreads();
  for (int sft = blockDim.x / 2; sft > 0; sft >>= 1) {
    if ((int)threadIdx.x < sft) red[threadIdx.x] += red[threadIdx.x + sft];
    __syncthreads();
  }
  if (threadIdx.x == 0) db[o] = red[0];
}

// fully-connected layer: dW_fc[o][k] = dh[o] z[k], db_fc = dh (dh already through leaky')
__global__ void cnn_fc_bwd(const float *__restrict__ dh, const float *__restrict__ z, int C0, float *__restrict__ dW,
                           float *__restrict__ db) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)C0 * kCnnZ) return;
  const int o = (int)(idx / kCnnZ), k = (int)(idx % kCnnZ);
  dW[idx] = dh[o] * z[k];
  if (k == 0) db[o] = dh[o];
}

struct CnnLayout {
  size_t w[6], b[6];      // offsets of W and b of the fc layer (0) and convolutions 1..5
  int cin[6], cout[6], r[6];   // input channels, output channels, input resolution
  size_t act[6];          // offsets of each layer's output in the activation buffer
  size_t n_params, n_act, max_grad;
};

static CnnLayout cnn_layout(const uint32_t *ch) {
  CnnLayout L{};
  size_t o = 0;
  L.cin[0] = kCnnZ;
  L.cout[0] = (int)ch[0];
  L.r[0] = 1;
  L.w[0] = o;
  o += (size_t)ch[0] * kCnnZ;
  L.b[0] = o;
  o += ch[0];
  int r = 1;
  for (int k = 1; k <= 5; ++k) {
    L.cin[k] = (int)ch[k - 1];
    L.cout[k] = k < 5 ? (int)ch[k] : kCnnOut;
    L.r[k] = r;
    L.w[k] = o;
    o += (size_t)L.cin[k] * L.cout[k] * 64;
    L.b[k] = o;
    o += L.cout[k];
    r *= 2;
  }
  L.n_params = o;
  size_t a = 0, mg = 0;
  for (int k = 0; k <= 5; ++k) {
    const size_t rr = (size_t)(k == 0 ? 1 : 2 * L.r[k]);
    const size_t n = (size_t)L.cout[k] * rr * rr * rr;
    L.act[k] = a;
    a += n;
    mg = std::max(mg, n);
  }
  L.n_act = a;
  L.max_grad = mg;
  return L;
}

static unsigned blocks_for(size_t n) { return (unsigned)((n + 255) / 256); }

// Lanes per output of a layer with n outputs, each a sum over `terms` inputs (or outputs): enough
// that the launch reaches ~2^18 threads, at most 32 and no more than the terms.
static int cnn_split(size_t n, int terms) {
  int sp = 1;
  while (sp < 32 && sp < terms && n * (size_t)sp < (size_t(1) << 18)) sp *= 2;
  return sp;
}

// W^c = CNN_skel(z) into s->wvol; keeps the activations for the backward.
nr_status cnn_forward(nr_subject *s, cudaStream_t st) {
  const CnnLayout L = cnn_layout(s->cnn_ch);
  float *A = s->cnn_act;
  cnn_fc_fwd<<<blocks_for(L.cout[0]), 256, 0, st>>>(s->cnn + L.w[0], s->cnn + L.b[0], s->cnn_z, L.cout[0],
                                                     A + L.act[0]);
  for (int k = 1; k <= 5; ++k) {
    const size_t R = 2 * (size_t)L.r[k];
    const size_t nout = (size_t)L.cout[k] * R * R * R;
    const int sp = cnn_split(nout, L.cin[k]);
    if (sp == 1) {   // enough outputs for a thread to own whole sums
      const int r3 = L.r[k] * L.r[k] * L.r[k];
      cnn_convt_fwd_wide<<<dim3((r3 + kFwdThreads - 1) / kFwdThreads, (L.cout[k] + kFwdOut - 1) / kFwdOut, 8),
                           kFwdThreads, 0, st>>>(A + L.act[k - 1], s->cnn + L.w[k], s->cnn + L.b[k], L.cin[k],
                                                 L.cout[k], L.r[k], k < 5 ? 1 : 0, A + L.act[k]);
      continue;
    }
    cnn_convt_fwd<<<blocks_for(nout * sp), 256, 0, st>>>(A + L.act[k - 1], s->cnn + L.w[k], s->cnn + L.b[k],
                                                         L.cin[k], L.cout[k], L.r[k], k < 5 ? 1 : 0, sp,
                                                         A + L.act[k]);
  }
  const int V = kCnnRes * kCnnRes * kCnnRes;
  cnn_softmax_fwd<<<blocks_for(V), 256, 0, st>>>(A + L.act[5], s->cnn_prior, V, s->wvol);
  NR_CHECK_CUDA(cudaGetLastError());
  count_launches(7);
  return NR_OK;
}

// dL/dtheta_cnn into s->g_cnn from dL/dW^c in s->g_wvol (the forward's activations and
// s->wvol must be those of the current parameters).
nr_status cnn_backward(nr_subject *s, cudaStream_t st) {
  const CnnLayout L = cnn_layout(s->cnn_ch);
  const float *A = s->cnn_act;
  float *d0 = s->cnn_grad, *d1 = s->cnn_grad + L.max_grad;
  const int V = kCnnRes * kCnnRes * kCnnRes;
  cnn_softmax_bwd<<<blocks_for(V), 256, 0, st>>>(s->wvol, s->g_wvol, V, d0);
  int launched = 1;
  for (int k = 5; k >= 1; --k) {
    const size_t R = 2 * (size_t)L.r[k];
    const size_t nout = R * R * R;
    const float *x = A + L.act[k - 1], *w = s->cnn + L.w[k];
    float *gw = s->g_cnn + L.w[k];
    const int r = L.r[k], cin = L.cin[k], cout = L.cout[k];
    if (r >= 4)
      cnn_convt_bwd_weight_wide<<<dim3(cout, (cin + kWgIn - 1) / kWgIn), 64 * std::min(r, 8), 0, st>>>(
          x, d0, cin, cout, r, ((uintptr_t)x & 15) == 0, gw);
    else
      cnn_convt_bwd_weight_deep<<<dim3((cout * 16 + 255) / 256, cin), 256, 0, st>>>(x, d0, cout, r,
                                                                                    ((uintptr_t)gw & 15) == 0, gw);
    cnn_bias_grad<<<cout, nout >= 4096 ? 1024 : 256, 0, st>>>(d0, (int)nout, s->g_cnn + L.b[k]);
    if (r >= 8)
      cnn_convt_bwd_data_wide<<<dim3(r * r * r / 64, (cin + kBackIn - 1) / kBackIn), 256, 0, st>>>(x, w, d0, cin, cout,
                                                                                                  r, d1);
    else if (r == 4)
      cnn_convt_bwd_data_deep<4><<<cin, 256, 0, st>>>(x, w, d0, cout, d1);
    else if (r == 2)
      cnn_convt_bwd_data_deep<2><<<cin, 256, 0, st>>>(x, w, d0, cout, d1);
    else {
      const int sp = cnn_split(cin, cout);
      cnn_convt_bwd_data_first<<<blocks_for((size_t)cin * sp), 256, 0, st>>>(x, w, d0, cin, cout, sp, d1);
    }
    std::swap(d0, d1);
    launched += 3;
  }
  cnn_fc_bwd<<<blocks_for((size_t)L.cout[0] * kCnnZ), 256, 0, st>>>(d0, s->cnn_z, L.cout[0], s->g_cnn + L.w[0],
                                                                     s->g_cnn + L.b[0]);
  NR_CHECK_CUDA(cudaGetLastError());
  count_launches(launched + 1);
  return NR_OK;
}

size_t cnn_param_count(const uint32_t *ch) { return cnn_layout(ch).n_params; }

}  // namespace nr

using namespace nr;

extern "C" nr_status nr_set_weight_cnn(nr_subject *s, const uint32_t *channels, const float *params, const float *z,
                                       const float *log_prior, void *stream) {
  NR_REQUIRE(subject_ok(s), "nr_set_weight_cnn: invalid handle");
  NR_CHECK_CUDA(cudaSetDevice(s->device));
  cudaStream_t st = (cudaStream_t)stream;
  if (!params) {   // back to the directly stored volume (it keeps the last generated values)
    s->cnn_on = false;
    return NR_OK;
  }
  NR_REQUIRE(channels && z, "nr_set_weight_cnn: NULL channels or z");
  NR_REQUIRE(s->wres == (uint32_t)kCnnRes, "nr_set_weight_cnn: the subject's weight volume must be 32^3");
  for (int k = 0; k < 5; ++k)
    NR_REQUIRE(channels[k] >= 1 && channels[k] <= 4096, "nr_set_weight_cnn: channels[%d] must be 1..4096", k);
  const CnnLayout L = cnn_layout(channels);
  for (size_t i = 0; i < L.n_params; ++i)
    NR_REQUIRE(isfinite(params[i]), "nr_set_weight_cnn: non-finite weight %zu", i);
  float *bufs[] = {s->cnn, s->g_cnn, s->cnn_m, s->cnn_v, s->cnn_z, s->cnn_prior, s->cnn_act, s->cnn_grad};
  for (float *b : bufs)
    if (b) cudaFree(b);
  s->cnn = s->g_cnn = s->cnn_m = s->cnn_v = s->cnn_z = s->cnn_prior = s->cnn_act = s->cnn_grad = nullptr;
  s->cnn_on = false;
  s->n_cnn = 0;
  const size_t V = (size_t)kCnnRes * kCnnRes * kCnnRes;
  NR_CHECK_CUDA(cudaMalloc(&s->cnn, L.n_params * 4));
  NR_CHECK_CUDA(cudaMalloc(&s->g_cnn, L.n_params * 4));
  NR_CHECK_CUDA(cudaMalloc(&s->cnn_m, L.n_params * 4));
  NR_CHECK_CUDA(cudaMalloc(&s->cnn_v, L.n_params * 4));
  NR_CHECK_CUDA(cudaMalloc(&s->cnn_z, kCnnZ * 4));
  NR_CHECK_CUDA(cudaMalloc(&s->cnn_act, L.n_act * 4));
  NR_CHECK_CUDA(cudaMalloc(&s->cnn_grad, 2 * L.max_grad * 4));
  if (log_prior) NR_CHECK_CUDA(cudaMalloc(&s->cnn_prior, kCnnOut * V * 4));
  NR_CHECK_CUDA(cudaMemcpyAsync(s->cnn, params, L.n_params * 4, cudaMemcpyHostToDevice, st));
  NR_CHECK_CUDA(cudaMemcpyAsync(s->cnn_z, z, kCnnZ * 4, cudaMemcpyHostToDevice, st));
  if (log_prior) NR_CHECK_CUDA(cudaMemcpyAsync(s->cnn_prior, log_prior, kCnnOut * V * 4, cudaMemcpyHostToDevice, st));
  NR_CHECK_CUDA(cudaMemsetAsync(s->g_cnn, 0, L.n_params * 4, st));
  NR_CHECK_CUDA(cudaMemsetAsync(s->cnn_m, 0, L.n_params * 4, st));
  NR_CHECK_CUDA(cudaMemsetAsync(s->cnn_v, 0, L.n_params * 4, st));
  NR_CHECK_CUDA(cudaStreamSynchronize(st));   // the host arrays may be freed on return
  memcpy(s->cnn_ch, channels, sizeof(s->cnn_ch));
  s->n_cnn = L.n_params;
  s->cnn_t = 0;
  s->cnn_on = true;
  s->cnn_dirty = true;
  return NR_OK;
}

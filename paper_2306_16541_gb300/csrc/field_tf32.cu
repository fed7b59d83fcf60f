// field_tf32.cu -- the float32 tier on the tensor cores: the per-sample field (render and
// query modes) with both MLPs as warp-level layers at float32 accuracy (three TF32 products
// per step, tf32.cuh) instead of CUDA-core FMAs.
//
// Work split: each warp owns a tile of 32 samples.  The gathers (inverse-LBS warp, PE, hash
// encoding) run one sample per lane in float32 as in the CUDA-core kernel; every layer reads the
// tile in shared memory and leaves its output there (frag_fwd).  gamma(x_skel), which layers 1
// and 4 both see, waits in the warp's image in global memory in between (5 KB, L1/L2 resident).
#include "field.cuh"
#include "render.cuh"
#include "tf32.cuh"

namespace nr {

static_assert(kGamRows == kTf32Rows, "scratch rows");

template <int MODE>
__global__ void __launch_bounds__(kTf32Threads, 1) field_tf32_kernel(FieldParams P, FragLay W,
                                                                     const float4 *__restrict__ in, uint32_t n_fixed,
                                                                     const uint32_t *__restrict__ n_dev,
                                                                     float *__restrict__ out) {
  extern __shared__ float4 smem4[];
  float *sW = reinterpret_cast<float *>(smem4);
  float *sG = sW + W.total;                        // pose (and support boxes)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float *xt = sG + kPoseSmem + warp * kTileFloats;
  stage_frag_weights(P.blob, P.lay, W, P.hidden, sW);
  const float *sBox = stage_pose(P, sG, threadIdx.x, blockDim.x);
  __syncthreads();

  const FragLane L = frag_lane();
  const int warps = blockDim.x >> 5;
  float *img = P.tf32_scratch + ((size_t)blockIdx.x * warps + warp) * kGamRows * kTileRow;
  const int eb = (2 * P.L + 7) >> 3;               // blocks of inputs that hold features
  auto put = [=](int k, float v) {
    if (k < kGamRows) xt[frag_at(k, lane)] = v;
  };
  const uint32_t n = n_dev ? *n_dev : n_fixed;
  const uint32_t n_tiles = (n + 31) / 32;
  for (uint32_t tile = blockIdx.x * warps + warp; tile < n_tiles; tile += gridDim.x * warps) {
    const uint32_t j = tile * 32 + lane;
    const bool valid = j < n;
    float x0 = 0.f, x1 = 0.f, x2 = 0.f, delta = 0.f;
    if (valid) {
      if (MODE == kModeRender) {
        const float4 s = in[j];
        x0 = s.x;
        x1 = s.y;
        x2 = s.z;
        delta = s.w;
      } else {
        const float *q = reinterpret_cast<const float *>(in) + 3 * (size_t)j;
        x0 = q[0];
        x1 = q[1];
        x2 = q[2];
      }
    }
    float s0, s1, s2, S;
    lbs_warp(P, sG, x0, x1, x2, s0, s1, s2, S, sBox);
    float f0 = s0, f1 = s1, f2 = s2;
    if (MODE == kModeRender && !__any_sync(0xffffffffu, valid && S != 0.f)) {
      // no bone reaches any of the tile's samples: S = 0, alpha = (..) min(S, 1) = 0, and they add
      // nothing to their rays (of a finite field: a NaN shows only on rays that meet a bone)
      if (valid) reinterpret_cast<float4 *>(out)[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      continue;
    }
    float c[2][8][4], o[4];
    if (P.res_enabled) {
      pos_enc(P, s0, s1, s2, put);
      __syncwarp();
      tile_save(xt, img, kGamRows);
      frag_zero(c);
      frag_fwd<8>(L, xt, kGamRows / 8, sW + W.r1, kGamRows / 8, 0, c);
      frag_relu(L, P.bias1, c);
      frag_store<8>(L, c, xt);
#pragma unroll 1
      for (int l = 1; l < 4; ++l) {
        frag_zero(c);
        frag_fwd<8>(L, xt, 8, sW + (l == 1 ? W.r2 : l == 2 ? W.r3 : W.r4), l == 3 ? 8 + kGamRows / 8 : 8, 0, c);
        if (l == 3) {   // layer 4 sees [h3, gamma]
          tile_load(xt, img, kGamRows);
          frag_fwd<8>(L, xt, kGamRows / 8, sW + W.r4, 8 + kGamRows / 8, 8, c);
        }
        frag_relu(L, sW + (l == 1 ? W.r2b : l == 2 ? W.r3b : W.r4b), c);
        frag_store<8>(L, c, xt);
      }
      frag_out4(L, xt, sW + W.r5, sW + W.r5b, o);
      f0 += o[0];
      f1 += o[1];
      f2 += o[2];
    }
    const bool inside = hash_encode(P, f0, f1, f2, put);
    __syncwarp();
#pragma unroll 1
    for (int l = 0; l < P.hidden; ++l) {
      frag_zero(c);
      frag_fwd<8>(L, xt, l ? 8 : eb, sW + (l ? W.ch[l - 1] : W.c0), l ? 8 : kMlpIn / 8, 0, c);
      frag_relu(L, sW + (l ? W.chb[l - 1] : W.c0b), c);
      frag_store<8>(L, c, xt);
    }
    frag_out4(L, xt, sW + W.cl, sW + W.clb, o);
    if (valid) {
      const float cr = sigmoidf_(o[0]), cg = sigmoidf_(o[1]), cb = sigmoidf_(o[2]), sigma = softplusf_(o[3]);
      if (MODE == kModeRender) {
        const float a = inside ? -expm1f(-sigma * delta) * fminf(S, 1.f) : 0.f;
        reinterpret_cast<float4 *>(out)[j] = make_float4(cr, cg, cb, a);
      } else {
        float *q = out + (size_t)NR_QUERY_STRIDE * j;
        q[0] = s0; q[1] = s1; q[2] = s2; q[3] = S;
        q[4] = f0; q[5] = f1; q[6] = f2; q[7] = inside ? 1.f : 0.f;
        q[8] = cr; q[9] = cg; q[10] = cb; q[11] = sigma;
      }
    }
  }
}

nr_status launch_field_tf32(const FieldParams &P, int mode, const float4 *in, uint32_t n_fixed, const uint32_t *n_dev,
                            float *out, int device, cudaStream_t st) {
  if (!P.tf32_scratch) {
    set_error("the float32 tensor-core tier has no scratch buffer");
    return NR_ESTATE;
  }
  const FragLay W = frag_layout(P.hidden);
  // the warps whose tiles fit beside the weights (sixteen with two hidden layers, eleven with four)
  const size_t base = sizeof(float) * (W.total + kPoseSmem), tile_b = kTileFloats * sizeof(float);
  const int warps = (int)std::min<size_t>(kTf32Threads / 32, (227 * 1024 - base) / tile_b);
  const size_t smem = base + warps * tile_b;
  const int blocks = num_sms(device);
  if (mode == kModeRender) {
    NR_CHECK_CUDA(
        cudaFuncSetAttribute(field_tf32_kernel<kModeRender>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    field_tf32_kernel<kModeRender><<<blocks, 32 * warps, smem, st>>>(P, W, in, n_fixed, n_dev, out);
  } else {
    NR_CHECK_CUDA(
        cudaFuncSetAttribute(field_tf32_kernel<kModeQuery>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    field_tf32_kernel<kModeQuery><<<blocks, 32 * warps, smem, st>>>(P, W, in, n_fixed, n_dev, out);
  }
  NR_CHECK_CUDA(cudaGetLastError());
  return NR_OK;
}

}  // namespace nr

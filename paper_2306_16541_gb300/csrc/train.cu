// train.cu -- one training step (Sec. 5.2): stratified samples of a batch of
// pixel rays, the float32 field forward, compositing with the squared-error
// loss (or a caller's dL/dC), the hand-written backward (compositing adjoint,
// canonical MLP, hash scatter-add, residual MLP through the positional
// encoding, inverse-LBS scatter-add into the weight volume, and the pose
// refiner's dL/dG) and Adam.
//
// Work split:
//   * a warp takes 32 samples.  The gathers and their adjoints (LBS warp, PE, hash encoding) run
//     one sample per lane; the layer at hand -- an activation in the forward, a delta in the
//     backward -- lies in the warp's shared-memory tile (a row per feature), so both MLPs'
//     forward and backward layers (m16n8k8 TF32 MMAs, three per step for float32 accuracy) touch
//     shared memory and registers only.  Every activation that a weight gradient needs goes once
//     to a per-warp image in global memory, as 16-byte copies of the tile, with the ReLU's sign
//     bits beside it;
//   * weight gradients of a warp go into its block's private accumulator, whole MMA fragments
//     as 16-byte fire-and-forget adds; one kernel sums the block accumulators at the end;
//   * hash-table and weight-volume gradients are scattered with float2 / float atomics straight
//     into the gradient buffers, warp-aggregated: the lanes of a run that adds into one cell sum
//     first (run_sum);
//   * thread slots visit the batch's rays in a scattered order (ray_of), so that the rays in
//     flight together do not come from one image patch;
//   * the forward records which slots carry a gradient (live mask); the backward skips the rest.
#include <math.h>
#include <string.h>

#include "field.cuh"
#include "gather.cuh"
#include "render.cuh"
#include "tf32.cuh"

namespace nr {

// Bound by waits on L2 at the sixteen warps that registers and tiles allow (34 % tensor pipe, 36 %
// issue slots): a 2^18 x 128-sample step takes 132 ms, 230 with the activations in per-thread columns
// of global memory, and 142 with twelve warps of 168 registers.
constexpr int kTrainThreads = 512;   // at most: sixteen warps of 128 registers
constexpr size_t kTrainSmem = 227 * 1024;
constexpr size_t kQuadBytes = 512;

// Rows (of 32 floats) of a warp's global image, sized for the subject's hidden depth H.
struct Rows {
  int gam;     // gamma(x_skel)            kGamRows
  int rh;      // residual h1..h4          4 x 64
  int enc;     // hash encoding            32
  int ch;      // canonical h1..hH         H x 64
  int dgam;    // dL/d gamma               kGamRows
  int sign;    // per hidden layer, a lane's 64 ReLU signs      2 (4 + H)
  int dp;      // dL/d p_i per bone (pose refiner)  3 x 24
  int xs;      // the sample position               3
  int total;
};

static Rows make_rows(int H) {
  Rows r{};
  int o = 0;
  r.gam = o; o += kGamRows;
  r.rh = o; o += 4 * kWidth;
  r.enc = o; o += kMlpIn;
  r.ch = o; o += H * kWidth;
  r.dgam = o; o += kGamRows;
  r.sign = o; o += 2 * (4 + H);
  r.dp = o; o += 3 * kBones;
  r.xs = o; o += 3;
  r.total = o;
  return r;
}

struct TrainDev {
  const uint32_t *frame_id, *px, *py;
  const float *target;
  uint32_t n_rays, S;
  uint32_t ray_mul;       // coprime with n_rays: the order in which thread slots visit rays
  float loss_weight;      // lambda_mse
  uint64_t seed;
  float bg[3];
  const Frame *cams;
  const float *fG, *fbias1, *fomega;
  float4 *samp, *out;
  float *T;
  uint32_t *raycnt;
  uint32_t *live;         // per warp of 32 thread slots: bit l set if slot l's sample has a gradient
  float *loss;
  float2 *g_table;
  float *g_wvol;
  float4 *g_quad;         // corner-block sums of the weight-volume gradient (layout of wquad), or NULL
  float *scratch, *wacc;
  int acc_floats;         // floats per block accumulator
  int n_frames;
  Rows rw;
  float *dG;              // [F][24][12] dL/dG of every frame (pose refiner), or NULL
  int dG_acc;             // 1: the blocks sum dG in their accumulators first, behind the frame biases
  FragLay fl;             // shared-memory layout of the weights
  float *pred;            // [n][3] composited colours out, or NULL
  const float *grad_rgb;  // [n][3] dL/dC from the caller, or NULL (MSE against target)
  int forward_only;       // stop after compositing
};

// The ray whose samples thread slot q (of the fwd/bwd kernels) evaluates: slot q takes
// sample q mod S of ray (q / S) ray_mul mod n_rays.  With ray_mul near 0.618 n_rays the
// rays in flight at one time lie spread over the batch; taken in batch order they would be
// neighbours from one image patch whose scatter-adds all hit the same table entries and
// voxels at once.  Every ray is visited once since ray_mul is coprime with n_rays.
__device__ __forceinline__ uint32_t ray_of(const TrainDev &T, uint32_t q) {
  return (uint32_t)(((uint64_t)(q / T.S) * T.ray_mul) % T.n_rays);
}

// A multiplier coprime with n near the golden-ratio fraction of n (1 for n <= 2).
static uint32_t ray_multiplier(uint32_t n) {
  if (n <= 2) return 1;
  auto gcd = [](uint32_t a, uint32_t b) {
    while (b) {
      const uint32_t t = a % b;
      a = b;
      b = t;
    }
    return a;
  };
  uint32_t m = (uint32_t)(0.6180339887498949 * (double)n);
  if (m < 1) m = 1;
  while (gcd(m, n) != 1) ++m;
  return m;
}

// ----------------------------------------------------------------- rays
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t k) {
  // SplitMix64 (Steele, Lea and Flood 2014): output k of the generator seeded with `seed`
  uint64_t z = seed + k * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// One thread per (ray, bin): stratified sample t_i = lo + (i + u_i) D inside the
// clipped ray, delta_i = t_{i+1} - t_i, delta_{S-1} = hi - t_{S-1}.
__global__ void __launch_bounds__(256) train_samples_kernel(TrainDev T, float bx, float by, float bz, float Bx,
                                                            float By, float Bz) {
  const uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (q >= (uint64_t)T.n_rays * T.S) return;
  const uint32_t r = (uint32_t)(q / T.S), i = (uint32_t)(q % T.S);
  const Frame &F = T.cams[T.frame_id[r]];
  CamParams c;
  for (int k = 0; k < 9; ++k) c.R[k] = F.R[k];
  for (int k = 0; k < 3; ++k) c.t[k] = F.t[k];
  c.fx = F.fx; c.fy = F.fy; c.cx = F.cx; c.cy = F.cy; c.t_near = F.t_near; c.t_far = F.t_far;
  const float bmin[3] = {bx, by, bz}, bmax[3] = {Bx, By, Bz};
  float o[3], d[3], lo, hi;
  camera_origin(c, o);
  const bool hit = ray_setup(c, o, bmin, bmax, T.px[r], T.py[r], d, lo, hi);
  if (i == 0) T.raycnt[r] = hit ? T.S : 0u;
  if (!hit) {
    T.samp[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const float D = (hi - lo) / (float)T.S;
  auto u_of = [&](uint32_t ii) {
    const uint64_t z = splitmix64(T.seed, (uint64_t)r * T.S + ii + 1);
    return (float)(z >> 40) * (1.0f / 16777216.0f);
  };
  const float t = lo + ((float)i + u_of(i)) * D;
  const float tn = (i + 1 < T.S) ? lo + ((float)(i + 1) + u_of(i + 1)) * D : hi;
  T.samp[q] = make_float4(o[0] + t * d[0], o[1] + t * d[1], o[2] + t * d[2], tn - t);
}

// ------------------------------------------------- compositing and its adjoint
// Per ray: C = sum_i T_i alpha_i c_i + T_S bg, T_{i+1} = T_i (1 - alpha_i) (Eq. 3),
// loss term sum_k (C_k - C_gt,k)^2 / (3 N), g = dL/dC.  The reverse scan keeps
// B_i = sum_{j>i} alpha_j prod_{i<k<j}(1 - alpha_k) (c_j . g) + prod_{k>i}(1 - alpha_k) (bg . g)
// (B_{S-1} = bg . g, B_{i-1} = alpha_i (c_i . g) + (1 - alpha_i) B_i) so that
//   dL/dc_i = T_i alpha_i g,  dL/dalpha_i = T_i (c_i . g - B_i)
// without dividing by (1 - alpha_i).
__global__ void __launch_bounds__(256) train_composite_kernel(TrainDev T) {
  const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
  float lsum = 0.f;
  if (r < T.n_rays) {
    const size_t base = (size_t)r * T.S;
    const uint32_t cnt = T.raycnt[r];
    float Tr = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
    for (uint32_t i = 0; i < cnt; ++i) {
      const float4 v = T.out[base + i];
      T.T[base + i] = Tr;
      const float w = Tr * v.w;
      c0 = fmaf(w, v.x, c0);
      c1 = fmaf(w, v.y, c1);
      c2 = fmaf(w, v.z, c2);
      Tr *= 1.f - v.w;
    }
    const float C0 = fmaf(Tr, T.bg[0], c0), C1 = fmaf(Tr, T.bg[1], c1), C2 = fmaf(Tr, T.bg[2], c2);
    if (T.pred) {
      T.pred[3 * r] = C0;
      T.pred[3 * r + 1] = C1;
      T.pred[3 * r + 2] = C2;
    }
    float g0 = 0.f, g1 = 0.f, g2 = 0.f;
    if (T.grad_rgb) {   // the caller's dL/dC
      g0 = T.grad_rgb[3 * r];
      g1 = T.grad_rgb[3 * r + 1];
      g2 = T.grad_rgb[3 * r + 2];
    } else if (T.target) {
      const float e0 = C0 - T.target[3 * r], e1 = C1 - T.target[3 * r + 1], e2 = C2 - T.target[3 * r + 2];
      lsum = T.loss_weight * (e0 * e0 + e1 * e1 + e2 * e2);
      const float scale = 2.f * T.loss_weight / (3.f * (float)T.n_rays);
      g0 = scale * e0;
      g1 = scale * e1;
      g2 = scale * e2;
    }
    float B = T.bg[0] * g0 + T.bg[1] * g1 + T.bg[2] * g2;
    for (int i = T.forward_only ? -1 : (int)cnt - 1; i >= 0; --i) {
      const float4 v = T.out[base + i];
      const float Ti = T.T[base + i];
      const float cg = v.x * g0 + v.y * g1 + v.z * g2;
      const float ta = Ti * v.w;
      T.out[base + i] = make_float4(ta * g0, ta * g1, ta * g2, Ti * (cg - B));
      B = fmaf(v.w, cg, (1.f - v.w) * B);
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
  if ((threadIdx.x & 31) == 0) atomicAdd(T.loss, lsum / (3.f * (float)T.n_rays));
}

// ------------------------------------------------------- warp-aggregated scatter-add
// The samples of a warp lie in order along one ray (or a few, when S is not a multiple of
// 32), so lanes that add into the same cell (hash level cell, weight-volume cell) are runs of
// consecutive lanes.  run_sum sums the
// values of each run into its first lane (a segmented suffix sum over shuffles, stopping
// once no run is longer than the distance reached) and returns whether this lane heads a
// valid run: only head lanes issue the atomics, with the run's totals.  A run is a maximal
// stretch of valid lanes with equal keys (key_lo, key_hi); invalid lanes are runs of their
// own and add nothing.  Every lane of the warp must call it.
template <int NV>
__device__ __forceinline__ bool run_sum(uint32_t key_lo, uint32_t key_hi, bool valid, float (&v)[NV]) {
  const int lane = threadIdx.x & 31;
  const uint32_t plo = __shfl_up_sync(0xffffffffu, key_lo, 1), phi = __shfl_up_sync(0xffffffffu, key_hi, 1);
  const uint32_t vmask = __ballot_sync(0xffffffffu, valid);
  const bool pvalid = lane > 0 && ((vmask >> (lane - 1)) & 1u);
  const bool head = !valid || !pvalid || plo != key_lo || phi != key_hi;
  const uint32_t heads = __ballot_sync(0xffffffffu, head);
  const int run = __popc(heads & (0xffffffffu >> (31 - lane)));   // heads at lanes 0..lane
#pragma unroll 1
  for (int d = 1; d < 32; d <<= 1) {
    const int rd = __shfl_down_sync(0xffffffffu, run, d);
    const bool take = lane + d < 32 && rd == run;
    if (!__any_sync(0xffffffffu, take)) break;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const float o = __shfl_down_sync(0xffffffffu, v[k], d);
      if (take) v[k] += o;
    }
  }
  return head && valid;
}

// ---------------------------------------------------------------- backward
// Where the block accumulators hold dW[o][i] of a layer with 64 outputs: the MMA fragments of
// wgrad64 as they leave the registers, (8-column tile, 16-row tile, lane, value).
__host__ __device__ __forceinline__ int acc_index(int o, int i) {
  return (((i >> 3) * 4 + (o >> 4)) * 32 + (o & 7) * 4 + ((i & 7) >> 1)) * 4 + ((o >> 3) & 1) * 2 + (i & 1);
}

// Warp-level weight gradient of one layer with 64 outputs over the warp's 32 samples,
// dW[j][k] = sum_s d[s][j] h[s][k], as the product D^T H on the tensor cores (m16n8k8 TF32 MMAs,
// three per step for float32 accuracy): M = the 64 outputs in four 16-row tiles, K = the 32
// samples (taken four consecutive ones a lane, so that a fragment is a 16-byte load; the order of
// the sum is free), N = the inputs in nb tiles of 8.  D is the shared tile, H the global image of
// the layer's input.  Each finished 16 x 8 tile is added into the block's accumulator at acc
// (acc_index) as one 16-byte add per lane; the bias gradient sum_s d[s][j] goes to acc_b[j] and,
// when given, to acc_f[j].
__device__ __forceinline__ void wgrad64(const FragLane &L, const float *tile, const float *img, int nb, float *acc,
                                        float *acc_b, float *acc_f) {
  const int lane = threadIdx.x & 31;
  if (acc_b) {
    float s0 = 0.f, s1 = 0.f;
    const int sw = tile_sw(lane);
    const float4 *p0 = reinterpret_cast<const float4 *>(tile + lane * kTileRow);
    const float4 *p1 = reinterpret_cast<const float4 *>(tile + (lane + 32) * kTileRow);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 a = p0[q ^ sw], c = p1[q ^ sw];
      s0 += (a.x + a.y) + (a.z + a.w);
      s1 += (c.x + c.y) + (c.z + c.w);
    }
    atomicAdd(acc_b + lane, s0);
    atomicAdd(acc_b + lane + 32, s1);
    if (acc_f) {
      atomicAdd(acc_f + lane, s0);
      atomicAdd(acc_f + lane + 32, s1);
    }
  }
  const int row = L.g * kTileRow;
  const int at[2] = {row + ((L.t ^ tile_sw(L.g)) << 2), row + (((4 + L.t) ^ tile_sw(L.g)) << 2)};
  // two row tiles of D at a time, so that their hi/lo fragments take 64 registers; H is read once
  // per pair
#pragma unroll 1
  for (int mh = 0; mh < 4; mh += 2) {
    uint32_t ah[2][4][4], al[2][4][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float *d = tile + 16 * (mh + m) * kTileRow + at[j];
        const float4 u = *reinterpret_cast<const float4 *>(d), v = *reinterpret_cast<const float4 *>(d + 8 * kTileRow);
        tf32_split(u.x, ah[m][2 * j][0], al[m][2 * j][0]);
        tf32_split(v.x, ah[m][2 * j][1], al[m][2 * j][1]);
        tf32_split(u.y, ah[m][2 * j][2], al[m][2 * j][2]);
        tf32_split(v.y, ah[m][2 * j][3], al[m][2 * j][3]);
        tf32_split(u.z, ah[m][2 * j + 1][0], al[m][2 * j + 1][0]);
        tf32_split(v.z, ah[m][2 * j + 1][1], al[m][2 * j + 1][1]);
        tf32_split(u.w, ah[m][2 * j + 1][2], al[m][2 * j + 1][2]);
        tf32_split(v.w, ah[m][2 * j + 1][3], al[m][2 * j + 1][3]);
      }
    float4 nx0 = *reinterpret_cast<const float4 *>(img + at[0]), nx1 = *reinterpret_cast<const float4 *>(img + at[1]);
#pragma unroll 1
    for (int n = 0; n < nb; ++n) {
      const float hv[8] = {nx0.x, nx0.y, nx0.z, nx0.w, nx1.x, nx1.y, nx1.z, nx1.w};
      if (n + 1 < nb) {   // the next tile's loads run under this one's products
        const float *h = img + (n + 1) * 8 * kTileRow;
        nx0 = *reinterpret_cast<const float4 *>(h + at[0]);
        nx1 = *reinterpret_cast<const float4 *>(h + at[1]);
      }
      float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        uint32_t bh[2], bl[2];
        tf32_split(hv[2 * ks], bh[0], bl[0]);
        tf32_split(hv[2 * ks + 1], bh[1], bl[1]);
#pragma unroll
        for (int m = 0; m < 2; ++m) mma_tf32(c[m], al[m][ks], bh);
#pragma unroll
        for (int m = 0; m < 2; ++m) mma_tf32(c[m], ah[m][ks], bl);
#pragma unroll
        for (int m = 0; m < 2; ++m) mma_tf32(c[m], ah[m][ks], bh);
      }
#pragma unroll
      for (int m = 0; m < 2; ++m)
        atomicAdd(reinterpret_cast<float4 *>(acc) + (n * 4 + mh + m) * 32 + lane,
                  make_float4(c[m][0], c[m][1], c[m][2], c[m][3]));
    }
  }
}

// Same for a layer with n_out <= 4 outputs and 64 inputs: lane owns input rows k = lane, lane + 32
// of the image, the deltas are the tile's rows 0..n_out-1.
__device__ __forceinline__ void wgrad4(const float *tile, const float *img, int n_out, float *acc, float *acc_b) {
  const int lane = threadIdx.x & 31, sw = tile_sw(lane);
  float h0[32], h1[32];
  const float4 *p0 = reinterpret_cast<const float4 *>(img + lane * kTileRow);
  const float4 *p1 = reinterpret_cast<const float4 *>(img + (lane + 32) * kTileRow);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float4 a = p0[q ^ sw], c = p1[q ^ sw];
    h0[4 * q] = a.x; h0[4 * q + 1] = a.y; h0[4 * q + 2] = a.z; h0[4 * q + 3] = a.w;
    h1[4 * q] = c.x; h1[4 * q + 1] = c.y; h1[4 * q + 2] = c.z; h1[4 * q + 3] = c.w;
  }
#pragma unroll 1
  for (int j = 0; j < n_out; ++j) {
    const float4 *pd = reinterpret_cast<const float4 *>(tile + j * kTileRow);
    const int swj = tile_sw(j);
    float a0 = 0.f, a1 = 0.f, sb = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 d = pd[q ^ swj];
      a0 = fmaf(h0[4 * q], d.x, fmaf(h0[4 * q + 1], d.y, fmaf(h0[4 * q + 2], d.z, fmaf(h0[4 * q + 3], d.w, a0))));
      a1 = fmaf(h1[4 * q], d.x, fmaf(h1[4 * q + 1], d.y, fmaf(h1[4 * q + 2], d.z, fmaf(h1[4 * q + 3], d.w, a1))));
      sb += d.x + d.y + d.z + d.w;
    }
    atomicAdd(acc + lane * 4 + j, a0);
    atomicAdd(acc + (lane + 32) * 4 + j, a1);
    if (lane == 0) atomicAdd(acc_b + j, sb);
  }
}

// ------------------------------------------------------------ the forward of a tile
// A finished hidden layer: into the tile and, when the backward follows, its image and signs.
template <bool SAVE>
__device__ __forceinline__ void layer_done(const FragLane &L, const float (&c)[2][8][4], float *tile, float *img,
                                           float *sign) {
  frag_store<8>(L, c, tile);
  if (!SAVE) return;
  tile_save(tile, img, kWidth);
  uint32_t bits[2] = {0u, 0u};
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < 8; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q) bits[m] |= (c[m][n][q] > 0.f ? 1u : 0u) << (4 * n + q);
  reinterpret_cast<uint2 *>(sign)[threadIdx.x & 31] = make_uint2(bits[0], bits[1]);
}

// The backward's counterpart: the delta of the layer below, through its ReLU, into the tile.
__device__ __forceinline__ void delta_done(const FragLane &L, uint2 sign, float (&c)[2][8][4], float *tile) {
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < 8; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (!(((m ? sign.y : sign.x) >> (4 * n + q)) & 1u)) c[m][n][q] = 0.f;
  frag_store<8>(L, c, tile);
}

// One lane's sample through the field: its warped point, its canonical point, the four raw
// outputs and whether the canonical point lies in the box.
struct FieldOut {
  float xs0, xs1, xs2, S, xf0, xf1, xf2, o[4];
  bool inside;
};

// Both MLPs of the warp's tile for the 32 samples at s (lanes without a sample: zeros), the pose
// being training frame f's.  SAVE: activations, encodings and signs go to the image for the
// backward.  Every lane of the warp must take part.  Not inlined: compiled by itself, the forward
// gets the same fused multiply-adds in every kernel that calls it, so the colours of a step are
// those of the forward-only call bit for bit (inlined into the backward they differed in the last
// bit, and with them the side of a kink that a few samples fall on).
template <bool SAVE>
__device__ __noinline__ void field_forward(const FieldParams &P, const TrainDev &T, const FragLane &L,
                                              const float *sW, float *tile, float *img, const float4 s, bool active,
                                              uint32_t f, FieldOut &F) {
  const FragLay &W = T.fl;
  const Rows &R = T.rw;
  const int lane = threadIdx.x & 31;
  auto put = [=](int k, float v) {
    if (k < kGamRows) tile[frag_at(k, lane)] = v;
  };
  F.xs0 = F.xs1 = F.xs2 = F.S = 0.f;
  {  // four bones' corner blocks in flight at a time (the bits of lbs_warp)
    const float *G = T.fG + (size_t)f * kBones * 12;
    LbsState st;
    st.x0 = s.x;
    st.x1 = s.y;
    st.x2 = s.z;
    lbs_begin(P, G, nullptr, st, active);
    lbs_end(P, G, st, F.xs0, F.xs1, F.xs2, F.S);
  }
  if (active) {
    if (P.res_enabled) pos_enc(P, F.xs0, F.xs1, F.xs2, put);
  } else if (P.res_enabled) {
    for (int q = 0; q < kGamRows; ++q) put(q, 0.f);
  }
  F.xf0 = F.xs0;
  F.xf1 = F.xs1;
  F.xf2 = F.xs2;
  float c[2][8][4];
  auto sign_of = [&](int l) { return img + (R.sign + 2 * l) * kTileRow; };
  if (P.res_enabled) {
    __syncwarp();
    tile_save(tile, img + R.gam * kTileRow, kGamRows);
    frag_zero(c);
    frag_fwd<8>(L, tile, kGamRows / 8, sW + W.r1, kGamRows / 8, 0, c);
    frag_relu_rows(L, T.fbias1, (int)f, c);
    layer_done<SAVE>(L, c, tile, img + R.rh * kTileRow, sign_of(0));
#pragma unroll 1
    for (int l = 1; l < 4; ++l) {
      frag_zero(c);
      frag_fwd<8>(L, tile, 8, sW + (l == 1 ? W.r2 : l == 2 ? W.r3 : W.r4), l == 3 ? 8 + kGamRows / 8 : 8, 0, c);
      if (l == 3) {   // layer 4 sees [h3, gamma]
        tile_load(tile, img + R.gam * kTileRow, kGamRows);
        frag_fwd<8>(L, tile, kGamRows / 8, sW + W.r4, 8 + kGamRows / 8, 8, c);
      }
      frag_relu(L, sW + (l == 1 ? W.r2b : l == 2 ? W.r3b : W.r4b), c);
      layer_done<SAVE>(L, c, tile, img + (R.rh + l * kWidth) * kTileRow, sign_of(l));
    }
    float xr[4];
    frag_out4(L, tile, sW + W.r5, sW + W.r5b, xr);
    F.xf0 += xr[0];
    F.xf1 += xr[1];
    F.xf2 += xr[2];
  }
  F.inside = false;
  auto put_enc = [=](int k, float v) { tile[frag_at(k, lane)] = v; };
  if (active) {
    F.inside = hash_encode(P, F.xf0, F.xf1, F.xf2, put_enc);
  } else {
    for (int q = 0; q < kMlpIn; ++q) put_enc(q, 0.f);
  }
  __syncwarp();
  const int eb = (2 * P.L + 7) >> 3;   // blocks of inputs that hold features
  if (SAVE) tile_save(tile, img + R.enc * kTileRow, 8 * eb);
#pragma unroll 1
  for (int l = 0; l < P.hidden; ++l) {
    frag_zero(c);
    frag_fwd<8>(L, tile, l ? 8 : eb, sW + (l ? W.ch[l - 1] : W.c0), l ? 8 : kMlpIn / 8, 0, c);
    frag_relu(L, sW + (l ? W.chb[l - 1] : W.c0b), c);
    layer_done<SAVE>(L, c, tile, img + (R.ch + l * kWidth) * kTileRow, sign_of(4 + l));
  }
  frag_out4(L, tile, sW + W.cl, sW + W.clb, F.o);
}

// A slot's (r, g, b, alpha).
__device__ __forceinline__ float4 slot_colour(const FieldOut &F, float delta) {
  const float a = F.inside ? -expm1f(-softplusf_(F.o[3]) * delta) * fminf(F.S, 1.f) : 0.f;
  return make_float4(sigmoidf_(F.o[0]), sigmoidf_(F.o[1]), sigmoidf_(F.o[2]), a);
}

// ------------------------------------------------------------ forward field
// The float32 field with the pose of each sample's frame.  Writes (r, g, b, alpha) per sample
// slot (zero for a ray that misses the box).
__global__ void __launch_bounds__(kTrainThreads, 1) train_fwd_kernel(FieldParams P, TrainDev T) {
  extern __shared__ float4 smem4[];
  float *sW = reinterpret_cast<float *>(smem4);
  const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  float *tile = sW + T.fl.total + warp * kTileFloats;
  stage_frag_weights(P.blob, P.lay, T.fl, P.hidden, sW);
  __syncthreads();
  const FragLane L = frag_lane();
  float *img = T.scratch + ((size_t)blockIdx.x * warps + warp) * T.rw.total * kTileRow;
  const uint32_t n = T.n_rays * T.S;
  const uint32_t step = gridDim.x * blockDim.x;
  const uint32_t n_iter = (n + step - 1) / step;
  for (uint32_t it = 0; it < n_iter; ++it) {
    const uint32_t q = it * step + blockIdx.x * blockDim.x + threadIdx.x;   // thread slot
    const uint32_t r = q < n ? ray_of(T, q) : 0;
    const uint32_t j = r * T.S + q % T.S;                                       // sample slot
    const bool active = q < n && T.raycnt[r] != 0;
    if (!__any_sync(0xffffffffu, active)) {   // 32 slots of rays that miss the box
      if (q < n) T.out[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if ((threadIdx.x & 31) == 0 && q < n) T.live[q >> 5] = 0u;
      continue;
    }
    const uint32_t f = active ? T.frame_id[r] : 0;
    const float4 s = active ? T.samp[j] : make_float4(0.f, 0.f, 0.f, 0.f);
    FieldOut F;
    field_forward<false>(P, T, L, sW, tile, img, s, active, f, F);
    {
      // the slots whose samples carry a gradient (in the box, warped into the canonical box);
      // the backward skips the others, which add exactly zero
      const uint32_t lw = __ballot_sync(0xffffffffu, active && F.inside);
      if ((threadIdx.x & 31) == 0 && q < n) T.live[q >> 5] = lw;
    }
    if (q < n) T.out[j] = active ? slot_colour(F, s.w) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// The compositing adjoint of train_composite_kernel for the RB rays whose slots a block holds
// (ray slots rs0 .. rs0 + RB - 1; local ray lr's samples are the block's slots lr S ..), by the
// block's first warp.  Slot i's (r, g, b, alpha) lies in its warp's tile, at slot_at(i), on entry
// and its (dL/dc, dL/dalpha) on exit; the transmittance in front of it goes 128 floats behind.
// Same arithmetic in the same order, the slots loaded eight ahead of the chain.
__device__ __forceinline__ int slot_at(uint32_t i) { return (int)(i >> 5) * kTileFloats + (int)(i & 31) * 4; }
__device__ __forceinline__ int slot_T(uint32_t i) { return (int)(i >> 5) * kTileFloats + 128 + (int)(i & 31); }

__device__ __forceinline__ void composite_rays(const TrainDev &T, float *tiles, uint32_t rs0, uint32_t RB) {
  const int lane = threadIdx.x & 31;
  float lsum = 0.f;
  for (uint32_t lr = lane; lr < RB; lr += 32) {
    const uint32_t rs = rs0 + lr;
    if (rs >= T.n_rays) break;
    const uint32_t r = (uint32_t)(((uint64_t)rs * T.ray_mul) % T.n_rays);
    const uint32_t i0 = lr * T.S;
    const uint32_t cnt = T.raycnt[r];
    float Tr = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
    for (uint32_t i = 0; i < cnt; i += 8) {
      float4 v[8];
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k)
        if (i + k < cnt) v[k] = *reinterpret_cast<const float4 *>(tiles + slot_at(i0 + i + k));
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) {
        if (i + k >= cnt) break;
        tiles[slot_T(i0 + i + k)] = Tr;
        const float w = Tr * v[k].w;
        c0 = fmaf(w, v[k].x, c0);
        c1 = fmaf(w, v[k].y, c1);
        c2 = fmaf(w, v[k].z, c2);
        Tr *= 1.f - v[k].w;
      }
    }
    const float C0 = fmaf(Tr, T.bg[0], c0), C1 = fmaf(Tr, T.bg[1], c1), C2 = fmaf(Tr, T.bg[2], c2);
    if (T.pred) {
      T.pred[3 * r] = C0;
      T.pred[3 * r + 1] = C1;
      T.pred[3 * r + 2] = C2;
    }
    float g0 = 0.f, g1 = 0.f, g2 = 0.f;
    if (T.grad_rgb) {
      g0 = T.grad_rgb[3 * r];
      g1 = T.grad_rgb[3 * r + 1];
      g2 = T.grad_rgb[3 * r + 2];
    } else if (T.target) {
      const float e0 = C0 - T.target[3 * r], e1 = C1 - T.target[3 * r + 1], e2 = C2 - T.target[3 * r + 2];
      lsum += T.loss_weight * (e0 * e0 + e1 * e1 + e2 * e2);
      const float scale = 2.f * T.loss_weight / (3.f * (float)T.n_rays);
      g0 = scale * e0;
      g1 = scale * e1;
      g2 = scale * e2;
    }
    float B = T.bg[0] * g0 + T.bg[1] * g1 + T.bg[2] * g2;
    for (uint32_t e = cnt; e > 0;) {   // samples e - 1, e - 2, ..: eight at a time
      const uint32_t m = e < 8u ? e : 8u;
      float4 v[8];
      float t[8];
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k)
        if (k < m) {
          v[k] = *reinterpret_cast<const float4 *>(tiles + slot_at(i0 + e - 1 - k));
          t[k] = tiles[slot_T(i0 + e - 1 - k)];
        }
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) {
        if (k >= m) break;
        const float cg = v[k].x * g0 + v[k].y * g1 + v[k].z * g2;
        const float ta = t[k] * v[k].w;
        *reinterpret_cast<float4 *>(tiles + slot_at(i0 + e - 1 - k)) =
            make_float4(ta * g0, ta * g1, ta * g2, t[k] * (cg - B));
        B = fmaf(v[k].w, cg, (1.f - v[k].w) * B);
      }
      e -= m;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
  if (lane == 0 && lsum != 0.f) atomicAdd(T.loss, lsum / (3.f * (float)T.n_rays));
}

// A warp per 32 samples: forward (activations to the warp's image), backward, scatter-adds and the
// warp's weight gradients.
// FUSED: the block takes groups of whole rays (RB = blockDim / S of them), evaluates every sample
// once, composites its rays in shared memory and goes straight on to the backward, so that neither
// train_fwd_kernel nor train_composite_kernel is needed.
template <bool FUSED>
__global__ void __launch_bounds__(kTrainThreads, 1) train_bwd_kernel(FieldParams P, TrainDev T) {
  extern __shared__ float4 smem4[];
  float *sW = reinterpret_cast<float *>(smem4);
  float *tiles = sW + T.fl.total;                      // a tile per warp
  stage_frag_weights(P.blob, P.lay, T.fl, P.hidden, sW);
  __syncthreads();
  const BlobLayout &Ly = P.lay;                        // the gradient accumulators' layout
  const FragLay &W = T.fl;
  const Rows &R = T.rw;
  const FragLane L = frag_lane();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float *tile = tiles + warp * kTileFloats;
  float *img = T.scratch + ((size_t)blockIdx.x * (blockDim.x >> 5) + warp) * R.total * kTileRow;
  float *acc = T.wacc + (size_t)blockIdx.x * T.acc_floats;
  float *accF = acc + Ly.total;                        // per-frame first-layer bias gradients [F][64]
  float *accG = T.dG_acc ? accF + T.n_frames * kWidth : T.dG;   // dL/dG [F][24][12]
  const int H = P.hidden;
  const uint32_t n = T.n_rays * T.S;
  const uint32_t step = gridDim.x * blockDim.x;
  const uint32_t RB = FUSED ? blockDim.x / T.S : 0u, SB = RB * T.S;   // FUSED: rays and slots a group
  const uint32_t n_units = FUSED ? (T.n_rays + RB - 1) / RB : (n + step - 1) / step;
  for (uint32_t it = FUSED ? blockIdx.x : 0u; it < n_units; it += FUSED ? gridDim.x : 1u) {
    const uint32_t q = FUSED ? it * SB + threadIdx.x : it * step + blockIdx.x * blockDim.x + threadIdx.x;  // slot
    const bool qv = q < n && (!FUSED || threadIdx.x < SB);
    const uint32_t q0 = q - lane;                                               // the warp's first slot
    const uint32_t r = qv ? ray_of(T, q) : 0;
    const uint32_t j = r * T.S + q % T.S;                                       // sample slot
    bool active;
    if constexpr (FUSED) {
      active = qv && T.raycnt[r] != 0;   // every slot of a ray that meets the box is evaluated
    } else {
      // the forward's mask: a slot outside it (no box hit, or warped out of the canonical box)
      // adds exactly zero to every gradient, and a warp without live slots has nothing to do
      const uint32_t lw = q0 < n ? T.live[q0 >> 5] : 0u;
      if (lw == 0u) continue;
      active = (lw >> lane) & 1u;
    }
    const uint32_t f = active ? T.frame_id[r] : 0;
    float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!FUSED && active) g4 = __ldcs(T.out + j);
    const bool run = !FUSED || __any_sync(0xffffffffu, active);   // warp-uniform
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    FieldOut F{};
    if (run) {
      if (active) s = __ldcs(T.samp + j);
      field_forward<true>(P, T, L, sW, tile, img, s, active, f, F);
    }
    if constexpr (FUSED) {
      // each slot's (r, g, b, alpha), the rays composited by the first warp, its adjoint back
      if (threadIdx.x < SB)
        *reinterpret_cast<float4 *>(tiles + slot_at(threadIdx.x)) =
            active ? slot_colour(F, s.w) : make_float4(0.f, 0.f, 0.f, 0.f);
      __syncthreads();
      if (warp == 0) composite_rays(T, tiles, it * RB, RB);
      __syncthreads();
      if (active) g4 = *reinterpret_cast<const float4 *>(tiles + slot_at(threadIdx.x));
      // no live slot in the warp: its tile is left as it is until the next group's forward
      if (__ballot_sync(0xffffffffu, active && F.inside) == 0u) continue;
    }
    active = active && F.inside;
    float dcl[4] = {0.f, 0.f, 0.f, 0.f}, dS_alpha = 0.f;
    if (active) {
      // ---------------- alpha, rgb, sigma
      const float sig = softplusf_(F.o[3]);
      const float e = expf(-sig * s.w);
      const float lk = fminf(F.S, 1.f);
      const float dsig = g4.w * s.w * e * lk;
      dS_alpha = F.S < 1.f ? g4.w * -expm1f(-sig * s.w) : 0.f;
      const float gc[3] = {g4.x, g4.y, g4.z};
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float c = sigmoidf_(F.o[k]);
        dcl[k] = gc[k] * c * (1.f - c);
      }
      dcl[3] = dsig * sigmoidf_(F.o[3]);
    }
    __syncwarp();   // every lane has its adjoint
#pragma unroll
    for (int k = 0; k < 8; ++k) tile[frag_at(k, lane)] = k < 4 ? dcl[k] : 0.f;
    __syncwarp();
    float c[2][8][4];
    auto sign_of = [&](int l) { return reinterpret_cast<const uint2 *>(img + (R.sign + 2 * l) * kTileRow)[lane]; };
    // ---------------- canonical MLP backward: each layer's weight gradient summed as soon as its
    // delta is in the tile, then the delta of the layer below
    {
      wgrad4(tile, img + (R.ch + (H - 1) * kWidth) * kTileRow, 4, acc + Ly.cl, acc + Ly.clb);
#pragma unroll 1
      for (int l = H; l >= 1; --l) {   // the delta of layer l is in the tile (l = H: the outputs)
        const uint2 sg = sign_of(4 + l - 1);
        if (l < H) wgrad64(L, tile, img + (R.ch + (l - 1) * kWidth) * kTileRow, 8, acc + Ly.ch[l - 1], acc + Ly.chb[l - 1], nullptr);
        frag_zero(c);
        frag_back<8>(L, tile, l == H ? 1 : 8, sW + (l == H ? W.cl : W.ch[l - 1]), 8, 0, c);
        delta_done(L, sg, c, tile);
      }
      const int eb = (2 * P.L + 7) >> 3;
      wgrad64(L, tile, img + R.enc * kTileRow, eb, acc + Ly.c0, acc + Ly.c0b, nullptr);
      float d[2][4][4];
      frag_zero(d);
      frag_back<4>(L, tile, 8, sW + W.c0, kMlpIn / 8, 0, d);
      frag_store<4>(L, d, tile);
    }
    float dx0 = 0.f, dx1 = 0.f, dx2 = 0.f;
    {
      // ---------------- hash backward: warp-aggregated scatter-add and dL/dx_final
      const float p0 = active ? (F.xf0 - P.bmin[0]) * P.inv_box[0] : 0.f;
      const float p1 = active ? (F.xf1 - P.bmin[1]) * P.inv_box[1] : 0.f;
      const float p2 = active ? (F.xf2 - P.bmin[2]) * P.inv_box[2] : 0.f;
      for (int l = 0; l < P.L; ++l) {
        const float da = active ? tile[frag_at(2 * l, lane)] : 0.f;
        const float db = active ? tile[frag_at(2 * l + 1, lane)] : 0.f;
        const uint32_t N = P.level_res[l];
        const float fn = (float)N;
        const float q0 = p0 * fn, q1 = p1 * fn, q2 = p2 * fn;
        const float a0 = fminf(floorf(q0), fn - 1.f), a1 = fminf(floorf(q1), fn - 1.f),
                    a2 = fminf(floorf(q2), fn - 1.f);
        const float fr[3] = {__fsub_rn(q0, a0), __fsub_rn(q1, a1), __fsub_rn(q2, a2)};
        HashCell c;
        hash_cell(P, l, p0, p1, p2, c);
        float2 tv[8];   // the corners, loaded before the exchange below
#pragma unroll
        for (int k = 0; k < 8; ++k)
          tv[k] = active ? __ldg(P.table32 + (size_t)l * (P.T_mask + 1) + c.idx[k]) : make_float2(0.f, 0.f);
        float v[16];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          v[2 * k] = c.w[k] * da;
          v[2 * k + 1] = c.w[k] * db;
        }
        const uint32_t ka = (uint32_t)a0 | ((uint32_t)a1 << 16), kb = (uint32_t)a2;
        if (run_sum<16>(ka, kb, active, v)) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            atomicAdd(T.g_table + (size_t)l * (P.T_mask + 1) + c.idx[k], make_float2(v[2 * k], v[2 * k + 1]));
        }
        if (active) {
          float gp0 = 0.f, gp1 = 0.f, gp2 = 0.f;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const float sv = tv[k].x * da + tv[k].y * db;
            const float wx = (k & 1) ? fr[0] : 1.f - fr[0], wy = ((k >> 1) & 1) ? fr[1] : 1.f - fr[1],
                        wz = (k >> 2) ? fr[2] : 1.f - fr[2];
            const float sx = (k & 1) ? 1.f : -1.f, sy = ((k >> 1) & 1) ? 1.f : -1.f, sz = (k >> 2) ? 1.f : -1.f;
            gp0 = fmaf(sv, sx * wy * wz, gp0);
            gp1 = fmaf(sv, wx * sy * wz, gp1);
            gp2 = fmaf(sv, wx * wy * sz, gp2);
          }
          dx0 = fmaf(gp0, fn, dx0);
          dx1 = fmaf(gp1, fn, dx1);
          dx2 = fmaf(gp2, fn, dx2);
        }
      }
      dx0 *= P.inv_box[0];
      dx1 *= P.inv_box[1];
      dx2 *= P.inv_box[2];
    }
    float ds0 = dx0, ds1 = dx1, ds2 = dx2;
    if (P.res_enabled) {
      // ---------------- residual MLP backward (x_final = x_skel + x_res), tensor cores
      const uint32_t fl = qv ? T.frame_id[r] : 0u;   // the frames of the warp's slots: one, if they agree
      const uint32_t fl0 = __shfl_sync(0xffffffffu, fl, 0);
      const bool one = __all_sync(0xffffffffu, !qv || fl == fl0) && (q0 < n && (!FUSED || warp * 32u < SB));
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 8; ++k) tile[frag_at(k, lane)] = k == 0 ? dx0 : k == 1 ? dx1 : k == 2 ? dx2 : 0.f;
      __syncwarp();
      wgrad4(tile, img + (R.rh + 3 * kWidth) * kTileRow, 3, acc + Ly.r5, acc + Ly.r5b);
#pragma unroll 1
      for (int l = 4; l >= 1; --l) {   // l = 4: the outputs' delta in the tile; below, hidden layer l + 1's
        const uint2 sg = sign_of(l - 1);
        const int IB = l == 3 ? 8 + kGamRows / 8 : 8;
        if (l < 4)
          wgrad64(L, tile, img + (R.rh + (l - 1) * kWidth) * kTileRow, 8, acc + (l == 3 ? Ly.r4 : l == 2 ? Ly.r3 : Ly.r2),
                  acc + (l == 3 ? Ly.r4b : l == 2 ? Ly.r3b : Ly.r2b), nullptr);
        if (l == 3) {   // layer 4's gamma inputs: weight gradient and the first part of dL/dgamma
          wgrad64(L, tile, img + R.gam * kTileRow, kGamRows / 8, acc + Ly.r4 + kWidth * kWidth, nullptr, nullptr);
          float d[2][kGamRows / 8][4];
          frag_zero(d);
          frag_back<kGamRows / 8>(L, tile, 8, sW + W.r4, IB, 8, d);
          float4 *o = reinterpret_cast<float4 *>(img + R.dgam * kTileRow) + lane;
#pragma unroll
          for (int k = 0; k < 2 * (kGamRows / 8); ++k)
            o[32 * k] = make_float4(d[k & 1][k >> 1][0], d[k & 1][k >> 1][1], d[k & 1][k >> 1][2], d[k & 1][k >> 1][3]);
        }
        frag_zero(c);
        frag_back<8>(L, tile, l == 4 ? 1 : 8, sW + (l == 4 ? W.r5 : l == 3 ? W.r4 : l == 2 ? W.r3 : W.r2), IB, 0, c);
        delta_done(L, sg, c, tile);
      }
      wgrad64(L, tile, img + R.gam * kTileRow, kGamRows / 8, acc + Ly.r1, acc + Ly.r1b,
              one ? accF + fl0 * kWidth : nullptr);
      if (!one) {  // per-frame sums of delta1 (for W_Omega): lane owns rows lane, lane + 32
        const float *d0 = tile + lane * kTileRow, *d1 = tile + (lane + 32) * kTileRow;
        int cur = -1;
        float s0 = 0.f, s1 = 0.f;
        for (int sI = 0; sI < 32; ++sI) {
          if (q0 + sI >= n || (FUSED && (uint32_t)(warp * 32 + sI) >= SB)) break;
          const int fr = (int)__shfl_sync(0xffffffffu, fl, sI);
          if (fr != cur) {
            if (cur >= 0) {
              atomicAdd(accF + cur * kWidth + lane, s0);
              atomicAdd(accF + cur * kWidth + lane + 32, s1);
            }
            cur = fr;
            s0 = s1 = 0.f;
          }
          const int at = frag_at(lane, sI) - lane * kTileRow;
          s0 += d0[at];
          s1 += d1[at];
        }
        if (cur >= 0) {
          atomicAdd(accF + cur * kWidth + lane, s0);
          atomicAdd(accF + cur * kWidth + lane + 32, s1);
        }
      }
      {  // dL/dgamma = layer 4's part + W1_gamma^T delta1 (the pose columns of W1: per frame, above)
        float d[2][kGamRows / 8][4];
        frag_zero(d);
        frag_back<kGamRows / 8>(L, tile, 8, sW + W.r1, kGamRows / 8, 0, d);
        const float4 *o = reinterpret_cast<const float4 *>(img + R.dgam * kTileRow) + lane;
#pragma unroll
        for (int k = 0; k < 2 * (kGamRows / 8); ++k) {
          const float4 v = o[32 * k];
          d[k & 1][k >> 1][0] += v.x;
          d[k & 1][k >> 1][1] += v.y;
          d[k & 1][k >> 1][2] += v.z;
          d[k & 1][k >> 1][3] += v.w;
        }
        frag_store<kGamRows / 8>(L, d, tile);
      }
      if (active) {
          // through gamma: d gamma / d x_skel
          auto dg = [&](int k) { return tile[frag_at(k, lane)]; };
          const float xh[3] = {(F.xs0 - P.box_c[0]) * P.box_ih[0], (F.xs1 - P.box_c[1]) * P.box_ih[1],
                               (F.xs2 - P.box_c[2]) * P.box_ih[2]};
          float dh[3] = {dg(0), dg(1), dg(2)};
          for (int k = 0; k < P.res_freqs; ++k) {
            const float sc = (float)(1 << k);
            const float wk = P.hann[k] * sc * 3.14159265358979f;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              float sn, cs;
              sincospif(sc * xh[a], &sn, &cs);
              dh[a] += wk * (dg(3 + 6 * k + a) * cs - dg(6 + 6 * k + a) * sn);
            }
          }
          ds0 += dh[0] * P.box_ih[0];
          ds1 += dh[1] * P.box_ih[1];
          ds2 += dh[2] * P.box_ih[2];
      }
    }
    float *dp = img + R.dp * kTileRow, *xs = img + R.xs * kTileRow;
    {
      // ---------------- inverse-LBS backward: warp-aggregated scatter into the weight volume
      // and, for the pose refiner, dL/dp_i of each candidate p_i = G_i x:
      //   x_skel = sum_i w_i p_i / D,  w_i = W_i(p_i)
      //   dL/dp_i = (w_i / D) dL/dx_skel + dL/dw_i grad W_i(p_i)
      const float D = fmaxf(F.S, kEpsW);
      // one division per sample: a per-bone quotient with a vanishing numerator (far from the
      // body S, and with it the gradient reaching x_skel, goes to zero) takes the division's
      // slow path 24 times a sample
      const float inv_D = 1.f / D;
      const float m = F.S > kEpsW ? 1.f : 0.f;
      const float *G = T.fG + (size_t)f * kBones * 12;
      const int R = P.wres, R3 = R * R * R;
      const size_t QC = quad_channel(R);
      if (T.dG && active) {
        xs[lane] = s.x;
        xs[kTileRow + lane] = s.y;
        xs[2 * kTileRow + lane] = s.z;
      }
      for (int i = 0; i < kBones; ++i) {
        const float *g = G + 12 * i;
        const float p0 = fmaf(g[0], s.x, fmaf(g[1], s.y, fmaf(g[2], s.z, g[3])));
        const float p1 = fmaf(g[4], s.x, fmaf(g[5], s.y, fmaf(g[6], s.z, g[7])));
        const float p2 = fmaf(g[8], s.x, fmaf(g[9], s.y, fmaf(g[10], s.z, g[11])));
        const float dw = (ds0 * (p0 - m * F.xs0) + ds1 * (p1 - m * F.xs1) + ds2 * (p2 - m * F.xs2)) * inv_D + dS_alpha;
        const float ux = (p0 - P.bmin[0]) * P.vol_scale[0];
        const float uy = (p1 - P.bmin[1]) * P.vol_scale[1];
        const float uz = (p2 - P.bmin[2]) * P.vol_scale[2];
        if (T.dG && active) {
          float gx, gy, gz;
          const float w = trilinear_quad_grad(P.wquad + (size_t)i * QC, R, ux, uy, uz, gx, gy, gz);
          const float a = w * inv_D;
          dp[(3 * i + 0) * kTileRow + lane] = fmaf(a, ds0, dw * gx * P.vol_scale[0]);
          dp[(3 * i + 1) * kTileRow + lane] = fmaf(a, ds1, dw * gy * P.vol_scale[1]);
          dp[(3 * i + 2) * kTileRow + lane] = fmaf(a, ds2, dw * gz * P.vol_scale[2]);
        }
        const float fx0 = floorf(ux), fy0 = floorf(uy), fz0 = floorf(uz);
        const bool in_range = fx0 >= -1.f && fy0 >= -1.f && fz0 >= -1.f && fx0 < (float)R && fy0 < (float)R &&
                              fz0 < (float)R;
        const bool valid = active && dw != 0.f && in_range;
        const int ix = valid ? (int)fx0 : 0, iy = valid ? (int)fy0 : 0, iz = valid ? (int)fz0 : 0;
        const float fx = __fsub_rn(ux, fx0), fy = __fsub_rn(uy, fy0), fz = __fsub_rn(uz, fz0);
        float v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c)
          v[c] = dw * (((c & 1) ? fx : 1.f - fx) * (((c >> 1) & 1) ? fy : 1.f - fy) * ((c >> 2) ? fz : 1.f - fz));
        const uint32_t key = (uint32_t)(ix + 1) | ((uint32_t)(iy + 1) << 10) | ((uint32_t)(iz + 1) << 20);
        if (run_sum<8>(key, 0u, valid, v)) {
          if (T.g_quad) {   // the cell's two corner blocks, one 16-byte add each
            const int R1 = R + 1;
            float4 *e = T.g_quad + (size_t)i * QC + ((iz + 1) * R1 + (iy + 1)) * R1 + (ix + 1);
            atomicAdd(e, make_float4(v[0], v[1], v[2], v[3]));
            atomicAdd(e + R1 * R1, make_float4(v[4], v[5], v[6], v[7]));
          } else {
            float *chg = T.g_wvol + (size_t)i * R3;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const int ax = ix + (c & 1), ay = iy + ((c >> 1) & 1), az = iz + (c >> 2);
              if (ax < 0 || ay < 0 || az < 0 || ax >= R || ay >= R || az >= R) continue;
              atomicAdd(chg + (az * R + ay) * R + ax, v[c]);
            }
          }
        }
      }
    }
    if (T.dG && !active)   // the refiner's reduction reads these rows of every lane
      for (int q = 0; q < 3 * kBones + 3; ++q) dp[q * kTileRow + lane] = 0.f;   // (xs follows dp)
    __syncwarp();
    if (T.dG) {
      // dL/dG_i of each frame: dR_i += dp_i x^T, dt_i += dp_i over the warp's 32 samples;
      // lane owns 9 of the 24 x 12 entries and sums them per run of equal frames
      const int fl = qv ? (int)T.frame_id[r] : -1;
      const int f0 = __shfl_sync(0xffffffffu, fl, 0);
      if (__all_sync(0xffffffffu, fl == f0) && f0 >= 0) {
        // one frame in the warp: C[3i + r][c] = sum_s dp_i[s][r] (x_s, y_s, z_s, 1)[c] as one
        // tensor-core product (M = 72 rows of dp in 16-row tiles, N = 4 columns padded to 8,
        // K = the 32 samples; m16n8k8 TF32, three products per step)
        const int g = lane >> 2, t = lane & 3;
        float *dst = accG + (size_t)f0 * kBones * 12;
        uint32_t bh[4][2], bl[4][2];   // B[s][c] = (x, y, z, 1)[c] of sample s, zero for c >= 4
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          const int s0 = 8 * ks + t;
          const float v0 = g < 3 ? xs[g * kTileRow + s0] : (g == 3 ? 1.f : 0.f);
          const float v1 = g < 3 ? xs[g * kTileRow + s0 + 4] : (g == 3 ? 1.f : 0.f);
          tf32_split(v0, bh[ks][0], bl[ks][0]);
          tf32_split(v1, bh[ks][1], bl[ks][1]);
        }
#pragma unroll 1
        for (int mt = 0; mt < 5; ++mt) {
          const int o0 = 16 * mt + g, o8 = o0 + 8;
          float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {
            const int s0 = 8 * ks + t;
            uint32_t ah[4], al[4];
            tf32_split(o0 < 3 * kBones ? dp[o0 * kTileRow + s0] : 0.f, ah[0], al[0]);
            tf32_split(o8 < 3 * kBones ? dp[o8 * kTileRow + s0] : 0.f, ah[1], al[1]);
            tf32_split(o0 < 3 * kBones ? dp[o0 * kTileRow + s0 + 4] : 0.f, ah[2], al[2]);
            tf32_split(o8 < 3 * kBones ? dp[o8 * kTileRow + s0 + 4] : 0.f, ah[3], al[3]);
            mma_tf32(c, al, bh[ks]);
            mma_tf32(c, ah, bl[ks]);
            mma_tf32(c, ah, bh[ks]);
          }
          // c = C[o0][2t], C[o0][2t + 1], C[o8][2t], C[o8][2t + 1]
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int o = q >= 2 ? o8 : o0, cc = 2 * t + (q & 1);
            if (o < 3 * kBones && cc < 4 && c[q] != 0.f) atomicAdd(dst + (o / 3) * 12 + (o % 3) * 4 + cc, c[q]);
          }
        }
      } else {
      for (int o = lane; o < kBones * 12; o += 32) {
        const int i = o / 12, rr = (o % 12) >> 2, c = o & 3;
        const float *dpr = dp + (3 * i + rr) * kTileRow;
        const float *xr = xs + (c < 3 ? c : 0) * kTileRow;
        int cur = -1;
        float v = 0.f;
        for (int sI = 0; sI < 32; ++sI) {
          const int fr = __shfl_sync(0xffffffffu, fl, sI);
          if (fr < 0) break;
          if (fr != cur) {
            if (cur >= 0 && v != 0.f) atomicAdd(accG + cur * kBones * 12 + o, v);
            cur = fr;
            v = 0.f;
          }
          v = fmaf(dpr[sI], c < 3 ? xr[sI] : 1.f, v);
        }
        if (cur >= 0 && v != 0.f) atomicAdd(accG + cur * kBones * 12 + o, v);
      }
      }
    }
    __syncwarp();
  }
}

// The weight-volume gradient from its corner-block sums: a vertex lies in up to four blocks of its
// plane (as corner 0 of its own cell, 1 of the cell before in x, 2 in y, 3 in both).
__global__ void __launch_bounds__(256) fold_quad_kernel(const float4 *__restrict__ quad, int R, float *__restrict__ g) {
  const size_t QC = quad_channel(R), R3 = (size_t)R * R * R;
  const size_t n = R3 * kBones;
  const int R1 = R + 1;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(e / R3), v = (int)(e % R3);
    const int x = v % R, y = (v / R) % R, z = v / (R * R);
    const float4 *q = quad + (size_t)c * QC + ((size_t)(z + 1) * R1 + y) * R1 + x;
    g[e] = (__ldg(&q[R1 + 1].x) + __ldg(&q[R1].y)) + (__ldg(&q[1].z) + __ldg(&q[0].w));
  }
}

// Sum of the per-block accumulators: red[e] = sum_w wacc[w][e].
__global__ void reduce_acc_kernel(const float *__restrict__ wacc, int n_warps, int A, float *__restrict__ red) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= A) return;
  float s = 0.f;
  for (int w = 0; w < n_warps; ++w) s += wacc[(size_t)w * A + e];
  red[e] = s;
}

// Gradients in the packed master layout (W[out][in], b) from the accumulators' sums (fragment
// order, acc_index); the joint-angle columns of the residual first layer get
// dL/dW_Omega[j][m] = sum_f (sum of delta1 over frame f)[j] * Omega_f[m].
struct ScatterArgs {
  MasterOffsets m;
  BlobLayout b;
  int g, pose_dim, n_frames, hidden, mlp_in;
};

__global__ void scatter_res_kernel(const float *__restrict__ red, const float *__restrict__ fomega, ScatterArgs a,
                                   float *__restrict__ g_res) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.m.n_res) return;
  const float *accF = red + a.b.total;
  // find the layer
  const int rin[5] = {a.g + a.pose_dim, kWidth, kWidth, kWidth + a.g, kWidth};
  const int rout[5] = {kWidth, kWidth, kWidth, kWidth, 3};
  const int wt[5] = {a.b.r1, a.b.r2, a.b.r3, a.b.r4, a.b.r5};
  const int bb[5] = {a.b.r1b, a.b.r2b, a.b.r3b, a.b.r4b, a.b.r5b};
  for (int l = 0; l < 5; ++l) {
    if (e >= a.m.r[l] && e < a.m.rb[l]) {
      const int q = e - a.m.r[l], j = q / rin[l], k = q % rin[l];
      float v;
      if (l == 0 && k >= a.g) {
        const int mm = k - a.g;
        v = 0.f;
        for (int f = 0; f < a.n_frames; ++f) v = fmaf(accF[f * kWidth + j], fomega[f * a.pose_dim + mm], v);
      } else {
        v = red[wt[l] + (l == 4 ? k * 4 + j : acc_index(j, k))];
      }
      g_res[e] = v;
      return;
    }
    if (e >= a.m.rb[l] && e < a.m.rb[l] + rout[l]) {
      g_res[e] = red[bb[l] + (e - a.m.rb[l])];
      return;
    }
  }
}

__global__ void scatter_mlp_kernel(const float *__restrict__ red, ScatterArgs a, float *__restrict__ g_mlp) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.m.n_mlp) return;
  const int H = a.hidden;
  for (int l = 0; l <= H; ++l) {
    const int in = l == 0 ? a.mlp_in : kWidth;
    const int out = l == H ? 4 : kWidth;
    const int wt = l == 0 ? a.b.c0 : (l == H ? a.b.cl : a.b.ch[l - 1]);
    const int bb = l == 0 ? a.b.c0b : (l == H ? a.b.clb : a.b.chb[l - 1]);
    if (e >= a.m.c[l] && e < a.m.cb[l]) {
      const int q = e - a.m.c[l], j = q / in, k = q % in;
      g_mlp[e] = red[wt + (l == H ? k * 4 + j : acc_index(j, k))];
      return;
    }
    if (e >= a.m.cb[l] && e < a.m.cb[l] + out) {
      g_mlp[e] = red[bb + (e - a.m.cb[l])];
      return;
    }
  }
}

// Adam with bias correction (Kingma and Ba 2015; Sec. 5.2 uses beta = (0.9, 0.99)):
// m = b1 m + (1 - b1) g, v = b2 v + (1 - b2) g^2, p -= lr (m c1) / (sqrt(v c2) + eps),
// c1 = 1 / (1 - b1^t), c2 = 1 / (1 - b2^t).  Every entry is updated.
__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, size_t n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
  }
}

template <typename P_>
static nr_status grow(P_ *&ptr, size_t &cap, size_t need) {
  if (need <= cap) return NR_OK;
  if (ptr) cudaFree(ptr);
  ptr = nullptr;
  cap = 0;
  NR_CHECK_CUDA(cudaMalloc((void **)&ptr, need * sizeof(P_)));
  cap = need;
  return NR_OK;
}

}  // namespace nr

using namespace nr;

extern "C" nr_status nr_train_step(nr_subject *s, const nr_train_batch *b, float *loss_out, void *stream) {
  NR_REQUIRE(subject_ok(s), "nr_train_step: invalid handle");
  NR_REQUIRE(b, "nr_train_step: NULL batch");
  NR_REQUIRE(b->n_rays >= 1 && b->frame_id && b->px && b->py, "nr_train_step: empty or NULL batch");
  const bool fwd_only = (b->flags & NR_FORWARD_ONLY) != 0;
  NR_REQUIRE(b->target_rgb || b->grad_rgb || fwd_only, "nr_train_step: neither target_rgb nor grad_rgb");
  NR_REQUIRE(b->n_samples >= 1 && b->n_samples <= 1024, "nr_train_step: n_samples must be 1..1024");
  NR_REQUIRE((uint64_t)b->n_rays * b->n_samples <= (1ull << 31), "nr_train_step: batch too large");
  NR_REQUIRE(b->lr >= 0.f && b->beta1 >= 0.f && b->beta1 < 1.f && b->beta2 >= 0.f && b->beta2 < 1.f && b->eps > 0.f,
             "nr_train_step: bad Adam hyper-parameters");
  for (int k = 0; k < 4; ++k) NR_REQUIRE(b->lr_scale[k] >= 0.f, "nr_train_step: negative lr_scale");
  NR_REQUIRE(b->loss_weight >= 0.f && b->lr_scale_refiner >= 0.f && b->lr_scale_cnn >= 0.f,
             "nr_train_step: negative loss_weight or lr scale");
  if (s->n_frames == 0) {
    set_error("nr_train_step: call nr_set_frames first");
    return NR_ESTATE;
  }
  NR_CHECK_CUDA(cudaSetDevice(s->device));
  cudaStream_t st = (cudaStream_t)stream;
  nr_status r;
  if ((r = prepare_params(s, st)) != NR_OK) return r;
  const bool refine = s->ref_layers != 0;
  int launched = 0;
  if (refine) {   // every frame's G and updated angles from its refined pose (Sec. 4.1)
    if ((r = launch_refine_fk(s, s->f_omega, 3 * kBones, s->f_root, 3, (int)s->n_frames, s->f_G, s->f_omega_o,
                              3 * kBones, st)) != NR_OK)
      return r;
    s->fG_refined = true;
  } else if (s->fG_refined) {   // the refiner was switched off: back to the estimated poses
    NR_CHECK_CUDA(cudaMemcpyAsync(s->f_G, s->h_fG.data(), s->h_fG.size() * 4, cudaMemcpyHostToDevice, st));
    NR_CHECK_CUDA(cudaStreamSynchronize(st));
    s->fG_refined = false;
  }
  if ((r = fold_frame_biases(s, st)) != NR_OK) return r;
  nr_render_opts o{};
  o.mlp_dtype = NR_F32;
  o.feat_dtype = NR_F32;
  o.hann_alpha = b->hann_alpha;
  FieldParams P = field_params(s, &o);
  P.bone_box = nullptr;   // training differentiates every bone channel
  const size_t n = (size_t)b->n_rays * b->n_samples;
  const int blocks = num_sms(s->device);
  // dL/dG of a few frames is summed per block first, in the block's accumulator (in shared memory it
  // took the place of four warps' tiles), of more straight into f_dG.  One frame's 288 sums are few
  // enough for the adds of all blocks to collide: 16,384 rays x 128 take 9.23 ms per block and 9.32
  // straight.  From four frames to sixty-four the two measure alike (8.92 and 8.94, 8.97 and 8.95,
  // 8.93 and 8.93 at 4, 16 and 64); beyond, clearing and summing 152 x 288 floats a frame shows (300
  // rays x 64, 200 frames: 814 us against 778).
  const bool dG_acc = refine && s->n_frames <= 16;
  const size_t n_dG = (size_t)s->n_frames * kBones * 12;
  const int A = s->lay.total + (int)s->n_frames * kWidth + (dG_acc ? (int)n_dG : 0);
  if (n > s->tw_samples) {              // the three per-sample buffers grow together
    size_t c0 = 0, c1 = 0, c2 = 0;
    if (s->t_samp) cudaFree(s->t_samp);
    if (s->t_out) cudaFree(s->t_out);
    if (s->t_T) cudaFree(s->t_T);
    s->t_samp = nullptr;
    s->t_out = nullptr;
    s->t_T = nullptr;
    s->tw_samples = 0;
    if ((r = grow(s->t_samp, c0, n)) != NR_OK) return r;
    if ((r = grow(s->t_out, c1, n)) != NR_OK) return r;
    if ((r = grow(s->t_T, c2, n)) != NR_OK) return r;
    s->tw_samples = n;
  }
  if ((r = grow(s->t_raycnt, s->tw_rays, (size_t)b->n_rays)) != NR_OK) return r;
  if ((r = grow(s->t_live, s->tw_live, ((size_t)b->n_rays * b->n_samples + 31) / 32)) != NR_OK) return r;
  const Rows rows = make_rows((int)s->hidden);
  const FragLay fl = frag_layout((int)s->hidden);
  // the warps whose tiles fit beside the weights (sixteen with two hidden layers, twelve with four)
  const size_t smem_w = sizeof(float) * fl.total;
  const size_t tile_b = kTileFloats * sizeof(float);
  const int warps_max = (int)std::min<size_t>(kTrainThreads / 32, (kTrainSmem - smem_w) / tile_b);
  // a step whose rays fit a block whole runs forward, compositing and backward in one kernel
  // (train_bwd_kernel<true>) over groups of 32 warps / S rays; else the forward and the
  // compositing adjoint run first
  const bool fused = !fwd_only && b->n_samples <= (uint32_t)(32 * warps_max);
  const int warps_b = fused ? (int)((32u * warps_max / b->n_samples * b->n_samples + 31) / 32) : warps_max;
  // Corner-block sums of the weight-volume gradient take two 16-byte adds a cell instead of eight
  // 4-byte ones, for a buffer to clear and fold (4 x 24 / 25 of the volume's bytes and a shell):
  // taken while that is below kQuadBytes per sample.  2400 rays x 128 samples at 32^3 (15.5 MB)
  // took 1.486 ms with them and 1.528 without, 0.14 ns a sample: what clearing and folding 420
  // bytes cost at 6 TB/s.
  const size_t n_quad = quad_channel((int)s->wres) * kBones;
  const bool quad = !fwd_only && n_quad * sizeof(float4) <= kQuadBytes * n;
  if ((r = grow(s->t_scratch, s->tw_scratch, (size_t)blocks * rows.total * kTileRow * (kTrainThreads / 32))) != NR_OK)
    return r;
  const size_t n_acc = (size_t)blocks;                 // one accumulator per block
  if ((r = grow(s->t_wacc, s->tw_acc, n_acc * A)) != NR_OK) return r;
  if ((r = grow(s->t_red, s->tw_red, (size_t)A)) != NR_OK) return r;
  if (!s->loss_acc) NR_CHECK_CUDA(cudaMalloc(&s->loss_acc, sizeof(float)));
  if (!s->adam_m) {
    s->n_params_total = s->n_wvol + s->n_table + s->n_mlp + s->n_res;
    NR_CHECK_CUDA(cudaMalloc(&s->adam_m, s->n_params_total * 4));
    NR_CHECK_CUDA(cudaMalloc(&s->adam_v, s->n_params_total * 4));
    NR_CHECK_CUDA(cudaMemsetAsync(s->adam_m, 0, s->n_params_total * 4, st));
    NR_CHECK_CUDA(cudaMemsetAsync(s->adam_v, 0, s->n_params_total * 4, st));
    s->adam_t = 0;
  }
  if (quad) {
    if ((r = grow(s->t_gquad, s->tw_gquad, n_quad)) != NR_OK) return r;
    NR_CHECK_CUDA(cudaMemsetAsync(s->t_gquad, 0, n_quad * sizeof(float4), st));
    const size_t bones = (size_t)kBones * s->wres * s->wres * s->wres;   // the channels that the fold writes
    NR_CHECK_CUDA(cudaMemsetAsync(s->g_wvol + bones, 0, (s->n_wvol - bones) * 4, st));
  } else {
    NR_CHECK_CUDA(cudaMemsetAsync(s->g_wvol, 0, s->n_wvol * 4, st));
  }
  NR_CHECK_CUDA(cudaMemsetAsync(s->g_table, 0, s->n_table * 4, st));
  NR_CHECK_CUDA(cudaMemsetAsync(s->t_wacc, 0, n_acc * A * 4, st));
  NR_CHECK_CUDA(cudaMemsetAsync(s->loss_acc, 0, sizeof(float), st));
  if (refine) {
    if ((r = grow(s->f_dG, s->f_dG_cap, n_dG)) != NR_OK) return r;
    NR_CHECK_CUDA(cudaMemsetAsync(s->f_dG, 0, n_dG * 4, st));
    NR_CHECK_CUDA(cudaMemsetAsync(s->g_ref, 0, s->n_ref * 4, st));
  }

  TrainDev T{};
  T.frame_id = b->frame_id;
  T.px = b->px;
  T.py = b->py;
  T.target = b->target_rgb;
  T.n_rays = b->n_rays;
  T.S = b->n_samples;
  T.ray_mul = ray_multiplier(b->n_rays);
  T.loss_weight = b->loss_weight > 0.f ? b->loss_weight : 1.f;
  T.seed = b->step_seed;
  for (int k = 0; k < 3; ++k) T.bg[k] = b->bg[k];
  T.cams = s->f_cam;
  T.fG = s->f_G;
  T.fbias1 = s->f_bias1;
  T.fomega = s->f_omega;
  T.samp = s->t_samp;
  T.out = s->t_out;
  T.T = s->t_T;
  T.raycnt = s->t_raycnt;
  T.live = s->t_live;
  T.loss = s->loss_acc;
  T.g_table = reinterpret_cast<float2 *>(s->g_table);
  T.g_wvol = s->g_wvol;
  T.g_quad = quad ? s->t_gquad : nullptr;
  T.scratch = s->t_scratch;
  T.wacc = s->t_wacc;
  T.acc_floats = A;
  T.n_frames = (int)s->n_frames;
  T.rw = rows;
  T.dG = refine ? s->f_dG : nullptr;
  T.dG_acc = dG_acc ? 1 : 0;
  T.fl = fl;
  T.pred = b->pred_rgb;
  T.grad_rgb = fwd_only ? nullptr : b->grad_rgb;
  T.forward_only = fwd_only ? 1 : 0;

  train_samples_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(T, s->bmin[0], s->bmin[1], s->bmin[2], s->bmax[0],
                                                                     s->bmax[1], s->bmax[2]);
  NR_CHECK_CUDA(cudaGetLastError());
  if (!fused) {
    const size_t smem_f = smem_w + warps_max * tile_b;
    NR_CHECK_CUDA(cudaFuncSetAttribute(train_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_f));
    train_fwd_kernel<<<blocks, 32 * warps_max, smem_f, st>>>(P, T);
    NR_CHECK_CUDA(cudaGetLastError());
    train_composite_kernel<<<(b->n_rays + 255) / 256, 256, 0, st>>>(T);
    NR_CHECK_CUDA(cudaGetLastError());
    launched += 2;
  }
  if (fwd_only) {
    count_launches(launched + 2);
    if (loss_out) {
      NR_CHECK_CUDA(cudaMemcpyAsync(loss_out, s->loss_acc, sizeof(float), cudaMemcpyDeviceToHost, st));
      NR_CHECK_CUDA(cudaStreamSynchronize(st));
    }
    return NR_OK;
  }
  const size_t smem_b = smem_w + warps_b * tile_b;
  if (fused) {
    NR_CHECK_CUDA(
        cudaFuncSetAttribute(train_bwd_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_b));
    train_bwd_kernel<true><<<blocks, 32 * warps_b, smem_b, st>>>(P, T);
  } else {
    NR_CHECK_CUDA(
        cudaFuncSetAttribute(train_bwd_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_b));
    train_bwd_kernel<false><<<blocks, 32 * warps_b, smem_b, st>>>(P, T);
  }
  NR_CHECK_CUDA(cudaGetLastError());
  if (quad) {
    const int nb = (int)std::min<size_t>(((size_t)kBones * s->wres * s->wres * s->wres + 255) / 256, (size_t)blocks * 8);
    fold_quad_kernel<<<nb, 256, 0, st>>>(s->t_gquad, (int)s->wres, s->g_wvol);
    ++launched;
  }
  reduce_acc_kernel<<<(A + 255) / 256, 256, 0, st>>>(s->t_wacc, (int)n_acc, A, s->t_red);
  ScatterArgs sa{};
  sa.m = master_offsets(s);
  sa.b = s->lay;
  sa.g = res_gamma_dims(s);
  sa.pose_dim = 3 * (int)s->K;
  sa.n_frames = (int)s->n_frames;
  sa.hidden = (int)s->hidden;
  sa.mlp_in = (int)s->mlp_in;
  if (s->res_enabled) {
    scatter_res_kernel<<<(sa.m.n_res + 255) / 256, 256, 0, st>>>(s->t_red, refine ? s->f_omega_o : s->f_omega, sa,
                                                                 s->g_res);
  } else {
    NR_CHECK_CUDA(cudaMemsetAsync(s->g_res, 0, s->n_res * 4, st));
  }
  scatter_mlp_kernel<<<(sa.m.n_mlp + 255) / 256, 256, 0, st>>>(s->t_red, sa, s->g_mlp);
  NR_CHECK_CUDA(cudaGetLastError());
  launched += 5;   // samples, backward, reduction, two scatters
  if (refine && (r = launch_refine_bwd(s, s->f_omega, 3 * kBones, s->f_root, 3, (int)s->n_frames,
                                       dG_acc ? s->t_red + s->lay.total + s->n_frames * kWidth : s->f_dG,
                                       s->t_red + s->lay.total, s->g_ref, st)) != NR_OK)
    return r;
  if (s->cnn_on && (r = cnn_backward(s, st)) != NR_OK) return r;   // dL/dW^c -> CNN_skel
  if (!(b->flags & NR_GRAD_ONLY)) {
    const uint32_t mask = b->train_mask ? b->train_mask : NR_TRAIN_ALL;
    s->adam_t += 1;
    const double c1 = 1.0 / (1.0 - pow((double)b->beta1, (double)s->adam_t));
    const double c2 = 1.0 / (1.0 - pow((double)b->beta2, (double)s->adam_t));
    struct G_ {
      uint32_t bit;
      float *p, *g;
      size_t n, off;
      float scale;
    } groups[4] = {{NR_TRAIN_WVOL, s->wvol, s->g_wvol, s->n_wvol, 0, b->lr_scale[0]},
                   {NR_TRAIN_HASH, s->table, s->g_table, s->n_table, s->n_wvol, b->lr_scale[1]},
                   {NR_TRAIN_MLP, s->mlp, s->g_mlp, s->n_mlp, s->n_wvol + s->n_table, b->lr_scale[2]},
                   {NR_TRAIN_RES, s->res, s->g_res, s->n_res, s->n_wvol + s->n_table + s->n_mlp, b->lr_scale[3]}};
    for (const auto &g : groups) {
      if (!(mask & g.bit) || (g.bit == NR_TRAIN_RES && !s->res_enabled)) continue;
      if (g.bit == NR_TRAIN_WVOL && s->cnn_on) continue;   // the volume is generated, not stored
      const float lr = b->lr * (g.scale > 0.f ? g.scale : 1.f);
      const int nb = (int)std::min<size_t>((g.n + 255) / 256, (size_t)blocks * 8);
      adam_kernel<<<nb, 256, 0, st>>>(g.p, g.g, s->adam_m + g.off, s->adam_v + g.off, g.n, lr, b->beta1, b->beta2,
                                      b->eps, (float)c1, (float)c2);
      ++launched;
    }
    if (s->cnn_on && (mask & NR_TRAIN_CNN)) {
      s->cnn_t += 1;
      const double q1 = 1.0 / (1.0 - pow((double)b->beta1, (double)s->cnn_t));
      const double q2 = 1.0 / (1.0 - pow((double)b->beta2, (double)s->cnn_t));
      const float lr = b->lr * (b->lr_scale_cnn > 0.f ? b->lr_scale_cnn : 1.f);
      const int nb = (int)std::min<size_t>((s->n_cnn + 255) / 256, (size_t)blocks * 8);
      adam_kernel<<<nb, 256, 0, st>>>(s->cnn, s->g_cnn, s->cnn_m, s->cnn_v, s->n_cnn, lr, b->beta1, b->beta2, b->eps,
                                      (float)q1, (float)q2);
      ++launched;
      s->cnn_dirty = true;
    }
    if (refine && (mask & NR_TRAIN_REFINER)) {
      s->ref_t += 1;
      const double r1 = 1.0 / (1.0 - pow((double)b->beta1, (double)s->ref_t));
      const double r2 = 1.0 / (1.0 - pow((double)b->beta2, (double)s->ref_t));
      const float lr = b->lr * (b->lr_scale_refiner > 0.f ? b->lr_scale_refiner : 1.f);
      const int nb = (int)std::min<size_t>((s->n_ref + 255) / 256, (size_t)blocks * 8);
      adam_kernel<<<nb, 256, 0, st>>>(s->ref, s->g_ref, s->ref_m, s->ref_v, s->n_ref, lr, b->beta1, b->beta2, b->eps,
                                      (float)r1, (float)r2);
      ++launched;
      s->pose_dirty = s->pose_set;   // the current pose's refinement moved
    }
    NR_CHECK_CUDA(cudaGetLastError());
    s->params_dirty = true;
    s->bias_dirty = true;
  }
  count_launches(launched);
  if (loss_out) {
    NR_CHECK_CUDA(cudaMemcpyAsync(loss_out, s->loss_acc, sizeof(float), cudaMemcpyDeviceToHost, st));
    NR_CHECK_CUDA(cudaStreamSynchronize(st));
  }
  return NR_OK;
}

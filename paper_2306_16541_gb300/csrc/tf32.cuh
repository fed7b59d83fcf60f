// tf32.cuh -- float32-accurate warp-level layers on the tensor cores, shared by the
// training kernels and the float32 render tier on the tensor cores.
//
// Each float32 operand is split into two TF32 parts (x = hi + lo, both exact in TF32); a
// product x y is taken as hi_x lo_y + lo_x hi_y + hi_x hi_y (three m16n8k8 MMAs, the dropped
// lo_x lo_y term lies below float32 rounding), so the layers keep float32 accuracy.
//
// A warp owns a tile of 32 samples.  The input of a layer lies in shared memory as rows of 32
// samples (a row per feature); the output leaves the MMAs in registers and becomes the next
// input in the same place, so a layer touches no global memory.  The product is C = X W^T with
// M = the samples (two 16-row tiles), N = the outputs in tiles of 8, K = the inputs in steps of
// 8: two row tiles share each weight fragment, so that one fragment (two 4-byte loads and two
// splits) feeds six MMAs.  m16n8k8 TF32 takes two cycles an SM (measured: 2.0), which bounds a
// 64 x 64 layer to 768 cycles a tile; the loads and splits need about a third of the issue slots.
#pragma once

#include "common.cuh"

namespace nr {

// ------------------------------------------------------------------ tiles
constexpr int kTileRow = 32;                     // floats a row: one per sample
constexpr int kTileFloats = kWidth * kTileRow;   // a tile of 64 rows
constexpr int kGamRows = 40;                     // rows of gamma(x_skel): the 39 used and a zero row

// Sample s of row r: the row's eight 16-byte chunks are permuted by the low bits of r, so that
// the accesses below -- one row by all lanes, four rows by eight samples (fragments), eight rows
// by four chunks (weight gradients) -- each touch 32 distinct banks.
__device__ __forceinline__ int tile_sw(int r) { return ((r & 1) << 2) | (r & 2); }
__device__ __forceinline__ int frag_at(int r, int s) {
  return r * kTileRow + ((((s >> 2) ^ tile_sw(r)) << 2) | (s & 3));
}

// A lane's places in the fragments: g = lane / 4, t = lane % 4.  Fragment columns 2t and 2t + 1
// stand for features t and t + 4 of their block of eight (the columns of W are taken in that
// order), so that an output block is the input block of the next layer, lane by lane.
struct FragLane {
  int g, t;
  int a[4];        // offsets of samples g, g + 8, g + 16, g + 24 in row t of a block
  int f0, b0;      // weight offsets in an 8 x 8 block: forward (then f0 ^ 4), backward (then b1)
  int b1;
};

__device__ __forceinline__ FragLane frag_lane() {
  FragLane L;
  const int lane = threadIdx.x & 31;
  L.g = lane >> 2;
  L.t = lane & 3;
#pragma unroll
  for (int q = 0; q < 4; ++q) L.a[q] = frag_at(L.t, 8 * q + L.g);
  const int p = (L.g >> 1) | ((L.g & 1) << 2);   // the feature of column g
  L.f0 = p * 8 + (L.t ^ (p & 4));
  L.b0 = L.t * 8 + p;
  L.b1 = (L.t + 4) * 8 + (p ^ 4);
  return L;
}

// ---------------------------------------------------------------- weights
// The shared-memory copy of the weights: W[out][in] in 8 x 8 blocks, block (ob, ib) at
// (ob IB + ib) 64, element (o, i) of a block at o 8 + (i ^ (o & 4)).  One copy serves both
// directions without bank conflicts: a forward fragment reads eight rows by four columns, a
// backward fragment four rows by eight columns.  The gamma inputs take kGamRows columns, the four
// outputs of a last layer a block of eight rows with zeros.
struct FragLay {
  int r1, r2, r3, r4, r5, c0, ch[kMaxHidden], cl;
  int r2b, r3b, r4b, r5b, c0b, chb[kMaxHidden], clb;
  int total;   // floats
};

__host__ __device__ inline FragLay frag_layout(int H) {
  FragLay p{};
  int o = 0;
  auto take = [&](int n) {
    const int r = o;
    o += n;
    return r;
  };
  p.r1 = take(kWidth * kGamRows);
  p.r2 = take(kWidth * kWidth);
  p.r3 = take(kWidth * kWidth);
  p.r4 = take(kWidth * (kWidth + kGamRows));
  p.r5 = take(8 * kWidth);
  p.c0 = take(kWidth * kMlpIn);
  for (int l = 0; l < H - 1; ++l) p.ch[l] = take(kWidth * kWidth);
  p.cl = take(8 * kWidth);
  p.r2b = take(kWidth);
  p.r3b = take(kWidth);
  p.r4b = take(kWidth);
  p.r5b = take(4);
  p.c0b = take(kWidth);
  for (int l = 0; l < H - 1; ++l) p.chb[l] = take(kWidth);
  p.clb = take(4);
  p.total = o;
  return p;
}

// Fills the shared copy from the transposed float32 blob ([in][out] per layer).  Block-collective.
__device__ __forceinline__ void stage_frag_weights(const float *__restrict__ blob, const BlobLayout &b,
                                                   const FragLay &p, int H, float *sW) {
  auto mat = [&](int src, int in, int out, int dst, int IB, int ib0) {
    const int rows = (out + 7) & ~7;
    for (int e = threadIdx.x; e < in * rows; e += blockDim.x) {
      const int i = e / rows, o = e - i * rows;
      sW[dst + ((o >> 3) * IB + ib0 + (i >> 3)) * 64 + (o & 7) * 8 + ((i & 7) ^ (o & 4))] =
          o < out ? __ldg(blob + src + i * out + o) : 0.f;
    }
  };
  auto vec = [&](int src, int n, int dst) {
    for (int e = threadIdx.x; e < n; e += blockDim.x) sW[dst + e] = __ldg(blob + src + e);
  };
  mat(b.r1, kGamRows, kWidth, p.r1, kGamRows / 8, 0);
  mat(b.r2, kWidth, kWidth, p.r2, 8, 0);
  mat(b.r3, kWidth, kWidth, p.r3, 8, 0);
  mat(b.r4, kWidth + kGamRows, kWidth, p.r4, 8 + kGamRows / 8, 0);
  mat(b.r5, kWidth, 4, p.r5, 8, 0);
  mat(b.c0, kMlpIn, kWidth, p.c0, kMlpIn / 8, 0);
  vec(b.r2b, kWidth, p.r2b);
  vec(b.r3b, kWidth, p.r3b);
  vec(b.r4b, kWidth, p.r4b);
  vec(b.r5b, 4, p.r5b);
  vec(b.c0b, kWidth, p.c0b);
  for (int l = 0; l < H - 1; ++l) {
    mat(b.ch[l], kWidth, kWidth, p.ch[l], 8, 0);
    vec(b.chb[l], kWidth, p.chb[l]);
  }
  mat(b.cl, kWidth, 4, p.cl, 8, 0);
  vec(b.clb, 4, p.clb);
}

// ------------------------------------------------------------------- MMAs
// x = hi + lo: hi = x rounded to TF32 (to nearest, ties away: add half a unit of the last kept
// bit to the magnitude, clear the rest), lo = x - hi, whose low bits the MMA ignores once the
// same half unit is added.  For finite x the values of cvt.rna.tf32.f32, whose two conversions
// take 3.0 cycles an SM against 1.3 for integer and float32 operations (measured).
// x = NaN or infinity: x - hi is the NaN of the arithmetic, 0x7fffffff, whatever hi became (the add
// carries a NaN of that form into -0).  There the half unit would do the same to lo; the signed
// maximum keeps it, and is lo + 0x1000 for every other value, so that one NaN part carries the
// operand through the products (it adds nothing measurable: a 2^18-ray step 133.88 ms without it
// and 133.88 with, a 2400-ray step 1.378 and 1.381).
__device__ __forceinline__ void tf32_split(float x, uint32_t &hi, uint32_t &lo) {
  hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  const uint32_t d = __float_as_uint(x - __uint_as_float(hi));
  lo = (uint32_t)max((int)(d + 0x1000u), (int)d);
}

__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// c[m][n] += X B over KB blocks of eight input rows of `tile`.  B's fragment of (block ks, tile
// n) lies at W + ks ks_step + n n_step, its two values at offsets w0 and w1.  c[m][n] holds, for
// samples 16m + g (values 0, 1) and 16m + g + 8 (2, 3), features 8n + t and 8n + t + 4.
// The order of the products and of the steps is fixed, so a layer gives the same bits wherever
// it runs.  Every lane of the warp must take part.
template <int NT>
__device__ __forceinline__ void frag_mma(const FragLane &L, const float *tile, int kb, const float *W, int ks_step,
                                         int n_step, int w0, int w1, float (&c)[2][NT][4]) {
#pragma unroll 1
  for (int ks = 0; ks < kb; ++ks) {
    const float *x = tile + ks * 8 * kTileRow;
    uint32_t ah[2][4], al[2][4];
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      tf32_split(x[L.a[2 * m]], ah[m][0], al[m][0]);
      tf32_split(x[L.a[2 * m + 1]], ah[m][1], al[m][1]);
      tf32_split(x[L.a[2 * m] + 4 * kTileRow], ah[m][2], al[m][2]);
      tf32_split(x[L.a[2 * m + 1] + 4 * kTileRow], ah[m][3], al[m][3]);
    }
    const float *w = W + ks * ks_step;
    // two output tiles at a time: four independent accumulators lie between the dependent MMAs
    // of one (21 cycles apart at best)
#pragma unroll
    for (int n = 0; n < NT; n += 2) {
      uint32_t bh[2][2], bl[2][2];
#pragma unroll
      for (int e = 0; e < 2; ++e)
        if (n + e < NT) {
          tf32_split(w[(n + e) * n_step + w0], bh[e][0], bl[e][0]);
          tf32_split(w[(n + e) * n_step + w1], bh[e][1], bl[e][1]);
        }
#pragma unroll
      for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
          for (int m = 0; m < 2; ++m)
            if (n + e < NT) mma_tf32(c[m][n + e], p == 1 ? al[m] : ah[m], p == 0 ? bl[e] : bh[e]);
    }
  }
}

template <int NT>
__device__ __forceinline__ void frag_zero(float (&c)[2][NT][4]) {
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q) c[m][n][q] = 0.f;
}

// Forward product of a layer: W at its shared copy of IB input blocks, KB of them from block ib0.
template <int NT>
__device__ __forceinline__ void frag_fwd(const FragLane &L, const float *tile, int kb, const float *W, int IB, int ib0,
                                         float (&c)[2][NT][4]) {
  frag_mma<NT>(L, tile, kb, W + ib0 * 64, 64, IB * 64, L.f0, L.f0 ^ 4, c);
}

// Backward product, out[s][i] = sum_o delta[s][o] W[o][i] over KB output blocks, for the NT input
// blocks from ib0.
template <int NT>
__device__ __forceinline__ void frag_back(const FragLane &L, const float *tile, int kb, const float *W, int IB, int ib0,
                                          float (&c)[2][NT][4]) {
  frag_mma<NT>(L, tile, kb, W + ib0 * 64, IB * 64, 64, L.b0, L.b1, c);
}

// c into the tile's rows (every lane has read the tile's old rows by then).
template <int NT>
__device__ __forceinline__ void frag_store(const FragLane &L, const float (&c)[2][NT][4], float *tile) {
  __syncwarp();
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      float *r = tile + n * 8 * kTileRow;
      r[L.a[2 * m]] = c[m][n][0];
      r[L.a[2 * m] + 4 * kTileRow] = c[m][n][1];
      r[L.a[2 * m + 1]] = c[m][n][2];
      r[L.a[2 * m + 1] + 4 * kTileRow] = c[m][n][3];
    }
  __syncwarp();
}

// c = relu(c + bias) with the bias of a shared vector.
__device__ __forceinline__ void frag_relu(const FragLane &L, const float *b, float (&c)[2][8][4]) {
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    const float v0 = b[8 * n + L.t], v1 = b[8 * n + L.t + 4];
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      c[m][n][0] = fmaxf(c[m][n][0] + v0, 0.f);
      c[m][n][1] = fmaxf(c[m][n][1] + v1, 0.f);
      c[m][n][2] = fmaxf(c[m][n][2] + v0, 0.f);
      c[m][n][3] = fmaxf(c[m][n][3] + v1, 0.f);
    }
  }
}

// The same with row `fr` of per-frame biases, each sample's row taken from the lane that owns it.
__device__ __forceinline__ void frag_relu_rows(const FragLane &L, const float *__restrict__ fb, int fr,
                                               float (&c)[2][8][4]) {
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float *b = fb + (size_t)__shfl_sync(0xffffffffu, fr, 16 * m + 8 * h + L.g) * kWidth + L.t;
#pragma unroll
      for (int n = 0; n < 8; ++n) {
        c[m][n][2 * h] = fmaxf(c[m][n][2 * h] + b[8 * n], 0.f);
        c[m][n][2 * h + 1] = fmaxf(c[m][n][2 * h + 1] + b[8 * n + 4], 0.f);
      }
    }
}

// The first `rows` rows of the tile to or from a global image of it (16-byte chunks in order).
__device__ __forceinline__ void tile_save(const float *tile, float *img, int rows) {
  const int lane = threadIdx.x & 31;
#pragma unroll 4
  for (int e = lane; e < rows * 8; e += 32) reinterpret_cast<float4 *>(img)[e] = reinterpret_cast<const float4 *>(tile)[e];
}
__device__ __forceinline__ void tile_load(float *tile, const float *img, int rows) {
  const int lane = threadIdx.x & 31;
  __syncwarp();   // the lanes' reads of the old rows, and their parts of the image
#pragma unroll 5
  for (int e = lane; e < rows * 8; e += 32) reinterpret_cast<float4 *>(tile)[e] = reinterpret_cast<const float4 *>(img)[e];
  __syncwarp();
}

// The last layer of an MLP: the four outputs of each lane's sample, bias added, through rows
// 0..3 of the tile.
__device__ __forceinline__ void frag_out4(const FragLane &L, float *tile, const float *W, const float *b,
                                          float (&o)[4]) {
  float c[2][1][4];
  frag_zero(c);
  frag_fwd<1>(L, tile, 8, W, 8, 0, c);
  const float v = b[L.t];
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    c[m][0][0] += v;
    c[m][0][2] += v;
    c[m][0][1] = c[m][0][3] = 0.f;
  }
  frag_store<1>(L, c, tile);
#pragma unroll
  for (int k = 0; k < 4; ++k) o[k] = tile[frag_at(k, threadIdx.x & 31)];
  __syncwarp();
}

}  // namespace nr

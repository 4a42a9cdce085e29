// Training of the learned predictor on the GPU (not in the paper).
//
// Samples come from the encoder (12 floats per reference slot: 8 features, 3
// target displacements, valid flag).  The valid ones are compacted in order
// (flags, scan, scatter).  mlp_steps_kernel then runs every SGD step of the
// call in one cooperative launch, two grid barriers per step (gradients of
// the sample tiles; their sum and its norm; every block updates its own copy
// of the weights).  Every sum has an order fixed by the batch and the number
// of blocks, so training is deterministic on a GPU.
// Loss: (1/B) sum_i sum_a (o_ia - y_ia)^2.
#include "codec.cuh"

using namespace tera;

namespace {

constexpr int kDense = 11;     // dense sample: 8 features + 3 targets

// late[0]: a wait of the scan was given up (cleared here); late[1]: valid samples.
__global__ void sample_flags_kernel(const float* __restrict__ samples, u64 n, u32* __restrict__ flags,
                                    u32* __restrict__ late) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *late = 0;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x)
    flags[i] = samples[i * kSampleFloats + 11] != 0.0f ? 1u : 0u;
}

__global__ void sample_compact_kernel(const float* __restrict__ samples, u64 n,
                                      const u32* __restrict__ flags, const u32* __restrict__ pos,
                                      float* __restrict__ dense, u32* late) {
  if (*late) return;  // positions are missing
  if (blockIdx.x == 0 && threadIdx.x == 0) late[1] = pos[n];
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x) {
    if (!flags[i]) continue;
    const float* s = samples + i * kSampleFloats;
    float* d = dense + (u64)pos[i] * kDense;
    for (int k = 0; k < kDense; ++k) d[k] = s[k];
  }
}

// ---------------- the training kernel ----------------
//
// A block of four warps takes tiles of 32 R samples: lane l holds samples l
// and (R = 2) l + 32, a warp a quarter of the neurons.  A tile is three 32 R x
// 64 x 64 products (second layer, its backward pass, the gradient of W2) and
// small ones around them: 13.9 K multiply-adds a sample, FP32 because the
// weights and gradients are (the tensor cores round operands to 19 bits or
// fewer).  What decides the layout is shared memory: a load returns 128 bytes
// a clock to the SM, so a load whose lanes differ costs four clocks for 16
// bytes a lane, and one whose lanes agree costs one.  Weights (and, for the
// gradient of W2, the errors) are therefore read by all lanes together and
// serve 8 R multiply-adds a lane; with 4 x 2 register tiles and no common
// operand a tile of 32 samples took 5.2 us, three times its FP32 time.
// The gradient's sums stay in registers over a block's tiles.
//
// Measured at batch 8192 (128 tiles of 64): 15.8 us a step, one kernel for all
// steps; with a kernel of one thread per sample, one that summed the blocks'
// gradients and one block for the update it was 76 us (100 steps: 7.67 ->
// 1.67 ms, compaction included).  A step is about 9 us of the tile (its shared
// memory wavefronts alone are 11 K clocks, its issue slots 10.4 K) and 6 us of
// the two grid barriers, the sum over the blocks and the update.
//
// R = 2 halves the loads per multiply-add; R = 1 spreads a batch that would
// leave SMs without a tile (one 64-sample tile takes as long on one SM as two
// 32-sample tiles one after the other).

constexpr int kTrainThreads = 128;
constexpr int kTrainPerSm = 2;     // blocks per SM
constexpr int kRow = kMlpH + 4;    // padded row: float4 columns of 8 rows fall in distinct banks
constexpr int kXRow = 12;
constexpr int kGradStride = (kMlpParams + 3) & ~3;  // one block's gradient, 16-byte rows
constexpr int kSmemW = kMlpParams + 4 * kMlpH + 1;  // weights with W2's rows padded to kRow
// per warp: gradients of W1, W3, b1, b2 and b3 over its quarter of the samples
constexpr int kSmall = 512 + 192 + 64 + 64 + 4;

template <int R>
struct TrainSmem {
  float W[(kSmemW + 3) & ~3];
  float x[32 * R * kXRow];  // features and targets
  float a1[32 * R * kRow];
  float a2[32 * R * kRow];
  float g2[32 * R * kRow];
  float g1[32 * R * kRow];
  float go[32 * R * 4];
  float po[4 * 32 * R * 4];  // each warp's share of the outputs
  float red[kTrainThreads];
  float wsum[kTrainThreads / 32];
  float step;
  int late;
};
static_assert(2 * 32 * kRow >= 4 * kSmall, "a1 and a2 hold the warps' small gradients");

// Where parameter q lies in the padded weights.
__device__ __forceinline__ int padded(int q) {
  if (q < kMlpW2) return q;
  const int row = q < kMlpB2 ? (q - kMlpW2) / kMlpH : kMlpH;
  return q + 4 * row;
}
constexpr int kPB2 = kMlpB2 + 4 * kMlpH, kPW3 = kMlpW3 + 4 * kMlpH, kPB3 = kMlpB3 + 4 * kMlpH;

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

struct TrainArgs {
  const float* dense;  // [nv * kDense] valid samples
  u64 nv;
  u64 batch;
  int steps;
  float lr, clip;
  float* params;       // read, and written when the steps are done (null: grad_out alone)
  const float* params_in;
  float* partial;      // [blocks * kGradStride]
  float* grad;         // [kGradStride] (mlp_grad: the caller's)
  float* ssq;          // [blocks] squares of each block's slice of the gradient
  u32* barrier;        // zero at launch
  DevStatus* st;
};

// Every block of the (cooperative, so co-resident) launch arrives and waits
// for the others; the wait gives up after a minute of the global timer
// (TERA_ETIMEOUT, false in every thread of the block).
__device__ __forceinline__ bool grid_barrier(const TrainArgs& A, int* s_late, u32 target) {
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" : : "l"(A.barrier) : "memory");
    u32 v;
    u64 t0, t;
    int late = 0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (u64 poll = 1;; ++poll) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(A.barrier) : "memory");
      if ((int)(v - target) >= 0) break;  // the count may wrap
      if ((poll & 255) == 0) {
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > 60000000000ull || poll > (1ull << 32)) {
          latch(A.st, TERA_ETIMEOUT);
          late = 1;
          break;
        }
      }
    }
    *s_late = late;
  }
  __syncthreads();
  return *s_late == 0;
}

// Value i (sample i / kDense) of tile `tile` of the step that starts at valid
// sample `start`; zero past the batch.
__device__ __forceinline__ float dense_at(const TrainArgs& A, u64 start, u64 tile, int samples,
                                          int i) {
  const u64 s = tile * (u64)samples + (u64)(i / kDense);
  if (s >= A.batch) return 0.0f;
  u64 r = start + s;
  if (r >= A.nv) r = r - A.nv < A.nv ? r - A.nv : r % A.nv;
  return __ldg(A.dense + r * kDense + i % kDense);
}

__device__ __forceinline__ float fma4(const float4 a, const float4 b, float acc) {
  acc = __fmaf_rn(a.x, b.x, acc);
  acc = __fmaf_rn(a.y, b.y, acc);
  acc = __fmaf_rn(a.z, b.z, acc);
  return __fmaf_rn(a.w, b.w, acc);
}

__device__ __forceinline__ float relu(float v) { return v > 0.0f ? v : 0.0f; }

template <int R>
__global__ void __launch_bounds__(kTrainThreads, kTrainPerSm) mlp_steps_kernel(TrainArgs A) {
  extern __shared__ __align__(16) uint8_t train_smem[];
  TrainSmem<R>& S = *reinterpret_cast<TrainSmem<R>*>(train_smem);
  constexpr int kTile = 32 * R;                                        // samples of a tile
  constexpr int kX = (kTile * kDense + kTrainThreads - 1) / kTrainThreads;  // its values a thread
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int n0 = 16 * warp;  // this warp's neurons
  const u32 G = gridDim.x;
  const u64 tiles = (A.batch + kTile - 1) / kTile;
  const float scale = __fdiv_rn(2.0f, (float)A.batch);
  for (int q = t; q < kMlpParams; q += kTrainThreads) S.W[padded(q)] = A.params_in[q];
  u32 arrivals = 0;
  u64 start = 0;
  // this block's first tile of the first step; later ones are read one ahead
  float xr[kX];
#pragma unroll
  for (int i = 0; i < kX; ++i) {
    const int e = t + i * kTrainThreads;
    xr[i] = e < kTile * kDense ? dense_at(A, start, blockIdx.x, kTile, e) : 0.0f;
  }
  for (int step = 0; step < A.steps; ++step) {
    u64 next_start = start + A.batch;
    if (next_start >= A.nv) next_start %= A.nv;
    float w2[16][2] = {};               // gradient of W2: rows n0 + c, columns lane, lane + 32
    float w1[2][8] = {}, w3[2][3] = {}; // of W1 rows and W3 columns lane, lane + 32
    float b1[2] = {}, b2[2] = {}, b3[3] = {};
    for (u64 tile = blockIdx.x; tile < tiles; tile += G) {
#pragma unroll
      for (int i = 0; i < kX; ++i) {
        const int e = t + i * kTrainThreads;
        if (e < kTile * kDense) S.x[e / kDense * kXRow + e % kDense] = xr[i];
      }
      __syncthreads();
      {  // the next tile's samples arrive while this one is computed
        const bool more = tile + G < tiles;
#pragma unroll
        for (int i = 0; i < kX; ++i) {
          const int e = t + i * kTrainThreads;
          if (e < kTile * kDense)
            xr[i] = dense_at(A, more ? start : next_start, more ? tile + G : (u64)blockIdx.x,
                             kTile, e);
        }
      }
      // first layer
      {
        float4 xa[R], xb[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          xa[r] = ld4(S.x + (lane + 32 * r) * kXRow);
          xb[r] = ld4(S.x + (lane + 32 * r) * kXRow + 4);
        }
#pragma unroll
        for (int c = 0; c < 16; c += 4) {
          float h[R][4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float* w = S.W + kMlpW1 + (n0 + c + j) * kMlpIn;
            const float4 wa = ld4(w), wb = ld4(w + 4);
            const float bias = S.W[kMlpB1 + n0 + c + j];
#pragma unroll
            for (int r = 0; r < R; ++r) h[r][j] = relu(fma4(wb, xb[r], fma4(wa, xa[r], bias)));
          }
#pragma unroll
          for (int r = 0; r < R; ++r)
            *reinterpret_cast<float4*>(S.a1 + (lane + 32 * r) * kRow + n0 + c) =
                make_float4(h[r][0], h[r][1], h[r][2], h[r][3]);
        }
      }
      __syncthreads();
      // second layer and this warp's share of the outputs
      float h2[R][16];
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const float bias = S.W[kPB2 + n0 + c];
#pragma unroll
        for (int r = 0; r < R; ++r) h2[r][c] = bias;
      }
#pragma unroll 2
      for (int k = 0; k < kMlpH; k += 4) {
        float4 a[R];
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] = ld4(S.a1 + (lane + 32 * r) * kRow + k);
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const float4 w = ld4(S.W + kMlpW2 + (n0 + c) * kRow + k);
#pragma unroll
          for (int r = 0; r < R; ++r) h2[r][c] = fma4(w, a[r], h2[r][c]);
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float o[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int c = 0; c < 16; c += 4) {
#pragma unroll
          for (int j = 0; j < 4; ++j) h2[r][c + j] = relu(h2[r][c + j]);
          const float4 h = make_float4(h2[r][c], h2[r][c + 1], h2[r][c + 2], h2[r][c + 3]);
          *reinterpret_cast<float4*>(S.a2 + (lane + 32 * r) * kRow + n0 + c) = h;
#pragma unroll
          for (int a = 0; a < 3; ++a) o[a] = fma4(ld4(S.W + kPW3 + a * kMlpH + n0 + c), h, o[a]);
        }
        *reinterpret_cast<float4*>(S.po + (warp * kTile + lane + 32 * r) * 4) =
            make_float4(o[0], o[1], o[2], 0.0f);
      }
      __syncthreads();
      // the outputs' errors, back through W3
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int s = lane + 32 * r;
        float o[3] = {S.W[kPB3], S.W[kPB3 + 1], S.W[kPB3 + 2]};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const float4 v = ld4(S.po + (w * kTile + s) * 4);
          o[0] += v.x;
          o[1] += v.y;
          o[2] += v.z;
        }
        const bool live = tile * kTile + s < A.batch;
        float go[3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
          go[a] = live ? __fmul_rn(__fsub_rn(o[a], S.x[s * kXRow + kMlpIn + a]), scale) : 0.0f;
        if (warp == 0)
          *reinterpret_cast<float4*>(S.go + 4 * s) = make_float4(go[0], go[1], go[2], 0.0f);
#pragma unroll
        for (int c = 0; c < 16; c += 4) {
          const float4 u = ld4(S.W + kPW3 + n0 + c), v = ld4(S.W + kPW3 + kMlpH + n0 + c),
                       w = ld4(S.W + kPW3 + 2 * kMlpH + n0 + c);
          float4 g;
          g.x = h2[r][c] > 0.0f ? __fmaf_rn(go[2], w.x, __fmaf_rn(go[1], v.x, go[0] * u.x)) : 0.0f;
          g.y = h2[r][c + 1] > 0.0f ? __fmaf_rn(go[2], w.y, __fmaf_rn(go[1], v.y, go[0] * u.y)) : 0.0f;
          g.z = h2[r][c + 2] > 0.0f ? __fmaf_rn(go[2], w.z, __fmaf_rn(go[1], v.z, go[0] * u.z)) : 0.0f;
          g.w = h2[r][c + 3] > 0.0f ? __fmaf_rn(go[2], w.w, __fmaf_rn(go[1], v.w, go[0] * u.w)) : 0.0f;
          *reinterpret_cast<float4*>(S.g2 + s * kRow + n0 + c) = g;
        }
      }
      __syncthreads();
      // back through W2
      {
        float acc[R][16] = {};
#pragma unroll 1
        for (int j = 0; j < kMlpH; j += 4) {
          float g[R][4];
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const float4 v = ld4(S.g2 + (lane + 32 * r) * kRow + j);
            g[r][0] = v.x;
            g[r][1] = v.y;
            g[r][2] = v.z;
            g[r][3] = v.w;
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < 16; c += 4) {
              const float4 w = ld4(S.W + kMlpW2 + (j + i) * kRow + n0 + c);
#pragma unroll
              for (int r = 0; r < R; ++r) {
                acc[r][c] = __fmaf_rn(w.x, g[r][i], acc[r][c]);
                acc[r][c + 1] = __fmaf_rn(w.y, g[r][i], acc[r][c + 1]);
                acc[r][c + 2] = __fmaf_rn(w.z, g[r][i], acc[r][c + 2]);
                acc[r][c + 3] = __fmaf_rn(w.w, g[r][i], acc[r][c + 3]);
              }
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int c = 0; c < 16; c += 4) {
            const int at = (lane + 32 * r) * kRow + n0 + c;
            const float4 h = ld4(S.a1 + at);
            *reinterpret_cast<float4*>(S.g1 + at) =
                make_float4(h.x > 0.0f ? acc[r][c] : 0.0f, h.y > 0.0f ? acc[r][c + 1] : 0.0f,
                            h.z > 0.0f ? acc[r][c + 2] : 0.0f, h.w > 0.0f ? acc[r][c + 3] : 0.0f);
          }
      }
      // gradient of W2
#pragma unroll 2
      for (int s = 0; s < kTile; ++s) {
        const float ha = S.a1[s * kRow + lane], hb = S.a1[s * kRow + lane + 32];
#pragma unroll
        for (int c = 0; c < 16; c += 4) {
          const float4 g = ld4(S.g2 + s * kRow + n0 + c);
          w2[c][0] = __fmaf_rn(g.x, ha, w2[c][0]);
          w2[c][1] = __fmaf_rn(g.x, hb, w2[c][1]);
          w2[c + 1][0] = __fmaf_rn(g.y, ha, w2[c + 1][0]);
          w2[c + 1][1] = __fmaf_rn(g.y, hb, w2[c + 1][1]);
          w2[c + 2][0] = __fmaf_rn(g.z, ha, w2[c + 2][0]);
          w2[c + 2][1] = __fmaf_rn(g.z, hb, w2[c + 2][1]);
          w2[c + 3][0] = __fmaf_rn(g.w, ha, w2[c + 3][0]);
          w2[c + 3][1] = __fmaf_rn(g.w, hb, w2[c + 3][1]);
        }
      }
      __syncthreads();
      // the small gradients, each warp over its quarter of the samples
#pragma unroll 2
      for (int s = warp * (kTile / 4); s < (warp + 1) * (kTile / 4); ++s) {
        const float4 xa = ld4(S.x + s * kXRow), xb = ld4(S.x + s * kXRow + 4), go = ld4(S.go + 4 * s);
        b3[0] += go.x;
        b3[1] += go.y;
        b3[2] += go.z;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float g = S.g1[s * kRow + lane + 32 * i], h = S.a2[s * kRow + lane + 32 * i];
          b1[i] += g;
          b2[i] += S.g2[s * kRow + lane + 32 * i];
          w1[i][0] = __fmaf_rn(g, xa.x, w1[i][0]);
          w1[i][1] = __fmaf_rn(g, xa.y, w1[i][1]);
          w1[i][2] = __fmaf_rn(g, xa.z, w1[i][2]);
          w1[i][3] = __fmaf_rn(g, xa.w, w1[i][3]);
          w1[i][4] = __fmaf_rn(g, xb.x, w1[i][4]);
          w1[i][5] = __fmaf_rn(g, xb.y, w1[i][5]);
          w1[i][6] = __fmaf_rn(g, xb.z, w1[i][6]);
          w1[i][7] = __fmaf_rn(g, xb.w, w1[i][7]);
          w3[i][0] = __fmaf_rn(go.x, h, w3[i][0]);
          w3[i][1] = __fmaf_rn(go.y, h, w3[i][1]);
          w3[i][2] = __fmaf_rn(go.z, h, w3[i][2]);
        }
      }
      __syncthreads();
    }
    // the block's gradient (blocks beyond the tiles do not exist: G <= tiles);
    // the small ones' four shares meet in shared memory, in parameter order:
    // W1 | b1 | b2 | W3 | b3
    {
      float* out = A.partial + (u64)blockIdx.x * kGradStride;
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        __stcg(out + kMlpW2 + (n0 + c) * kMlpH + lane, w2[c][0]);
        __stcg(out + kMlpW2 + (n0 + c) * kMlpH + lane + 32, w2[c][1]);
      }
      float* sm = S.a1 + warp * kSmall;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int j = lane + 32 * i;
        *reinterpret_cast<float4*>(sm + 8 * j) = make_float4(w1[i][0], w1[i][1], w1[i][2], w1[i][3]);
        *reinterpret_cast<float4*>(sm + 8 * j + 4) =
            make_float4(w1[i][4], w1[i][5], w1[i][6], w1[i][7]);
        sm[512 + j] = b1[i];
        sm[576 + j] = b2[i];
#pragma unroll
        for (int a = 0; a < 3; ++a) sm[640 + a * kMlpH + j] = w3[i][a];
      }
      if (lane < 3) sm[832 + lane] = lane == 0 ? b3[0] : (lane == 1 ? b3[1] : b3[2]);
      __syncthreads();
      for (int q = t; q < 835; q += kTrainThreads) {
        const float v = S.a1[q] + S.a1[kSmall + q] + S.a1[2 * kSmall + q] + S.a1[3 * kSmall + q];
        __stcg(out + (q < 576 ? q : q + kMlpB2 - 576), v);
      }
    }
    arrivals += G;
    if (!grid_barrier(A, &S.late, arrivals)) return;
    // the sum over the blocks of this block's slice of the gradient: row
    // groups of consecutive blocks, each added in order with kFlight loads in
    // flight, then the groups in order
    {
      constexpr int kFlight = 20;
      const int chunk = (kMlpParams + (int)G - 1) / (int)G;
      const int q0 = (int)blockIdx.x * chunk;
      const int n = kMlpParams - q0 < chunk ? (kMlpParams - q0 > 0 ? kMlpParams - q0 : 0) : chunk;
      const int groups = chunk < kTrainThreads ? kTrainThreads / chunk : 1;
      const int rows = ((int)G + groups - 1) / groups;
      const int rg = groups > 1 ? t / chunk : 0;
      const int r0 = rg * rows, r1 = r0 + rows < (int)G ? r0 + rows : (int)G;
      float ss = 0.0f;
      for (int c = groups > 1 ? t % chunk : t; c < n && rg < groups; c += kTrainThreads) {
        const float* src = A.partial + q0 + c;
        float acc = 0.0f;
        for (int r = r0; r < r1; r += kFlight) {
          float v[kFlight];
#pragma unroll
          for (int i = 0; i < kFlight; ++i)
            v[i] = r + i < r1 ? __ldcg(src + (u64)(r + i) * kGradStride) : 0.0f;
#pragma unroll
          for (int i = 0; i < kFlight; ++i) acc += v[i];
        }
        if (groups == 1) {
          __stcg(A.grad + q0 + c, acc);
          ss = __fmaf_rn(acc, acc, ss);
        } else {
          S.red[t] = acc;  // (one round: chunk < kTrainThreads)
        }
      }
      if (groups > 1) {
        __syncthreads();
        if (t < n) {
          float acc = S.red[t];
          for (int r = 1; r < groups; ++r) acc += S.red[r * chunk + t];
          __stcg(A.grad + q0 + t, acc);
          ss = __fmul_rn(acc, acc);
        }
      }
      if (A.params) {  // the slice's squares
        ss = warp_sum(ss);
        if (lane == 0) S.wsum[warp] = ss;
        __syncthreads();
        if (t == 0) {
          float v = S.wsum[0];
          for (int w = 1; w < kTrainThreads / 32; ++w) v += S.wsum[w];
          __stcg(A.ssq + blockIdx.x, v);
        }
      }
    }
    if (!A.params) return;  // the gradient alone
    arrivals += G;
    if (!grid_barrier(A, &S.late, arrivals)) return;
    // params -= lr c grad, c = min(1, clip / |grad|) when clip > 0, in every
    // block's own copy
    if (warp == 0) {
      float v = 0.0f;
      for (u32 b = lane; b < G; b += 32) v += __ldcg(A.ssq + b);
      v = warp_sum(v);
      if (lane == 0) {
        const float norm = __fsqrt_rn(v);
        const float c = (A.clip > 0.0f && norm > A.clip) ? __fdiv_rn(A.clip, norm) : 1.0f;
        S.step = __fmul_rn(A.lr, c);
      }
    }
    constexpr int kQuads = kGradStride / 4, kPer = (kQuads + kTrainThreads - 1) / kTrainThreads;
    float4 g[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int q = t + i * kTrainThreads;
      if (q < kQuads) g[i] = __ldcg(reinterpret_cast<const float4*>(A.grad) + q);
    }
    __syncthreads();
    const float by = S.step;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int q = 4 * (t + i * kTrainThreads);
      if (q >= kGradStride) continue;
      float* w = S.W + padded(q);  // the four of a quad lie together (rows are multiples of 4)
      w[0] = __fsub_rn(w[0], __fmul_rn(by, g[i].x));
      w[1] = __fsub_rn(w[1], __fmul_rn(by, g[i].y));
      w[2] = __fsub_rn(w[2], __fmul_rn(by, g[i].z));
      if (q + 3 < kMlpParams) w[3] = __fsub_rn(w[3], __fmul_rn(by, g[i].w));
    }
    start = next_start;
    __syncthreads();
  }
  if (A.params && blockIdx.x == 0)
    for (int q = t; q < kMlpParams; q += kTrainThreads) A.params[q] = S.W[padded(q)];
}

// Scratch layout in ctx->mlp_scratch (floats): partial [blocks * kGradStride] |
// grad [kGradStride] | ssq [blocks rounded up to 4] | barrier, late [2], spare (u32) | dense
// [n * 11] | flags [n+1] (u32) | pos [n+1] (u32)
struct TrainScratch {
  float *partial, *grad, *ssq, *dense;
  u32 *barrier, *late, *flags, *pos;
};

tera_status prepare(tera_ctx* ctx, u64 n, TrainScratch* t) {
  const u64 blocks = (u64)ctx->num_sms * kTrainPerSm;
  const u64 head = blocks * kGradStride + kGradStride + ((blocks + 3) & ~3ull) + 4;
  const u64 need = head + n * kDense + 2 * (n + 1) + 64;
  if (!ctx->mlp_scratch || ctx->mlp_scratch_cap < need) {
    cudaDeviceSynchronize();
    if (ctx->mlp_scratch) cudaFree(ctx->mlp_scratch);
    ctx->mlp_scratch = nullptr;
    if (cudaMalloc(reinterpret_cast<void**>(&ctx->mlp_scratch), sizeof(float) * need) != cudaSuccess) {
      cudaGetLastError();
      ctx->mlp_scratch_cap = 0;
      return TERA_ENOMEM;
    }
    ctx->mlp_scratch_cap = need;
  }
  float* b = ctx->mlp_scratch;
  t->partial = b;
  t->grad = b + blocks * kGradStride;
  t->ssq = t->grad + kGradStride;
  t->barrier = reinterpret_cast<u32*>(t->ssq + ((blocks + 3) & ~3ull));
  t->late = t->barrier + 1;
  t->dense = reinterpret_cast<float*>(t->barrier + 4);
  t->flags = reinterpret_cast<u32*>(t->dense + n * kDense);
  t->pos = t->flags + (n + 1);
  return TERA_OK;
}

tera_status compact(tera_ctx* ctx, const float* samples, u64 n, const TrainScratch& t, u64* nv,
                    cudaStream_t s) {
  const unsigned g = (unsigned)((n + 255) / 256 < 65535 ? (n + 255) / 256 + 1 : 65535);
  prof_begin(ctx, s);
  sample_flags_kernel<<<g, 256, 0, s>>>(samples, n, t.flags, t.late);
  tera_status st = check_launch(ctx, "sample_flags_kernel", s);
  if (st != TERA_OK) return st;
  if ((st = scan_u32(ctx, t.flags, nullptr, t.pos, n, s, t.late)) != TERA_OK) return st;
  prof_begin(ctx, s);
  sample_compact_kernel<<<g, 256, 0, s>>>(samples, n, t.flags, t.pos, t.dense, t.late);
  if ((st = check_launch(ctx, "sample_compact_kernel", s)) != TERA_OK) return st;
  u32 h[2] = {0, 0};
  if (cudaMemcpyAsync(h, t.late, sizeof(h), cudaMemcpyDeviceToHost, s) != cudaSuccess)
    return TERA_ECUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return TERA_ECUDA;
  if (h[0]) return TERA_ETIMEOUT;
  *nv = h[1];
  return TERA_OK;
}

// `steps` SGD steps on `batch` samples each (params), or one gradient
// (params null) into grad.  At most kTrainPerSm blocks per SM, which its registers
// and shared memory allow, so that the cooperative launch's blocks are resident
// together.
tera_status train_steps(tera_ctx* ctx, const TrainScratch& t, u64 nv, u64 batch, int steps,
                        const float* params_in, float* params, float* grad, float lr, float clip,
                        cudaStream_t s) {
  static PerDevice configured;
  if (configured.needed(ctx->device)) {
    if (cudaFuncSetAttribute(mlp_steps_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(TrainSmem<1>)) != cudaSuccess ||
        cudaFuncSetAttribute(mlp_steps_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(TrainSmem<2>)) != cudaSuccess)
      return TERA_ECUDA;
    configured.done(ctx->device);
  }
  TrainArgs A;
  A.dense = t.dense;
  A.nv = nv;
  A.batch = batch;
  A.steps = steps;
  A.lr = lr;
  A.clip = clip;
  A.params = params;
  A.params_in = params_in;
  A.partial = t.partial;
  A.grad = grad;
  A.ssq = t.ssq;
  A.barrier = t.barrier;
  A.st = ctx->d_status;
  // 64-sample tiles unless 32-sample ones find an SM each
  const bool small = batch <= 32 * (u64)ctx->num_sms;
  const u64 tiles = small ? (batch + 31) / 32 : (batch + 63) / 64;
  const u64 most = (u64)ctx->num_sms * kTrainPerSm;
  const unsigned blocks = (unsigned)(tiles < most ? tiles : most);
  if (cudaMemsetAsync(t.barrier, 0, sizeof(u32), s) != cudaSuccess) return TERA_ECUDA;
  prof_begin(ctx, s);
  void* args[] = {&A};
  cudaLaunchCooperativeKernel(small ? reinterpret_cast<const void*>(mlp_steps_kernel<1>)
                                    : reinterpret_cast<const void*>(mlp_steps_kernel<2>),
                              dim3(blocks), dim3(kTrainThreads), args,
                              small ? sizeof(TrainSmem<1>) : sizeof(TrainSmem<2>), s);
  return check_launch(ctx, "mlp_steps_kernel", s);
}

}  // namespace

extern "C" tera_status tera_mlp_grad(tera_ctx* ctx, const float* samples, uint64_t n,
                                     const float* params, float* grad, uint64_t* n_valid,
                                     void* stream) {
  TERA_CALL_RANGE("tera_mlp_grad");
  if (!ctx || !samples || !params || !grad || n == 0 || n > 0xFFFFFFF0ull) return TERA_EINVAL;
  cudaSetDevice(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  TrainScratch t;
  tera_status st = prepare(ctx, n, &t);
  if (st != TERA_OK) return st;
  u64 nv = 0;
  if ((st = compact(ctx, samples, n, t, &nv, s)) != TERA_OK) return st;
  if (n_valid) *n_valid = nv;
  if (nv == 0) return TERA_EINVAL;
  return train_steps(ctx, t, nv, nv, 1, params, nullptr, grad, 0.0f, 0.0f, s);
}

extern "C" tera_status tera_mlp_train(tera_ctx* ctx, const float* samples, uint64_t n,
                                      float* params, int steps, int batch, float lr, float clip,
                                      uint64_t* n_valid, void* stream) {
  TERA_CALL_RANGE("tera_mlp_train");
  if (!ctx || !samples || !params || n == 0 || n > 0xFFFFFFF0ull || steps < 0 || batch < 1 ||
      batch > (1 << 24))
    return TERA_EINVAL;
  cudaSetDevice(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  TrainScratch t;
  tera_status st = prepare(ctx, n, &t);
  if (st != TERA_OK) return st;
  u64 nv = 0;
  if ((st = compact(ctx, samples, n, t, &nv, s)) != TERA_OK) return st;
  if (n_valid) *n_valid = nv;
  if (nv == 0) return TERA_EINVAL;
  if (steps == 0) return TERA_OK;
  return train_steps(ctx, t, nv, (u64)batch, steps, params, params, t.grad, lr, clip, s);
}

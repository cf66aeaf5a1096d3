// mlp_kernels.cu -- the learned eps surrogate: 4 -> 32 (ReLU) -> 32 (ReLU) -> 1.
// Inputs x = (|d/r| components in decreasing order, r), d = cell centre minus
// sphere centre: the offset in the orientation fixed by the cube's symmetries
// (eps is invariant under sign flips and permutations of d).  The network
// predicts the correction to the linear approximation of Sec. 2.3.2
// (Eqs. 25-27): eps = clamp(eps_lin(|d|, r) + MLP(x), 0, 1).  It replaces the
// sub-division sampling for partial cells within reach of one particle and
// away from walls; 8^3 sampling stays the fallback and gives the labels the
// network is trained on (target: label - eps_lin).
//
// Parameters (FP32, packed): W1 [0,128) 32x4 row-major, b1 [128,160),
// W2 [160,1184) 32x32, b2 [1184,1216), W3 [1216,1248), b3 [1248].
//
// Training samples: SplitMix64 counter stream (value k of stream s is the
// SplitMix64 output for state s + (k+1)*0x9E3779B97F4A7C15; a uniform double
// is its top 53 bits times 2^-53).  Sample i uses values 5i..5i+4:
//   r = 2 + 10 u0; v = (2u1-1, 2u2-1, 2u3-1); rho = (r - sqrt3/2) + sqrt3 u4;
//   d = v * (rho / |v|); label = (8^3 samples of the cell inside) / 512.
// Every step is an IEEE-rounded FP64 operation (compiled with -fmad=false).
//
// Training: one block per 128-sample tile computes forward and backward in
// FP32 and the tile's gradient as sums over its samples (no atomics); the
// tiles are reduced in a fixed order; Adam (Kingma and Ba, 2015) updates the
// FP32 master weights.
//
// Inference: tiles of 128 inputs per CTA; layer 1 (K = 4) in FP32, layer 2
// on the 5th-generation tensor cores (tcgen05.mma, BF16 operands from shared
// memory, FP32 accumulator in tensor memory), layer 3 (N = 1) in FP32 after
// tcgen05.ld; in the mapping the same kernel turns the outputs into B.
#include <cuda_bf16.h>

#include "geom.cuh"
#include "psm_internal.cuh"

namespace psm {
namespace {

constexpr int OFF_B1 = 128, OFF_W2 = 160, OFF_B2 = 1184, OFF_W3 = 1216, OFF_B3 = 1248;
constexpr int NPARAM = 1249;

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long seed,
                                                         unsigned long long k) {
  unsigned long long z = seed + (k + 1ULL) * 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

__device__ __forceinline__ double uniform01(unsigned long long seed, unsigned long long k) {
  return (double)(splitmix64(seed, k) >> 11) * 0x1.0p-53;
}

// f(r) = V_a(r) - r + 1/2 of Eqs. 26-27 (training targets only; the mapping
// takes f(r) computed on the host for each particle)
__device__ double linear_fr(double r) {
  const double r2 = r * r;
  const double s = sqrt(r2 - 0.5);
  const double Va = (1.0 / 12.0 - r2) * atan((0.5 * s) / (0.5 - r2)) + s / 3.0 +
                    (r2 - 1.0 / 12.0) * atan(0.5 / s) - 4.0 / 3.0 * r2 * r * atan(0.25 / (r * s));
  return Va - r + 0.5;
}

// inputs of the network for offset d and radius r
__device__ __forceinline__ float4 network_input(double dx, double dy, double dz, double r) {
  double a = fabs(dx / r), b = fabs(dy / r), c = fabs(dz / r), t;
  if (b > a) { t = a; a = b; b = t; }
  if (c > a) { t = a; a = c; c = t; }
  if (c > b) { t = b; b = c; c = t; }
  return make_float4((float)a, (float)b, (float)c, (float)r);
}

// resid (optional): label - eps_lin, the network's training target
__global__ void samples_kernel(unsigned long long seed, long long first, long long count,
                               float* __restrict__ X, float* __restrict__ eps,
                               float* __restrict__ resid) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < count;
       t += (long long)gridDim.x * blockDim.x) {
    const unsigned long long i = (unsigned long long)(first + t);
    double u[5];
    for (int j = 0; j < 5; ++j) u[j] = uniform01(seed, 5ULL * i + j);
    const double r = 2.0 + 10.0 * u[0];
    double v0 = 2.0 * u[1] - 1.0, v1 = 2.0 * u[2] - 1.0, v2 = 2.0 * u[3] - 1.0;
    double nv = sqrt(v0 * v0 + v1 * v1 + v2 * v2);
    if (nv == 0.0) {
      v0 = 1.0; v1 = 0.0; v2 = 0.0; nv = 1.0;
    }
    const double rho = (r - kHalfSqrt3) + 1.7320508075688772935 * u[4];
    const double tt = rho / nv;
    const double d0 = v0 * tt, d1 = v1 * tt, d2 = v2 * tt;
    const int cnt = supersample_count_n<8>(d0, d1, d2, r);
    reinterpret_cast<float4*>(X)[t] = network_input(d0, d1, d2, r);
    const double label = (double)cnt * (1.0 / 512.0);
    eps[t] = (float)label;
    if (resid) {
      const double dist = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
      double lin = -(dist - r) + linear_fr(r);
      lin = lin < 0.0 ? 0.0 : (lin > 1.0 ? 1.0 : lin);
      resid[t] = (float)(label - lin);
    }
  }
}

// ---- training: forward + backward of one tile of samples.  A tile is 128
// samples, 8 to each of the block's 16 warps: a thread computes 4 samples x 2
// units of a layer, reading inputs and weights four at a time along the sum
// (rows of 36 floats: eight rows' 16-byte pieces fall in different banks), and
// only the warp itself meets between layers.  Every sum runs in a fixed order
// (a unit's over its inputs, a gradient's over the tile's samples), so the
// result does not depend on how the work is split.  One thread per sample, as
// before, left 4 warps an SM to two shared-memory reads per multiply-add.
constexpr int TILE = 128;
constexpr int ROW = 36;
constexpr int TRAIN_THREADS = 512;
static_assert(TRAIN_THREADS == 4 * TILE, "8 samples per warp");

// the network's parameters as the layers read them (W2 also transposed, for
// the backward product)
struct alignas(16) NetSmem {
  float w1[32][4];
  float b1[32];
  float w2[32][ROW];
  float w2t[32][ROW];
  float b2[32], w3[32];
  float b3, one;
};
// places (in floats) of packed parameter e
__device__ __forceinline__ int net_place(int e, int* second) {
  constexpr int B1 = 128, W2 = 160, W2T = W2 + 32 * ROW, B2 = W2T + 32 * ROW;
  *second = -1;
  if (e < OFF_W2) return e;  // w1, b1
  if (e < OFF_B2) {
    const int j = (e - OFF_W2) >> 5, k = (e - OFF_W2) & 31;
    *second = W2T + k * ROW + j;
    return W2 + j * ROW + k;
  }
  static_assert(OFF_B1 == B1 && OFF_W2 == W2 && OFF_W3 == OFF_B2 + 32 && OFF_B3 == OFF_W3 + 32,
                "b2, w3 and b3 follow one another");
  return B2 + (e - OFF_B2);
}
struct TrainSmem {
  NetSmem net;
  float4 x[TILE];
  float h1[TILE][ROW], h2[TILE][ROW];    // activations
  float dh1[TILE][ROW], dh2[TILE][ROW];  // gradients before the ReLU
  float4 dyl[TILE];                      // d loss / d y, squared residual
};

__device__ __forceinline__ void load_net(TrainSmem& S, const float* __restrict__ params) {
  float* n = reinterpret_cast<float*>(&S.net);
  for (int e = threadIdx.x; e < NPARAM; e += TRAIN_THREADS) {
    int b;
    const int a = net_place(e, &b);
    const float v = params[e];
    n[a] = v;
    if (b >= 0) n[b] = v;
  }
  if (threadIdx.x == 0) S.net.one = 1.0f;
}

// a lane's input of a tile: lanes 0-7 of warp w hold samples 8w .. 8w + 7
struct SampleIn {
  float x[4], t;
};
__device__ __forceinline__ void load_sample(const float* __restrict__ X,
                                            const float* __restrict__ t, long long first,
                                            int nrow, SampleIn& I) {
  const int s = 8 * (threadIdx.x >> 5) + (threadIdx.x & 31);
  const bool in = (threadIdx.x & 31) < 8 && s < nrow;
#pragma unroll
  for (int k = 0; k < 4; ++k) I.x[k] = in ? X[4 * (first + s) + k] : 0.f;
  I.t = in ? t[first + s] : 0.f;
}

__device__ __forceinline__ float4 row4(const float* row, int c) {
  return reinterpret_cast<const float4*>(row)[c];
}
__device__ __forceinline__ float chain4(float acc, const float4& w, const float4& v) {
  acc = fmaf(w.x, v.x, acc);
  acc = fmaf(w.y, v.y, acc);
  acc = fmaf(w.z, v.z, acc);
  return fmaf(w.w, v.w, acc);
}

// forward (and backward) of the warp's 8 samples; rows nrow and up count as zeros
template <bool BACK>
__device__ __forceinline__ void tile_rows(TrainSmem& S, int nrow, const SampleIn& I,
                                          float inv_m) {
  const int lane = threadIdx.x & 31, s0 = 8 * (threadIdx.x >> 5);
  const int sb = s0 + 4 * (lane >> 4), jg = lane & 15;  // samples sb .. sb + 3, units jg, jg + 16
  if (lane < 8) S.x[s0 + lane] = make_float4(I.x[0], I.x[1], I.x[2], I.x[3]);
  __syncwarp();
  float h1[4][2], h2[4][2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int j = jg + 16 * i;
    const float4 w = row4(S.net.w1[j], 0);
    const float b = S.net.b1[j];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float a = chain4(b, w, S.x[sb + r]);
      h1[r][i] = a > 0.f && sb + r < nrow ? a : 0.f;
      S.h1[sb + r][j] = h1[r][i];
    }
  }
  __syncwarp();
  float acc[4][2];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int i = 0; i < 2; ++i) acc[r][i] = S.net.b2[jg + 16 * i];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float4 wa = row4(S.net.w2[jg], c), wb = row4(S.net.w2[jg + 16], c);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 h = row4(S.h1[sb + r], c);
      acc[r][0] = chain4(acc[r][0], wa, h);
      acc[r][1] = chain4(acc[r][1], wb, h);
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      h2[r][i] = acc[r][i] > 0.f && sb + r < nrow ? acc[r][i] : 0.f;
      S.h2[sb + r][jg + 16 * i] = h2[r][i];
    }
  __syncwarp();
  if (lane < 8) {
    float y = S.net.b3;
#pragma unroll
    for (int c = 0; c < 8; ++c) y = chain4(y, row4(S.net.w3, c), row4(S.h2[s0 + lane], c));
    const float res = y - I.t;
    const float dy = 2.0f * res * inv_m;
    S.dyl[s0 + lane] = s0 + lane < nrow ? make_float4(dy, res * res, 0.f, 0.f)
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if constexpr (BACK) {
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float dy = S.dyl[sb + r].x;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        S.dh2[sb + r][jg + 16 * i] = h2[r][i] > 0.f ? dy * S.net.w3[jg + 16 * i] : 0.f;
        acc[r][i] = 0.f;
      }
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float4 wa = row4(S.net.w2t[jg], c), wb = row4(S.net.w2t[jg + 16], c);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float4 d = row4(S.dh2[sb + r], c);
        acc[r][0] = chain4(acc[r][0], wa, d);
        acc[r][1] = chain4(acc[r][1], wb, d);
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int i = 0; i < 2; ++i)
        S.dh1[sb + r][jg + 16 * i] = h1[r][i] > 0.f ? acc[r][i] : 0.f;
  }
}

// gradient of the tile (sums over its samples in order) and its squared
// residual: four warps take dW2, 4 x 2 entries per thread, two the rest (the
// biases' sums as products with one)
__device__ __forceinline__ void tile_grad(const TrainSmem& S, float* __restrict__ out) {
  const int warp = threadIdx.x >> 5;
  if (warp < 4) {
    const int jg = threadIdx.x & 7, kg = threadIdx.x >> 3;  // rows 4 jg .., columns 2 kg ..
    float g[4][2] = {};
#pragma unroll 8
    for (int q = 0; q < TILE; ++q) {
      const float4 d = row4(S.dh2[q], jg);
      const float2 h = reinterpret_cast<const float2*>(S.h1[q])[kg];
      g[0][0] = fmaf(d.x, h.x, g[0][0]);
      g[0][1] = fmaf(d.x, h.y, g[0][1]);
      g[1][0] = fmaf(d.y, h.x, g[1][0]);
      g[1][1] = fmaf(d.y, h.y, g[1][1]);
      g[2][0] = fmaf(d.z, h.x, g[2][0]);
      g[2][1] = fmaf(d.z, h.y, g[2][1]);
      g[3][0] = fmaf(d.w, h.x, g[3][0]);
      g[3][1] = fmaf(d.w, h.y, g[3][1]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      out[OFF_W2 + (4 * jg + c) * 32 + 2 * kg] = g[c][0];
      out[OFF_W2 + (4 * jg + c) * 32 + 2 * kg + 1] = g[c][1];
    }
  } else if (warp < 6) {
    const int it = threadIdx.x - 128, jg = it & 7;
    const float* v;         // four values per sample, rows of vs floats
    const float* a = &S.net.one;  // their factor, as floats apart
    int vs = ROW, as = 0, o, os = 1, n = 4;
    if (it < 32) {  // dW1
      v = S.dh1[0] + 4 * jg;
      a = reinterpret_cast<const float*>(S.x) + (it >> 3);
      as = 4;
      o = 16 * jg + (it >> 3);
      os = 4;
    } else if (it < 40) {
      v = S.dh1[0] + 4 * jg;
      o = OFF_B1 + 4 * jg;
    } else if (it < 48) {
      v = S.dh2[0] + 4 * jg;
      o = OFF_B2 + 4 * jg;
    } else if (it < 56) {
      v = S.h2[0] + 4 * jg;
      a = &S.dyl[0].x;
      as = 4;
      o = OFF_W3 + 4 * jg;
    } else {  // db3 and the loss
      v = &S.dyl[0].x;
      vs = 4;
      o = OFF_B3;
      n = it == 56 ? 2 : 0;
    }
    float g[4] = {};
#pragma unroll 8
    for (int q = 0; q < TILE; ++q) {
      const float4 d = row4(v + q * vs, 0);
      const float f = a[q * as];
      g[0] = fmaf(d.x, f, g[0]);
      g[1] = fmaf(d.y, f, g[1]);
      g[2] = fmaf(d.z, f, g[2]);
      g[3] = fmaf(d.w, f, g[3]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c < n) out[o + c * os] = g[c];
  }
}

__device__ __forceinline__ int tile_count(long long m, long long first) {
  return (int)(m - first < TILE ? m - first : TILE);
}

__global__ void __launch_bounds__(TRAIN_THREADS) train_tile_kernel(
    const float* __restrict__ params, long long m, const float* __restrict__ X,
    const float* __restrict__ t, float* __restrict__ partials) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(smem_raw);
  const long long first = (long long)blockIdx.x * TILE;
  const int nrow = tile_count(m, first);
  SampleIn I;
  load_sample(X, t, first, nrow, I);
  load_net(S, params);
  __syncthreads();
  tile_rows<true>(S, nrow, I, 1.0f / (float)m);
  __syncthreads();
  tile_grad(S, partials + (long long)blockIdx.x * (NPARAM + 1));
}

__global__ void grad_reduce_kernel(const float* __restrict__ partials, int nblocks,
                                   float* __restrict__ grad, float* __restrict__ loss,
                                   float inv_m) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e > NPARAM) return;
  float acc = 0.f;
  for (int b = 0; b < nblocks; ++b) acc += partials[(long long)b * (NPARAM + 1) + e];
  if (e < NPARAM) grad[e] = acc;
  else if (loss) *loss = acc * inv_m;
}

// one parameter's Adam step
__device__ __forceinline__ void adam(float gi, const AdamStep& a, float& p, float& m, float& v) {
  const float mi = 0.9f * m + 0.1f * gi;
  const float vi = 0.999f * v + 0.001f * gi * gi;
  m = mi;
  v = vi;
  const float mh = mi / a.bc1, vh = vi / a.bc2;
  p -= a.lr * mh / (sqrtf(vh) + 1e-8f);
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g,
                            float* __restrict__ m, float* __restrict__ v, AdamStep a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < NPARAM) adam(g[i], a, p[i], m[i], v[i]);
}

// ---- minibatch steps one after another in one launch: a cluster of 8 CTAs
// keeps the network in shared memory.  Per step the CTAs take the
// minibatch's tiles in turn and leave their gradients in `partials`; each CTA
// sums an eighth of the entries over the tiles in order, applies Adam (its
// moments stay in registers) and writes the new values into every CTA's copy.
// Two cluster barriers per step stand for the three launches they replace.
// Bound by latency: of the 8.8 us of a minibatch of 1024 samples most is the
// chain of layers, gradient sums, barriers and the sum over the tiles (a tile's
// multiply-adds alone would take 2 us of its SM).  Before, with one thread per
// sample and three launches, 35 us.
constexpr int CLUSTER = 8;
constexpr int SLICE = (NPARAM + CLUSTER - 1) / CLUSTER;

__device__ __forceinline__ void cluster_sync_all() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void store_cluster(const float* local, unsigned rank, float v) {
  unsigned a = (unsigned)__cvta_generic_to_shared(local), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(r), "f"(v) : "memory");
}

// minibatch i of the launch: samples b0 + i batch (mod nsamples' minibatches,
// per_epoch of them) ..; sched[i]: its Adam coefficients
__global__ void __cluster_dims__(CLUSTER, 1, 1) __launch_bounds__(TRAIN_THREADS, 1)
    train_cluster_kernel(float* __restrict__ params, float* __restrict__ mstate,
                         float* __restrict__ vstate, const float* __restrict__ X,
                         const float* __restrict__ t, long long nsamples, int batch,
                         long long per_epoch, long long mb0, int steps,
                         const AdamStep* __restrict__ sched, float* __restrict__ partials) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(smem_raw);
  const int rank = (int)blockIdx.x;  // the grid is one cluster
  const int e = rank * SLICE + (int)threadIdx.x;
  const bool own = threadIdx.x < SLICE && e < NPARAM;
  int pb = -1;
  const int pa = own ? net_place(e, &pb) : 0;
  float p = 0.f, mo = 0.f, ve = 0.f;
  if (own) {
    p = params[e];
    mo = mstate[e];
    ve = vstate[e];
  }
  load_net(S, params);
  cluster_sync_all();  // every CTA runs before its shared memory is written
  long long mb = mb0;
  SampleIn I;
  auto load_first = [&](long long b) {  // the CTA's first tile of minibatch b
    const long long s = b * batch, n = min((long long)batch, nsamples - s);
    const long long first = (long long)rank * TILE;
    load_sample(X, t, s + first, first < n ? tile_count(n, first) : 0, I);
  };
  load_first(mb);
  for (int i = 0; i < steps; ++i) {
    const long long s = mb * batch;
    const int n = (int)min((long long)batch, nsamples - s);
    const int ntile = (n + TILE - 1) / TILE;
    const float inv_m = 1.0f / (float)(long long)n;
    const AdamStep a = sched[i];
    for (int k = rank; k < ntile; k += CLUSTER) {
      const int nrow = tile_count(n, (long long)k * TILE);
      if (k != rank) {
        load_sample(X, t, s + (long long)k * TILE, nrow, I);
        __syncthreads();  // the previous tile's gradient is done
      }
      tile_rows<true>(S, nrow, I, inv_m);
      __syncthreads();
      tile_grad(S, partials + (long long)k * (NPARAM + 1));
    }
    mb = mb + 1 == per_epoch ? 0 : mb + 1;
    if (i + 1 < steps) load_first(mb);  // on its way while the CTAs meet
    cluster_sync_all();
    if (own) {
      float g = 0.f;
#pragma unroll 8
      for (int k = 0; k < ntile; ++k) g += __ldcg(partials + (long long)k * (NPARAM + 1) + e);
      adam(g, a, p, mo, ve);
      const float* net = reinterpret_cast<const float*>(&S.net);
#pragma unroll
      for (unsigned r = 0; r < CLUSTER; ++r) {
        store_cluster(net + pa, r, p);
        if (pb >= 0) store_cluster(net + pb, r, p);
      }
    }
    cluster_sync_all();
  }
  if (own) {
    params[e] = p;
    mstate[e] = mo;
    vstate[e] = ve;
  }
}

// squared residuals of each minibatch's tiles (tiles per minibatch, the
// last one's may be fewer)
__global__ void __launch_bounds__(TRAIN_THREADS) train_loss_kernel(
    const float* __restrict__ params, const float* __restrict__ X, const float* __restrict__ t,
    long long nsamples, int batch, int tiles, long long ntiles, float* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(smem_raw);
  load_net(S, params);
  for (long long w = blockIdx.x; w < ntiles; w += gridDim.x) {
    const long long mb = w / tiles, first = (w - mb * tiles) * TILE, s = mb * batch;
    const long long n = min((long long)batch, nsamples - s);
    const int nrow = first < n ? tile_count(n, first) : 0;
    SampleIn I;
    load_sample(X, t, s + first, nrow, I);
    __syncthreads();  // the network; the previous tile's sum is done
    tile_rows<false>(S, nrow, I, 0.f);
    __syncthreads();
    if (threadIdx.x == 0) {
      float acc = 0.f;
#pragma unroll 8
      for (int q = 0; q < TILE; ++q) acc += S.dyl[q].y;
      out[w] = acc;
    }
  }
}

// ---- inference on the 5th-generation tensor cores.  One CTA of 128
// threads takes two tiles of 128 inputs at a time: each thread computes its
// two rows' layer 1 in FP32 (each weight read once for both) and writes the
// ReLU activations as BF16 into shared memory in the K-major core-matrix
// layout (8 rows x 16 bytes per core matrix); one thread issues each tile's
// layer-2 product h1 (128 x 32) x W2^T (32 x 32) as two tcgen05.mma (K = 16
// each, BF16 operands) into its own FP32 accumulator in tensor memory (32
// columns each) and one commit for the four; after the commit arrives on the
// mbarrier each warp reads its 32 rows of each tile back with tcgen05.ld and
// finishes layer 3 (bias, ReLU, dot with W3) in FP32.  Waits are bounded: a wait that gives up sets
// ST_TIMEOUT, waits once more for the tensor core and frees its tensor memory.
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

constexpr int INF_M = 128;         // rows per tile: the MMA's M
constexpr int INF_THREADS = 128;   // thread t owns row t; warp w reads TMEM lanes 32w..32w+31
constexpr int INF_PER_SM = 6;      // resident CTAs per SM: the grid is one wave of them
constexpr unsigned INF_TMEM_COLS = 64;  // two FP32 accumulators of N = 32 columns
constexpr unsigned long long kInferWaitNs = 1000000000ull;
// instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16
// A and B (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0), N / 8 at
// bits 17-22, M / 16 at bits 24-28
constexpr uint32_t kInferIdesc =
    (1u << 4) | (1u << 7) | (1u << 10) | ((32u >> 3) << 17) | ((unsigned)(INF_M >> 4) << 24);

struct InferSmem {
  alignas(128) unsigned char a[2][INF_M * 32 * 2];  // layer-1 activations of two tiles, BF16
  alignas(128) unsigned char b[32 * 32 * 2];     // W2 (N = 32 rows of K = 32), BF16
  float4 w1[32];
  float b1[32], b2[32], w3[32];
  float b3;
  unsigned tmem;
  unsigned long long bar;
};

// byte offset of the 16-byte chunk kc (elements 8kc..8kc+7) of row `row` in
// the K-major layout without swizzle: core matrices of 8 rows x 16 bytes, the
// K direction's four core matrices 128 bytes apart (leading byte offset),
// successive groups of 8 rows 512 bytes apart (stride byte offset)
__device__ __forceinline__ int kmajor_off(int row, int kc) {
  return (row >> 3) * 512 + kc * 128 + (row & 7) * 16;
}
__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
// shared-memory matrix descriptor of tcgen05: start address >> 4 (bits 0-13),
// leading byte offset >> 4 (bits 16-29), stride byte offset >> 4 (bits
// 32-45), the fixed value 1 at bits 46-48, base offset 0, no swizzle
__device__ __forceinline__ uint64_t kmajor_desc(const void* p) {
  return (uint64_t)((smem_addr(p) & 0x3FFFFu) >> 4) | ((uint64_t)(128 >> 4) << 16) |
         ((uint64_t)(512 >> 4) << 32) | (1ull << 46);
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ bool inf_mbar_test(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __noinline__ bool inf_mbar_wait(unsigned long long* bar, unsigned parity,
                                           unsigned long long limit_ns = kInferWaitNs) {
  if (inf_mbar_test(bar, parity)) return true;
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (inf_mbar_test(bar, parity)) return true;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > limit_ns) return false;
  }
}

// diagnostic: the inference kernel's bounded wait on an mbarrier that no
// commit arrives on gives up after limit_ns and raises ST_TIMEOUT
__global__ void infer_wait_selftest_kernel(unsigned* status, unsigned long long limit_ns) {
  __shared__ __align__(8) unsigned long long bar;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0 && !inf_mbar_wait(&bar, 0u, limit_ns)) atomicOr(status, ST_TIMEOUT);
}
__device__ __forceinline__ void tc_mma_bf16(unsigned d_tmem, uint64_t adesc, uint64_t bdesc,
                                            int accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(kInferIdesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_commit(unsigned long long* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_addr(bar))
      : "memory");
}
// 32 consecutive accumulator columns of this warp's 32 TMEM lanes, one lane per thread
__device__ __forceinline__ void tc_ld32(unsigned taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// B(eps) of Eq. 16 in the storage precision of the slot records
__device__ __forceinline__ void apply_weight(const InferSink& o, long long rec, float epsf) {
  if (o.fp32) {
    float B = epsf;
    if (o.nt && epsf != 0.f && epsf != 1.f) {
      const float tm = (float)(o.tau - 0.5);
      B = epsf * tm / ((1.f - epsf) + tm);
    }
    static_cast<float*>(o.V)[4 * rec + 3] = B;
  } else {
    const double eps = (double)epsf;
    double B = eps;
    if (o.nt && eps != 0.0 && eps != 1.0) B = eps * (o.tau - 0.5) / ((1.0 - eps) + (o.tau - 0.5));
    if (o.dfrec) static_cast<df*>(o.V)[4 * rec + 3] = df(B);
    else static_cast<double*>(o.V)[4 * rec + 3] = B;
  }
}

// raw network outputs (o.eps != NULL) or, in the mapping, eps = clamp(linear
// approximation + output, 0, 1) and its weight B into the item's slot record
// when the cell is within reach of this particle only (cells shared by two
// particles keep B = -1 and are sampled by the finish pass).  count: number
// of inputs, read from *count_dev when count < 0, at most cap.
__global__ void __launch_bounds__(INF_THREADS, INF_PER_SM) infer_tc_kernel(
    const float* __restrict__ P, long long count, const int* __restrict__ count_dev,
    long long cap, const float4* __restrict__ X, InferSink o, unsigned* status) {
  __shared__ InferSmem S;
  const int tid = threadIdx.x, warp = tid >> 5;
  long long n = count >= 0 ? count : (long long)*count_dev;
  if (n > cap) n = cap;
  // W2 as the B operand (row j = output neuron, K = input neuron), the
  // other parameters in FP32
  for (int i = tid; i < 32 * 4; i += INF_THREADS) {
    const int j = i >> 2, kc = i & 3;
    const float* w = P + OFF_W2 + j * 32 + kc * 8;
    *reinterpret_cast<uint4*>(S.b + kmajor_off(j, kc)) =
        make_uint4(pack_bf16(w[0], w[1]), pack_bf16(w[2], w[3]), pack_bf16(w[4], w[5]),
                   pack_bf16(w[6], w[7]));
  }
  if (tid < 32) {
    S.w1[tid] = make_float4(P[4 * tid], P[4 * tid + 1], P[4 * tid + 2], P[4 * tid + 3]);
    S.b1[tid] = P[OFF_B1 + tid];
    S.b2[tid] = P[OFF_B2 + tid];
    S.w3[tid] = P[OFF_W3 + tid];
  }
  if (tid == 0) {
    S.b3 = P[OFF_B3];
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&S.bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&S.tmem)),
                 "r"(INF_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_async_smem();  // W2 was written by the generic proxy, the MMA reads it
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = S.tmem;
  // A operands of the two tiles, K = 0..15 and 16..31 (chunks 0-1 and 2-3)
  const uint64_t ad00 = kmajor_desc(S.a[0]), ad01 = kmajor_desc(S.a[0] + 256);
  const uint64_t ad10 = kmajor_desc(S.a[1]), ad11 = kmajor_desc(S.a[1] + 256);
  const uint64_t bd0 = kmajor_desc(S.b), bd1 = kmajor_desc(S.b + 256);
  unsigned phase = 0;
  bool in_flight = false;
  // software pipeline: a tile's inputs (and, in the mapping, its slot item
  // and linear approximation) are loaded while the previous tile computes
  auto load_row = [&](long long r, float4& xr, int& it, float& ln) {
    xr = make_float4(0.f, 0.f, 0.f, 0.f);
    it = -1;
    ln = 0.f;
    if (r < n) {
      xr = X[r];
      if (!o.eps) {
        it = o.work[r];
        ln = o.lin[r];
      }
    }
  };
  // each iteration takes two tiles (rows r and r + 128 of a pair): layer 1
  // reads each weight once for both rows, one commit covers both products
  // and the CTA meets at two barriers per 256 rows
  const long long npairs = (n + 2 * INF_M - 1) / (2 * INF_M);
  float4 x0, x1;
  int item0, item1;
  float lin0, lin1;
  load_row((long long)blockIdx.x * (2 * INF_M) + tid, x0, item0, lin0);
  load_row((long long)blockIdx.x * (2 * INF_M) + INF_M + tid, x1, item1, lin1);
  // layer 3 and B(eps) of one row from its accumulator columns
  auto finish_row = [&](const float* acc, long long row, int item, float lin) {
    float y = 0.f;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const float v = acc[j] + S.b2[j];
      y = fmaf(S.w3[j], v > 0.f ? v : 0.f, y);
    }
    y += S.b3;
    if (row < n) {
      if (o.eps) {
        o.eps[row] = y;
      } else if (item >= 0) {  // item -1: an empty item (the fill pass lists
                               // only cells in reach of one particle)
        float eps = lin + y;
        eps = eps < 0.f ? 0.f : (eps > 1.f ? 1.f : eps);
        apply_weight(o, (item & 1) * o.cap + (item >> 1), eps);
      }
    }
  };
  for (long long pr = blockIdx.x; pr < npairs; pr += gridDim.x) {
    const long long row0 = pr * (2 * INF_M) + tid, row1 = row0 + INF_M;
    float4 xn0, xn1;
    int itemn0, itemn1;
    float linn0, linn1;
    const long long next = (pr + gridDim.x) * (2 * INF_M) + tid;
    load_row(next, xn0, itemn0, linn0);
    load_row(next + INF_M, xn1, itemn1, linn1);
    // layer 1 (FP32), ReLU, BF16 activations into the two A operands
#pragma unroll
    for (int kc = 0; kc < 4; ++kc) {
      uint32_t w0[4], w1[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        float v0[2], v1[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int j = 8 * kc + 2 * h + e;
          const float4 wj = S.w1[j];
          const float bj = S.b1[j];
          float a = fmaf(wj.x, x0.x, bj);
          a = fmaf(wj.y, x0.y, a);
          a = fmaf(wj.z, x0.z, a);
          a = fmaf(wj.w, x0.w, a);
          float b = fmaf(wj.x, x1.x, bj);
          b = fmaf(wj.y, x1.y, b);
          b = fmaf(wj.z, x1.z, b);
          b = fmaf(wj.w, x1.w, b);
          v0[e] = a > 0.f ? a : 0.f;
          v1[e] = b > 0.f ? b : 0.f;
        }
        w0[h] = pack_bf16(v0[0], v0[1]);
        w1[h] = pack_bf16(v1[0], v1[1]);
      }
      *reinterpret_cast<uint4*>(S.a[0] + kmajor_off(tid, kc)) =
          make_uint4(w0[0], w0[1], w0[2], w0[3]);
      *reinterpret_cast<uint4*>(S.a[1] + kmajor_off(tid, kc)) =
          make_uint4(w1[0], w1[1], w1[2], w1[3]);
    }
    fence_async_smem();
    __syncthreads();
    bool done = true;
    if (tid == 0) {
      tc_fence_after();
      tc_mma_bf16(tmem, ad00, bd0, 0);
      tc_mma_bf16(tmem, ad01, bd1, 1);
      tc_mma_bf16(tmem + 32u, ad10, bd0, 0);
      tc_mma_bf16(tmem + 32u, ad11, bd1, 1);
      tc_commit(&S.bar);
      done = inf_mbar_wait(&S.bar, phase);
    }
    in_flight = true;
    if (!__syncthreads_and(done)) {
      if (tid == 0) atomicOr(status, ST_TIMEOUT);
      break;
    }
    in_flight = false;
    phase ^= 1u;
    tc_fence_after();
    float acc[32];
    const unsigned lanes = (unsigned)(warp * 32) << 16;
    tc_ld32(tmem + lanes, acc);
    finish_row(acc, row0, item0, lin0);
    tc_ld32(tmem + lanes + 32u, acc);
    finish_row(acc, row1, item1, lin1);
    x0 = xn0;
    x1 = xn1;
    item0 = itemn0;
    item1 = itemn1;
    lin0 = linn0;
    lin1 = linn1;
    tc_fence_before();
    __syncthreads();  // the A tiles and the accumulators are free again
  }
  if (in_flight && tid == 0) inf_mbar_wait(&S.bar, phase);  // the MMA of a wait that gave up
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(INF_TMEM_COLS)
                 : "memory");
  }
}

}  // namespace

int launch_mlp_samples(unsigned long long seed, long long first, long long count, float* X,
                       float* eps, float* resid, cudaStream_t s) {
  if (count <= 0) return 0;
  long long blocks = (count + 255) / 256;
  if (blocks > 152 * 64) blocks = 152 * 64;
  samples_kernel<<<(unsigned)blocks, 256, 0, s>>>(seed, first, count, X, eps, resid);
  return 1;
}

int mlp_grad_blocks(long long m) { return (int)((m + TILE - 1) / TILE); }

int launch_mlp_loss_grad(const float* params, long long m, const float* X, const float* t,
                         float* grad_partials, int nblocks, float* grad, float* loss,
                         cudaStream_t s) {
  train_tile_kernel<<<nblocks, TRAIN_THREADS, sizeof(TrainSmem), s>>>(params, m, X, t,
                                                                      grad_partials);
  grad_reduce_kernel<<<(NPARAM + 1 + 255) / 256, 256, 0, s>>>(grad_partials, nblocks, grad,
                                                             loss, 1.0f / (float)m);
  return 2;
}

// Minibatches of up to kClusterTiles tiles train in the cluster kernel, all
// `steps` in one launch; larger ones, whose tiles fill more SMs than a cluster
// has, in three launches each.  Per minibatch of 8, 16, 32 and 64 tiles the
// cluster kernel takes 8.8, 14.8, 26.8 and 51 us, the launches 18.4 each.
constexpr int kClusterTiles = 16;
int launch_train_steps(float* params, float* mstate, float* vstate, const float* X, const float* t,
                       long long nsamples, int batch, long long per_epoch, long long mb0,
                       int steps, const AdamStep* sched_host, AdamStep* sched, float* partials,
                       float* grad, cudaStream_t s) {
  const int tiles = mlp_grad_blocks(batch < nsamples ? batch : nsamples);
  if (tiles <= kClusterTiles) {
    cudaMemcpyAsync(sched, sched_host, sizeof(AdamStep) * steps, cudaMemcpyHostToDevice, s);
    train_cluster_kernel<<<CLUSTER, TRAIN_THREADS, sizeof(TrainSmem), s>>>(
        params, mstate, vstate, X, t, nsamples, batch, per_epoch, mb0, steps, sched, partials);
    return 1;
  }
  for (int i = 0; i < steps; ++i) {
    const long long b0 = (mb0 + i) % per_epoch * batch;
    const long long m = nsamples - b0 < batch ? nsamples - b0 : batch;
    launch_mlp_loss_grad(params, m, X + 4 * b0, t + b0, partials, mlp_grad_blocks(m), grad,
                         nullptr, s);
    adam_kernel<<<(NPARAM + 255) / 256, 256, 0, s>>>(params, grad, mstate, vstate, sched_host[i]);
  }
  return 3 * steps;
}

long long train_loss_tiles(long long nsamples, int batch) {
  const long long b = batch < nsamples ? batch : nsamples;
  return (nsamples + b - 1) / b * mlp_grad_blocks(b);
}

int launch_train_loss(const float* params, const float* X, const float* t, long long nsamples,
                      int batch, float* out, cudaStream_t s) {
  const long long n = train_loss_tiles(nsamples, batch);
  const int tiles = mlp_grad_blocks(batch < nsamples ? batch : nsamples);
  const long long blocks = n < 152 * 2 ? n : 152 * 2;
  train_loss_kernel<<<(unsigned)blocks, TRAIN_THREADS, sizeof(TrainSmem), s>>>(
      params, X, t, nsamples, batch, tiles, n, out);
  return 1;
}

int mlp_train_configure() {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int smem = (int)sizeof(TrainSmem);
  int bad = cudaFuncSetAttribute(train_tile_kernel, a, smem) != cudaSuccess;
  bad |= cudaFuncSetAttribute(train_cluster_kernel, a, smem) != cudaSuccess;
  bad |= cudaFuncSetAttribute(train_loss_kernel, a, smem) != cudaSuccess;
  return bad;
}

int launch_wait_selftest_mlp(unsigned* status, unsigned long long limit_ns, cudaStream_t s) {
  infer_wait_selftest_kernel<<<1, 32, 0, s>>>(status, limit_ns);
  return 1;
}

// network outputs for m inputs (m_dev: count on the device, m < 0), at most
// cap; results to the sink
// resident inference CTAs on the device (all SMs), set by mlp_configure
static int g_infer_ctas = 0;

int mlp_configure() {
  // INF_PER_SM CTAs per SM (the launch bounds keep their registers within
  // the SM's file; 6 x 64 of the 512 tensor-memory columns) times the SMs;
  // shared memory for all of them (6 x 19 KB): the carveout's maximum.
  // (Eight CTAs of 64 registers spilled and measured 7% slower.)
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      sms <= 0 ||
      cudaFuncSetAttribute(infer_tc_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                           (int)cudaSharedmemCarveoutMaxShared) != cudaSuccess)
    return 1;
  g_infer_ctas = sms * INF_PER_SM;
  return 0;
}

int launch_mlp_infer(const float* params, long long m, const int* m_dev, long long cap,
                     const float* X, const InferSink& out, unsigned* status, cudaStream_t s) {
  const long long rows = m >= 0 ? (m < cap ? m : cap) : cap;
  if (rows <= 0) return 0;
  // one wave of CTAs, each looping over tiles (a second, partial wave would
  // leave SMs idle)
  long long blocks = (rows + 2 * INF_M - 1) / (2 * INF_M);  // pairs of tiles
  const long long wave = g_infer_ctas > 0 ? g_infer_ctas : 152 * INF_PER_SM;
  if (blocks > wave) blocks = wave;
  infer_tc_kernel<<<(unsigned)blocks, INF_THREADS, 0, s>>>(
      params, m, m_dev, cap, reinterpret_cast<const float4*>(X), out, status);
  return 1;
}

}  // namespace psm

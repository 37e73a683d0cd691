// Fitness kernels on CUDA cores: the FP32 path of small networks and the
// FP32 dispatch (GPU-MGFWA, Algorithm 1: "evaluate all the fitness of the
// sparks"; larger networks: k_fitness_x3.cu), the fixed-order reduction of
// per-tile partial sums shared with the tensor-core path, the sphere, and
// the FP64 re-computation of the reported best loss.
//
// The objective is the mean cross-entropy of an MLP whose flattened
// parameters are the spark (nn.Linear order), on the shared batch X:
//   h_1 = act(W_1 x_n + b_1), ..., z = W_L h_{L-1} + b_L,
//   f = (1/N) sum_n [max_c z_c + log sum_c exp(z_c - max_c z_c) - z_{y_n}].
#include "mgfwa_internal.cuh"

namespace mgfwa {

namespace {

constexpr int kMT = 128;      // samples per tile (one per thread of the tail)
constexpr int kHC = 64;       // hidden units per first-layer chunk
constexpr int kKT = 16;       // K per shared-memory stage
constexpr int kThreads = 256;

__device__ __forceinline__ float act_f(int a, float v) { return a == kActTanh ? tanhf(v) : fmaxf(v, 0.0f); }

__host__ __device__ __forceinline__ int odd_ld(int w) { return w + ((w & 1) == 0 ? 1 : 0); }

// One block = one spark row x 128 samples.  Layer 1 is a register-tiled
// SIMT GEMM (each thread 8 samples x 4 hidden units); the activated hidden
// tile stays in shared memory, later layers run one sample per thread, and
// the block's cross-entropy sum goes to partial[mt][row].
__global__ void __launch_bounds__(kThreads) k_fitness_simt(Mlp mlp, const float* __restrict__ rows, int64_t ld,
                                                           int32_t count, float* __restrict__ partial) {
  griddep_wait();
  griddep_launch_dependents();
  extern __shared__ __align__(16) float smem[];
  const int row = blockIdx.x, mt = blockIdx.y;
  const float* w = rows + (int64_t)row * ld;
  const int L = mlp.n_layers;
  const int d_in = mlp.widths[0], h1 = mlp.widths[1];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  int ldmax = 0;
  for (int l = 1; l <= L; ++l) ldmax = max(ldmax, odd_ld(mlp.widths[l]));
  float* Xs = smem;                 // [kKT][kMT]
  float* Ws = Xs + kKT * kMT;       // [kKT][kHC]
  float* bufA = Ws + kKT * kHC;     // [kMT][ldmax]
  float* bufB = bufA + kMT * ldmax; // [kMT][ldmax]
  const int64_t n0 = (int64_t)mt * kMT;
  const float* b1 = w + mlp.b_off[0];
  const int ldh = odd_ld(h1);

  for (int hc = 0; hc < h1; hc += kHC) {
    float acc[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = 0.0f;
    for (int k0 = 0; k0 < d_in; k0 += kKT) {
      {
        const int nl = tid >> 1, kk = (tid & 1) * 8;
        const int64_t n = n0 + nl;
        float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = a0;
        if (n < mlp.N) {
          const float* xr = mlp.X + n * d_in + k0 + kk;
          if (k0 + kk < d_in) a0 = *reinterpret_cast<const float4*>(xr);
          if (k0 + kk + 4 < d_in) a1 = *reinterpret_cast<const float4*>(xr + 4);
        }
        Xs[(kk + 0) * kMT + nl] = a0.x; Xs[(kk + 1) * kMT + nl] = a0.y;
        Xs[(kk + 2) * kMT + nl] = a0.z; Xs[(kk + 3) * kMT + nl] = a0.w;
        Xs[(kk + 4) * kMT + nl] = a1.x; Xs[(kk + 5) * kMT + nl] = a1.y;
        Xs[(kk + 6) * kMT + nl] = a1.z; Xs[(kk + 7) * kMT + nl] = a1.w;
      }
      {
        const int j = tid >> 2, kq = (tid & 3) * 4;
        float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
        if (hc + j < h1 && k0 + kq < d_in) b = *reinterpret_cast<const float4*>(w + (int64_t)(hc + j) * d_in + k0 + kq);
        Ws[(kq + 0) * kHC + j] = b.x; Ws[(kq + 1) * kHC + j] = b.y;
        Ws[(kq + 2) * kHC + j] = b.z; Ws[(kq + 3) * kHC + j] = b.w;
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < kKT; ++kk) {
        const float4 xa = *reinterpret_cast<const float4*>(Xs + kk * kMT + ty * 8);
        const float4 xb = *reinterpret_cast<const float4*>(Xs + kk * kMT + ty * 8 + 4);
        const float4 wv = *reinterpret_cast<const float4*>(Ws + kk * kHC + tx * 4);
        const float xr[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
        const float wr[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(xr[a], wr[b], acc[a][b]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int jj = hc + tx * 4 + b;
      if (jj < h1) {
        const float bias = b1[jj];
#pragma unroll
        for (int a = 0; a < 8; ++a) bufA[(ty * 8 + a) * ldh + jj] = act_f(mlp.acts[0], acc[a][b] + bias);
      }
    }
  }
  __syncthreads();

  float* in = bufA;
  int ldin = ldh;
  float* out = bufB;
  const int nl = tid & (kMT - 1), half = tid >> 7;
  for (int l = 1; l < L; ++l) {
    const int fi = mlp.widths[l], fo = mlp.widths[l + 1];
    const float* Wl = w + mlp.w_off[l];
    const float* bl = w + mlp.b_off[l];
    const int ldo = odd_ld(fo);
    const bool hidden = l + 1 < L;
    const float* a = in + nl * ldin;
    for (int j = half; j < fo; j += 2) {
      const float* wr = Wl + (int64_t)j * fi;
      float s = bl[j];
      for (int i = 0; i < fi; ++i) s = fmaf(wr[i], a[i], s);
      out[nl * ldo + j] = hidden ? act_f(mlp.acts[l], s) : s;
    }
    __syncthreads();
    float* t = in; in = out; out = t;
    ldin = ldo;
  }

  __shared__ float red[kThreads / 32];
  float ce = 0.0f;
  const int64_t n = n0 + tid;
  if (tid < kMT && n < mlp.N) {
    const float* z = in + tid * ldin;
    const int C = mlp.widths[L];
    float zmax = z[0];
    for (int c = 1; c < C; ++c) zmax = fmaxf(zmax, z[c]);
    float se = 0.0f;
    for (int c = 0; c < C; ++c) se += expf(z[c] - zmax);
    ce = (zmax + logf(se)) - z[mlp.y[n]];
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) ce += __shfl_xor_sync(0xffffffffu, ce, off);
  if ((tid & 31) == 0) red[tid >> 5] = ce;
  __syncthreads();
  if (tid == 0) {
    float s = red[0];
    for (int wi = 1; wi < kMT / 32; ++wi) s += red[wi];
    partial[(int64_t)mt * count + row] = s;
  }
}

// Small two-layer networks (d_in = DI, h1 = H1, C classes, all compile-time):
// one thread = one sample (its inputs in registers) of one spark, whose row is
// staged in shared memory and read as broadcasts.  Each hidden unit is
// accumulated over the inputs in ascending order from zero, then the bias is
// added and the activation applied, and each logit starts from its bias and
// accumulates the hidden units in ascending order: the same operations in the
// same order as k_fitness_simt, so every kernel here gives bitwise the same
// fitness.
template <int DI, int H1, int C>
struct SmallNet {
  static constexpr int D = DI * H1 + H1 + C * H1 + C;  // parameters per spark (nn.Linear order)
  static constexpr int kB1 = DI * H1, kW2 = kB1 + H1, kB2 = kW2 + C * H1;
  // cross-entropy of one sample
  static __device__ __forceinline__ float ce(const float* W, const float* x, int label, int act) {
    float z[C];
#pragma unroll
    for (int c = 0; c < C; ++c) z[c] = W[kB2 + c];
#pragma unroll
    for (int j = 0; j < H1; ++j) {
      float a = 0.0f;
#pragma unroll
      for (int i = 0; i < DI; ++i) a = fmaf(x[i], W[j * DI + i], a);
      a = act_f(act, a + W[kB1 + j]);
#pragma unroll
      for (int c = 0; c < C; ++c) z[c] = fmaf(W[kW2 + c * H1 + j], a, z[c]);
    }
    float zmax = z[0];
#pragma unroll
    for (int c = 1; c < C; ++c) zmax = fmaxf(zmax, z[c]);
    float se = 0.0f;
#pragma unroll
    for (int c = 0; c < C; ++c) se += expf(z[c] - zmax);
    float zy = z[0];
#pragma unroll
    for (int c = 1; c < C; ++c) zy = label == c ? z[c] : zy;
    return (zmax + logf(se)) - zy;
  }
};

// One block = 128 samples x up to `per` sparks, one after another; the
// block's cross-entropy sum per spark goes to partial[mt][row] (warp sums
// added in warp order, as in k_fitness_simt).  What bounds a small launch is
// the chain of one spark's 16 activations times the sparks a block takes in
// turn, so the launcher gives each block one spark until the blocks fill the
// GPU (200 and 20 sparks x 512 samples with eight per block: 14.3 us a
// launch either way; with one, whole generations went from 91 to 30 us).
constexpr int kSmallSparks = 8;
// Blocks per SM that the registers must allow, 40 a thread.  Left to itself the compiler takes 32, whose order of the
// chains costs a small launch 1 us of 4 (a run of 90 generations 2,855 us, 2,670 so); 64 gain as much again there but
// lose 2% where the blocks fill the GPU (N = 131,072, 200 sparks: 94.7 us, 93.9 so).
constexpr int kSmallBlocks = 12;

template <int DI, int H1, int C>
__global__ void __launch_bounds__(kMT, kSmallBlocks) k_fitness_small(Mlp mlp, const float* __restrict__ rows, int64_t ld,
                                                       int32_t count, int32_t per, float* __restrict__ partial) {
  using Net = SmallNet<DI, H1, C>;
  __shared__ float ws[kSmallSparks][Net::D];
  __shared__ float red[kSmallSparks][kMT / 32];
  griddep_wait();
  griddep_launch_dependents();
  const int s0 = blockIdx.x * per, mt = blockIdx.y;
  const int gs = min(per, count - s0);
  for (int g = 0; g < gs; ++g) {
    const float* row = rows + (int64_t)(s0 + g) * ld;
#pragma unroll
    for (int k0 = 0; k0 < Net::D; k0 += kMT)
      if (k0 + (int)threadIdx.x < Net::D) ws[g][k0 + threadIdx.x] = row[k0 + threadIdx.x];
  }
  const int64_t n = (int64_t)mt * kMT + threadIdx.x;
  const bool valid = n < mlp.N;
  float x[DI];
#pragma unroll
  for (int i = 0; i < DI; ++i) x[i] = valid ? mlp.X[n * DI + i] : 0.0f;
  const int label = valid ? mlp.y[n] : 0;
  const int act = mlp.acts[0];
  __syncthreads();
  for (int g = 0; g < gs; ++g) {
    float ce = valid ? Net::ce(ws[g], x, label, act) : 0.0f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ce += __shfl_xor_sync(0xffffffffu, ce, off);
    if ((threadIdx.x & 31) == 0) red[g][threadIdx.x >> 5] = ce;
  }
  __syncthreads();
  if ((int)threadIdx.x < gs) {
    float v = red[threadIdx.x][0];
#pragma unroll
    for (int wi = 1; wi < kMT / 32; ++wi) v += red[threadIdx.x][wi];
    partial[(int64_t)mt * count + s0 + threadIdx.x] = v;
  }
}

// True if the network is one that k_fitness_small is instantiated for, with
// the parameter layout it assumes.
bool small_net(const Mlp& mlp, int di, int h1, int c) {
  return mlp.n_layers == 2 && mlp.widths[0] == di && mlp.widths[1] == h1 && mlp.widths[2] == c &&
         mlp.w_off[0] == 0 && mlp.b_off[0] == (int64_t)di * h1 && mlp.w_off[1] == mlp.b_off[0] + h1 &&
         mlp.b_off[1] == mlp.w_off[1] + (int64_t)c * h1;
}

__global__ void k_fitness_finish(const float* __restrict__ partial, int32_t mtiles, int32_t count, float n_f,
                                 float* __restrict__ fit) {
  griddep_wait();
  griddep_launch_dependents();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= count) return;
  fit[r] = __fdiv_rn(tile_sum(partial, r, count, mtiles), n_f);
}

__global__ void __launch_bounds__(256) k_sphere(const float* __restrict__ rows, int64_t ld, int64_t D,
                                                float* __restrict__ fit) {
  griddep_wait();
  griddep_launch_dependents();
  __shared__ float red[8];
  const float* x = rows + (int64_t)blockIdx.x * ld;
  float s = 0.0f;
  for (int64_t d = threadIdx.x; d < D; d += blockDim.x) s = fmaf(x[d], x[d], s);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = red[0];
    for (int w = 1; w < 8; ++w) t += red[w];
    fit[blockIdx.x] = t;
  }
}

// FP64 forward of ns (<= kF64Samples) samples per block.  The FP64 pipe is
// what bounds it (about two FMAs a clock per SM, conversions from FP32 on the
// same pipe), so it should carry little else: 64 units x 32 inputs of a layer's
// weights (and, in the first layer, the samples' inputs) are converted once
// into shared memory, the next slab's loads in flight meanwhile, and each
// thread sums up to four (unit, sample) outputs, no lane reductions.  Each
// slab of 32 inputs is a chain of its own from zero in index order and the
// slabs are added in order, so the rounding error grows like a tree's.  The
// launcher picks ns so that the blocks fill whole waves of the SMs.  A run's
// read-back of the 784-64-10 network (N = 2048) 431 -> 306 us with it, of
// 3072-128-64-10 (N = 4096) 4,366 -> 3,290 us; before, four samples a block,
// a fifth of the pipe went to lane reductions and a quarter to conversions.
constexpr int kF64Samples = 16;
constexpr int kF64Units = 64, kF64K = 32, kF64Threads = 256;
constexpr int kF64Out = kF64Samples * kF64Units / kF64Threads;  // outputs per thread

__global__ void __launch_bounds__(kF64Threads) k_fitness_f64(Mlp mlp, const float* __restrict__ x, int ns, int wmax,
                                                             double* __restrict__ ce64) {
  griddep_wait();
  griddep_launch_dependents();
  extern __shared__ double sd[];
  double* ws = sd;                                  // [kF64Units][kF64K + 1]
  double* xs = ws + kF64Units * (kF64K + 1);        // [kF64K][kF64Samples]
  double* a = xs + kF64K * kF64Samples;             // [wmax][kF64Samples], wmax the widest layer output
  double* b = a + (size_t)wmax * kF64Samples;
  const int tid = threadIdx.x;
  const int64_t n0 = (int64_t)blockIdx.x * ns;
  const int L = mlp.n_layers;
  constexpr int kWL = kF64Units * kF64K / kF64Threads, kXL = kF64Samples * kF64K / kF64Threads;
  for (int l = 0; l < L; ++l) {
    const int fi = mlp.widths[l], fo = mlp.widths[l + 1];
    for (int u0 = 0; u0 < fo; u0 += kF64Units) {
      const int uc = min(kF64Units, fo - u0);
      const float* W = x + mlp.w_off[l] + (int64_t)u0 * fi;
      float wr[kWL], xr[kXL];
      auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < kWL; ++i) {
          const int e = tid + kF64Threads * i, u = e / kF64K, k = k0 + e % kF64K;
          wr[i] = u < uc && k < fi ? W[(int64_t)u * fi + k] : 0.0f;
        }
        if (l == 0) {
#pragma unroll
          for (int i = 0; i < kXL; ++i) {
            const int e = tid + kF64Threads * i, q = e / kF64K, k = k0 + e % kF64K;
            xr[i] = q < ns && n0 + q < mlp.N && k < fi ? mlp.X[(n0 + q) * fi + k] : 0.0f;
          }
        }
      };
      int unit[kF64Out], smp[kF64Out];
      double acc[kF64Out];
#pragma unroll
      for (int q = 0; q < kF64Out; ++q) {
        const int o = tid + kF64Threads * q;
        unit[q] = o / ns;
        smp[q] = o - unit[q] * ns;
        acc[q] = 0.0;
      }
      fetch(0);
      for (int k0 = 0; k0 < fi; k0 += kF64K) {
        __syncthreads();  // the slab before has been read
#pragma unroll
        for (int i = 0; i < kWL; ++i) {
          const int e = tid + kF64Threads * i;
          ws[e / kF64K * (kF64K + 1) + e % kF64K] = (double)wr[i];
        }
        if (l == 0) {
#pragma unroll
          for (int i = 0; i < kXL; ++i) {
            const int e = tid + kF64Threads * i;
            xs[e % kF64K * kF64Samples + e / kF64K] = (double)xr[i];
          }
        }
        __syncthreads();
        if (k0 + kF64K < fi) fetch(k0 + kF64K);
        const int kk = min(kF64K, fi - k0);
        const double* in = l == 0 ? xs : a + (size_t)k0 * kF64Samples;
#pragma unroll
        for (int q = 0; q < kF64Out; ++q) {
          if (unit[q] >= uc) continue;
          const double* wq = ws + unit[q] * (kF64K + 1);
          double p = 0.0;
#pragma unroll 8
          for (int k = 0; k < kk; ++k) p += wq[k] * in[k * kF64Samples + smp[q]];
          acc[q] += p;
        }
      }
#pragma unroll
      for (int q = 0; q < kF64Out; ++q) {
        if (unit[q] >= uc) continue;
        double v = acc[q] + (double)x[mlp.b_off[l] + u0 + unit[q]];
        if (l + 1 < L) v = mlp.acts[l] == kActTanh ? tanh(v) : (v > 0.0 ? v : 0.0);
        b[(u0 + unit[q]) * kF64Samples + smp[q]] = v;
      }
    }
    __syncthreads();
    double* t = a; a = b; b = t;
  }
  if (tid < ns && n0 + tid < mlp.N) {
    const double* z = a + tid;
    const int C = mlp.widths[L];
    double zmax = z[0];
    for (int c = 1; c < C; ++c) zmax = z[c * kF64Samples] > zmax ? z[c * kF64Samples] : zmax;
    double se = 0.0;
    for (int c = 0; c < C; ++c) se += exp(z[c * kF64Samples] - zmax);
    ce64[n0 + tid] = (zmax + log(se)) - z[mlp.y[n0 + tid] * kF64Samples];
  }
}

// Fixed-order mean (or sum of squares) in FP64 by one block.
__global__ void __launch_bounds__(256) k_reduce_f64(const double* __restrict__ v, const float* __restrict__ xf,
                                                    int64_t n, double scale, double* __restrict__ out) {
  griddep_wait();
  griddep_launch_dependents();
  __shared__ double red[256];
  double s = 0.0;
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
    if (xf != nullptr) {
      const double t = (double)xf[e];
      s += t * t;
    } else {
      s += v[e];
    }
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0] * scale;
}

size_t smem_for(const Mlp& mlp) {
  int ldmax = 0;
  for (int l = 1; l <= mlp.n_layers; ++l) ldmax = ldmax > odd_ld(mlp.widths[l]) ? ldmax : odd_ld(mlp.widths[l]);
  return sizeof(float) * ((size_t)kKT * kMT + (size_t)kKT * kHC + 2 * (size_t)kMT * ldmax);
}

}  // namespace

// What k_fitness_simt takes for 128 samples of a spark, as a share of an SM
// (fitted, as tile_ns in k_fitness_x3.cu): the first layer in steps of 16
// inputs and 64 hidden units, the later ones a sample a thread.  Where the
// activations leave room for one block per SM only it is a third slower.
int64_t fitness_simt_ns(const Mlp& mlp) {
  const int L = mlp.n_layers, h1 = mlp.widths[1], h2 = L == 3 ? mlp.widths[2] : 0;
  const int64_t pairs = (int64_t)(h2 + 1) / 2 * h1 + (int64_t)(mlp.widths[L] + 1) / 2 * mlp.widths[L - 1];
  const int64_t ns = 69LL * ((mlp.widths[0] + kKT - 1) / kKT * kKT) * ((h1 + kHC - 1) / kHC) + 18 * h1 + 11 * pairs +
                     (mlp.acts[0] == kActTanh ? 9 * h1 : 0) + (L == 3 && mlp.acts[1] == kActTanh ? 9 * h2 : 0);
  const size_t blocks = 232448 / (smem_for(mlp) + 1024);  // 227 KB per SM, 1 KB of each block's reserved
  return blocks < 2 ? ns * 4 / 3 : blocks > 2 ? ns * 9 / 10 : ns;
}

int launch_fitness_finish(const float* partial, int32_t mtiles, int32_t count, int64_t N, float* fit, cudaStream_t s) {
  if (count <= 0) return 0;
  return launch_pdl(k_fitness_finish, dim3((count + 255) / 256), dim3(256), 0, s, partial, mtiles, count, (float)N,
                    fit) == cudaSuccess
             ? 1
             : -1;
}

int launch_fitness_fp32(const Mlp& mlp, const float* rows, int64_t ld, int32_t count, float* partial,
                        uint32_t* status, uint64_t wait_budget, cudaStream_t s) {
  if (count <= 0) return 0;
  const int mtiles = (int)((mlp.N + kMT - 1) / kMT);
  if (small_net(mlp, 8, 16, 3)) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return -1;
    // one spark per block while one block per SM slot (16 of 128 threads) holds them, then up to kSmallSparks
    const int64_t pairs = (int64_t)count * mtiles, slots = (int64_t)sms * 16;
    const int per = (int)(pairs <= slots ? 1 : (pairs / slots < kSmallSparks ? pairs / slots : kSmallSparks));
    dim3 grid((count + per - 1) / per, mtiles);
    return launch_pdl(k_fitness_small<8, 16, 3>, grid, dim3(kMT), 0, s, mlp, rows, ld, count, (int32_t)per, partial) ==
                   cudaSuccess
               ? 1
               : -1;
  }
  if (fitness_x3_ok(mlp)) return launch_fitness_x3(mlp, rows, ld, count, partial, status, wait_budget, s);
  const size_t smem = smem_for(mlp);
  if (ensure_smem_limit<k_fitness_simt>(smem) != cudaSuccess) return -1;
  dim3 grid(count, mtiles);
  return launch_pdl(k_fitness_simt, grid, dim3(kThreads), smem, s, mlp, rows, ld, count, partial) == cudaSuccess
             ? 1
             : -1;
}

int launch_fitness_sphere(const float* rows, int64_t ld, int64_t D, int32_t count, float* fit, cudaStream_t s) {
  if (count <= 0) return 0;
  return launch_pdl(k_sphere, dim3(count), dim3(256), 0, s, rows, ld, D, fit) == cudaSuccess ? 1 : -1;
}

int launch_fitness_f64(const Mlp& mlp, const float* x, double* ce64, double* out, cudaStream_t s) {
  int dev = 0, sms = 0, wmax = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return -1;
  for (int l = 1; l <= mlp.n_layers; ++l) wmax = wmax > mlp.widths[l] ? wmax : mlp.widths[l];
  const int64_t waves = (mlp.N + (int64_t)kF64Samples * sms - 1) / ((int64_t)kF64Samples * sms);
  const int ns = (int)((mlp.N + waves * sms - 1) / (waves * sms));
  const size_t smem = sizeof(double) * ((size_t)kF64Units * (kF64K + 1) + (size_t)kF64K * kF64Samples +
                                        2 * (size_t)wmax * kF64Samples);
  if (smem > 48 * 1024 && ensure_smem_limit<k_fitness_f64>(smem) != cudaSuccess) return -1;
  k_fitness_f64<<<(unsigned)((mlp.N + ns - 1) / ns), kF64Threads, smem, s>>>(mlp, x, ns, wmax, ce64);
  if (cudaPeekAtLastError() != cudaSuccess) return -1;
  k_reduce_f64<<<1, 256, 0, s>>>(ce64, nullptr, mlp.N, 1.0 / (double)mlp.N, out);
  return cudaPeekAtLastError() == cudaSuccess ? 2 : -1;
}

int launch_sphere_f64(const float* x, int64_t D, double* out, cudaStream_t s) {
  k_reduce_f64<<<1, 256, 0, s>>>(nullptr, x, D, 1.0, out);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace mgfwa

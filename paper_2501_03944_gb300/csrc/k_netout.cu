// The paper's own testbed objective (Sec. 4.1, Eq. 1): the scalar output of
// a fixed network whose input is the search vector,
//   a_0 = x;  a_l = act(W_l a_{l-1} + b_l) for hidden layers;  f = W_L a_{L-1} + b_L.
// Here the sparks are the rows of a batch and the weights are shared, so each
// layer is one dense product [rows x fan_in] x [fan_in x fan_out] with the
// bias and the activation in its epilogue (FP32 on the CUDA cores).  The
// summation order of every output is fixed by the layer's fan-in alone (four
// contiguous chunks of i, each a chain of fmaf in index order, the chunk sums
// added in chunk order, then the bias), so a spark's fitness does not depend
// on which sparks share the launch.  The last layer writes the fitness.  An
// FP64 forward of one vector (a launch per layer) gives the reported best
// fitness.
#include "mgfwa_internal.cuh"

namespace mgfwa {

namespace {

constexpr int kBK = 16;      // k-slab depth
constexpr int kGroups = 4;   // fan-in chunks, one per 64-thread group
constexpr int kPadK = kBK + 4;   // slab row stride: eight rows' float4s lie in distinct banks

// Tile geometry for TR x TC outputs per thread: 8 TR rows x 8 TC columns per
// block, ST slabs of A and W in flight per group (cp.async ring).
template <int TR, int TC, int ST>
struct NetTile {
  static constexpr int kTM = 8 * TR, kTN = 8 * TC;
  static constexpr int kPadW = kTN + 8;                // partial tile row stride
  static constexpr int kSlab = (kTM + kTN) * kPadK;  // A rows, then W rows, k contiguous
  static constexpr int kGroupFloats = ST * kSlab;
  static constexpr size_t kSmem = sizeof(float) * kGroups * kGroupFloats;
  static_assert(kTM * kPadW <= kGroupFloats, "partial tiles must fit in the slab space");
};

__device__ __forceinline__ float act32(int a, float v) {
  if (a == kActTanh) return tanhf(v);
  if (a == kActGelu) return 0.5f * v * (1.0f + erff(v * 0.70710678118654752f));
  return fmaxf(v, 0.0f);
}

// 4- and 16-byte asynchronous global -> shared copies; src_bytes = 0 writes
// zeros without reading (the source address must still be a valid one).
__device__ __forceinline__ void cp_async4(float* dst, const float* src, uint32_t src_bytes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src, uint32_t src_bytes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The fan-in chunk of group g: [g c, min((g + 1) c, k)) with c = 16 ceil(k / 64).
__host__ __device__ __forceinline__ int chunk_len(int k) { return kBK * ((k + kBK * kGroups - 1) / (kBK * kGroups)); }

// out[r][j] = act(sum_i A[r][i] W[j][i] + b[j]) (no activation when act < 0)
// for r < rows, j < n; A row stride lda, out row stride ldo.  One 256-thread
// block per (8 TR) x (8 TC) output tile.  Group g (threads 64 g ..) multiplies
// the tile over its fan-in chunk, TR x TC outputs per thread (rows ty + 8 i,
// columns tx + 8 j): k-slabs of A and W rows are copied asynchronously into
// the group's ring of ST slabs as they lie in memory (V4: 16 bytes at a
// time, else 4), ST - 1 slabs in flight while one is multiplied, one group
// barrier per slab; a thread reads four k of a row per 16-byte shared load.
// The four partial tiles then meet in shared memory and every thread adds
// them in group order for TR of the tile's outputs, adds the bias and applies
// the activation.  A quarter of the fan-in per group cuts each block's serial
// slab chain to a quarter, which is what bounds the small-row launches (the
// guiding sparks).  The weights do not depend on the previous kernel, so the
// first slabs' W rows are copied before its end is waited for.  Every shape
// computes every output with the same operations in the same order, so the
// choice never changes a result.
template <int TR, int TC, int ST, bool V4>
__global__ void __launch_bounds__(256, TR * TC > 32 ? 1 : TR == 4 ? 3 : 2)
    k_net_layer(const float* __restrict__ A, int64_t lda, int32_t rows, const float* __restrict__ W,
                const float* __restrict__ bias, int32_t k, int32_t n, int32_t act, float* __restrict__ out,
                int64_t ldo) {
  using Tile = NetTile<TR, TC, ST>;
  constexpr int kTM = Tile::kTM, kTN = Tile::kTN, kPadW = Tile::kPadW, kW = V4 ? 4 : 1;  // kW floats per copy
  // slabs [group][stage]{A [kTM][kPadK], W [kTN][kPadK]}; afterwards the partial tiles [group][kTM][kPadW]
  extern __shared__ __align__(16) float sm[];
  const int g = threadIdx.x >> 6, t = threadIdx.x & 63;
  const int tx = t & 7, ty = t >> 3;
  const int r0 = blockIdx.x * kTM, j0 = blockIdx.y * kTN;  // row tiles on x: up to 2^24 rows
  const int c = chunk_len(k);
  const int kbeg = g * c, kend = min(kbeg + c, k);
  const int slabs = kend > kbeg ? (kend - kbeg + kBK - 1) / kBK : 0;
  float* const base = sm + g * Tile::kGroupFloats;
  // a thread copies k offset kq of slab rows rq, rq + kRows, ...: neighbouring
  // threads read one row's consecutive floats
  constexpr int kPer = kBK / kW, kRows = 64 / kPer;
  const int kq = (t % kPer) * kW, rq = t / kPer;
  auto copy = [&](float* dst, const float* src, bool in, const float* safe) {
    if (V4)
      cp_async16(dst, in ? src : safe, in ? 16u : 0u);
    else
      cp_async4(dst, in ? src : safe, in ? 4u : 0u);
  };
  auto fetch_w = [&](int slab, int stage) {
    const int k0 = kbeg + slab * kBK + kq;
    float* w = base + stage * Tile::kSlab + kTM * kPadK + kq;
#pragma unroll
    for (int q = rq; q < kTN; q += kRows)
      copy(w + q * kPadK, W + (int64_t)(j0 + q) * k + k0, k0 < kend && j0 + q < n, W);
  };
  auto fetch_a = [&](int slab, int stage) {
    const int k0 = kbeg + slab * kBK + kq;
    float* a = base + stage * Tile::kSlab + kq;
#pragma unroll
    for (int q = rq; q < kTM; q += kRows)
      copy(a + q * kPadK, A + (int64_t)(r0 + q) * lda + k0, k0 < kend && r0 + q < rows, A);
  };
  auto group_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(g + 1) : "memory"); };
  float acc[TR][TC];
#pragma unroll
  for (int i = 0; i < TR; ++i)
#pragma unroll
    for (int j = 0; j < TC; ++j) acc[i][j] = 0.0f;
#pragma unroll
  for (int i = 0; i < ST - 1; ++i)
    if (i < slabs) fetch_w(i, i);
  griddep_wait();
  griddep_launch_dependents();
#pragma unroll
  for (int i = 0; i < ST - 1; ++i) {
    if (i < slabs) fetch_a(i, i);
    cp_async_commit();  // the first of these groups also holds the W copies above
  }
  for (int s = 0; s < slabs; ++s) {
    cp_async_wait<ST - 2>();  // this thread's copies of slab s have landed
    group_sync();             // everyone's have; everyone is done with slab s - 1
    const float* a = base + (s % ST) * Tile::kSlab + ty * kPadK;
    const float* w = base + (s % ST) * Tile::kSlab + (kTM + tx) * kPadK;
#pragma unroll
    for (int kk = 0; kk < kBK; kk += 4) {
      float4 av[TR], wv[TC];
#pragma unroll
      for (int i = 0; i < TR; ++i) av[i] = *reinterpret_cast<const float4*>(a + 8 * i * kPadK + kk);
#pragma unroll
      for (int j = 0; j < TC; ++j) wv[j] = *reinterpret_cast<const float4*>(w + 8 * j * kPadK + kk);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
          for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(lane_of(av[i], u), lane_of(wv[j], u), acc[i][j]);
    }
    // the ring slot of slab s + ST - 1 last held slab s - 1, which every
    // thread of the group finished before the barrier above
    if (s + ST - 1 < slabs) {
      fetch_w(s + ST - 1, (s + ST - 1) % ST);
      fetch_a(s + ST - 1, (s + ST - 1) % ST);
    }
    cp_async_commit();
  }
  cp_async_wait<0>();
  __syncthreads();  // every group done with its slabs: the space holds the partial tiles now
  float* part = sm + g * (kTM * kPadW);
#pragma unroll
  for (int i = 0; i < TR; ++i)
#pragma unroll
    for (int j = 0; j < TC; ++j) part[(ty + 8 * i) * kPadW + tx + 8 * j] = acc[i][j];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kTM * kTN / 256; ++q) {
    const int o = threadIdx.x + 256 * q, rr = o / kTN, cc = o % kTN;
    const int r = r0 + rr, j = j0 + cc;
    if (r >= rows || j >= n) continue;
    float z = sm[rr * kPadW + cc];
#pragma unroll
    for (int h = 1; h < kGroups; ++h) z += sm[h * (kTM * kPadW) + rr * kPadW + cc];
    z += bias[j];
    out[(int64_t)r * ldo + j] = act >= 0 ? act32(act, z) : z;
  }
}

// One layer of the FP64 forward of one vector: one warp per output, lanes
// striding over the fan-in in index order (coalesced weight reads), then a
// fixed xor tree and the bias.  `xin` is the FP32 vector for the first layer,
// `ain` the previous layer's FP64 outputs otherwise.  The layer's weights are
// read once by as many SMs as it has warps; one block reading every row
// through its own threads, uncoalesced, was one SM's latency-bound chain
// (reading back a run of the
// 1000-512x11-1 network 1,903 us so, 125 us with these 12 launches).
constexpr int kF64Warps = 4;

__global__ void __launch_bounds__(32 * kF64Warps) k_net_f64_layer(const float* __restrict__ W,
                                                                  const float* __restrict__ bias, int32_t fi,
                                                                  int32_t fo, int32_t act,
                                                                  const float* __restrict__ xin,
                                                                  const double* __restrict__ ain,
                                                                  double* __restrict__ out) {
  const int j = blockIdx.x * kF64Warps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  griddep_wait();
  griddep_launch_dependents();
  if (j >= fo) return;
  const float* w = W + (int64_t)j * fi;
  double s = 0.0;
#pragma unroll 8
  for (int i = lane; i < fi; i += 32) s += (double)w[i] * (xin != nullptr ? (double)xin[i] : ain[i]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane != 0) return;
  s += (double)bias[j];
  if (act >= 0)
    s = act == kActTanh ? tanh(s)
                        : (act == kActGelu ? 0.5 * s * (1.0 + erf(s * 0.70710678118654752440)) : fmax(s, 0.0));
  out[j] = s;
}

}  // namespace

namespace {
struct NetLaunch {
  const float* a;
  int64_t lda;
  int32_t count;
  const float *W, *b;
  int32_t fi, fo, ak;
  float* o;
  int64_t ldo;
};

template <int TR, int TC, int ST, bool V4>
cudaError_t net_layer(const NetLaunch& n, cudaStream_t s) {
  using Tile = NetTile<TR, TC, ST>;
  const cudaError_t e = ensure_smem_limit<k_net_layer<TR, TC, ST, V4>>(Tile::kSmem);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)((n.count + Tile::kTM - 1) / Tile::kTM), (unsigned)((n.fo + Tile::kTN - 1) / Tile::kTN));
  return launch_pdl(k_net_layer<TR, TC, ST, V4>, grid, dim3(256), Tile::kSmem, s, n.a, n.lda, n.count, n.W, n.b, n.fi,
                    n.fo, n.ak, n.o, n.ldo);
}

template <int TR, int TC, int ST>
cudaError_t net_layer(const NetLaunch& n, bool v4, cudaStream_t s) {
  return v4 ? net_layer<TR, TC, ST, true>(n, s) : net_layer<TR, TC, ST, false>(n, s);
}
}  // namespace

int launch_net_layer(const float* a, int64_t lda, int32_t count, const float* W, const float* b, int32_t fi,
                     int32_t fo, int32_t ak, float* o, int64_t ldo, cudaStream_t s) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                 cudaSuccess)
    return -1;
  // 16-byte copies where every row of both operands starts on 16 bytes (a
  // chunk starts at a multiple of 16, and k % 4 == 0 makes its end whole)
  const bool v4 = fi % 4 == 0 && lda % 4 == 0 &&
                  ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(W)) & 15u) == 0;
  const NetLaunch n = {a, lda, count, W, b, fi, fo, ak, o, ldo};
  auto blocks = [&](int tm, int tn) { return (int64_t)((count + tm - 1) / tm) * ((fo + tn - 1) / tn); };
  // Tiles of 64 x 64 where they occupy most SMs (a thread's 16 shared loads
  // then serve 256 FMAs, 12 serve 128 with 64 x 32, and the width of those
  // loads bounds the multiply: 1,000 x 512 x 512 22.5 us with 64 x 32, 20.6 us
  // with 64 x 64, caches cold), else the widest tile that fills the SMs; with
  // few rows 8-row tiles with eight slabs in flight (latency-bound: 40 x 512 x
  // 512 11.2 us with 32-row tiles, 7.2 us with these).
  cudaError_t e;
  if (4 * blocks(64, 64) >= 3 * sms)
    e = net_layer<8, 8, 4>(n, v4, s);
  else if (blocks(64, 32) >= sms)
    e = net_layer<8, 4, 3>(n, v4, s);
  else if (blocks(32, 32) >= sms)
    e = net_layer<4, 4, 3>(n, v4, s);
  else
    e = net_layer<1, 4, 8>(n, v4, s);
  return e == cudaSuccess ? 1 : -1;
}

int launch_net_output(const NetOut& net, const float* rows, int64_t ld, int32_t count, float* fit, float* scratch,
                      int64_t scratch_ld, cudaStream_t s) {
  if (count <= 0) return 0;
  const float* a = rows;
  int64_t lda = ld;
  int n = 0;
  for (int l = 0; l < net.n_layers; ++l) {
    const int fi = net.widths[l], fo = net.widths[l + 1];
    const bool last = l + 1 == net.n_layers;
    float* o = last ? fit : scratch + (int64_t)(l & 1) * scratch_ld * count;
    const int64_t ldo = last ? 1 : scratch_ld;
    if (launch_net_layer(a, lda, count, net.params + net.w_off[l], net.params + net.b_off[l], fi, fo,
                         last ? -1 : net.acts[l], o, ldo, s) < 0)
      return -1;
    ++n;
    a = o;
    lda = ldo;
  }
  return n;
}

int launch_net_output_f64(const NetOut& net, const float* x, double* scratch, double* out, cudaStream_t s) {
  const double* in = nullptr;
  for (int l = 0; l < net.n_layers; ++l) {
    const int fi = net.widths[l], fo = net.widths[l + 1];
    const bool last = l + 1 == net.n_layers;
    double* o = last ? out : scratch + (int64_t)(l & 1) * net.wmax;
    if (launch_pdl(k_net_f64_layer, dim3((unsigned)((fo + kF64Warps - 1) / kF64Warps)), dim3(32 * kF64Warps), 0, s,
                   net.params + net.w_off[l], net.params + net.b_off[l], fi, fo, last ? -1 : net.acts[l],
                   l == 0 ? x : (const float*)nullptr, in, o) != cudaSuccess)
      return -1;
    in = o;
  }
  return net.n_layers;
}

}  // namespace mgfwa

// FP32 fitness of spark rows with the first layer on the tensor cores at FP32
// accuracy: per-(sample tile, spark) cross-entropy sums, as k_fitness_simt
// gives them, straight from the FP32 rows and X (no operand copies, no
// workspace).
//
// The first layer is the contraction (N x d_in) . (d_in x h1 per spark); on
// the CUDA cores it is bound by FP32 FMA issue (k_fitness_simt: 34 TFLOP/s of
// the lanes' 80 on the 784-64-10 network).  Here each FP32 operand v is split
// into three BF16 parts, v1 = bf16(v), v2 = bf16(v - v1), v3 = bf16(v - v1 -
// v2), and six tcgen05 kind::f16 products per 16 inputs (a1b1, a1b2, a2b1,
// a2b2, a1b3, a3b1) leave out terms below about 2^-25 of each product, under
// FP32's own rounding.  The tensor core's accumulation truncates, so no sum
// runs in it for long: every block of 32 inputs starts a fresh TMEM
// accumulator (its corrections first, its two main products last) and the
// blocks are added in FP32 registers in block order, rounded to nearest.
//
// Measured (N = 2048, 784-64-10, 1,000 sparks): k_fitness_simt 6,042 us, here
// 1,600 us; 3072-128-64-10, N = 4096, 64 sparks: 8,599 -> 1,930 us.
//
// One persistent CTA per SM; a tile is 128 samples x 128 columns, the h1
// hidden units of V sparks side by side (every spark's columns are its own
// sums, so its fitness does not depend on which sparks share the tile).
// Warps 0-7 load X and W1 rows (16 bytes a lane, one block ahead), split them
// and store the parts in 64-byte swizzled shared-memory rows; warp 16 issues
// the MMAs; warps 8-15 add each block's accumulator into registers (64
// columns of one sample per thread), then run the rest of the network for the
// tile -- bias, activation, the remaining layers on the CUDA cores in
// k_fitness_simt's order, the loss -- while the other warps are already on
// the next tile.  What bounds it is the splitting (about 6 instructions per
// element, 2 x 4096 elements per 12 MMAs).
//
// An operand that is not finite (or rounds to a BF16 infinity) makes every
// sum it enters non-finite; each sum that is not finite, and no other, is
// computed again in FP32 in index order, so infinities and NaN end as they do
// in k_fitness_simt and do not reach a neighbour in the tile.
//
// Every wait is bounded; a CTA whose wait gives up sets a bit in the status
// word, if there is one, writes NaN sums for the tiles it has left and returns.
#include "mgfwa_internal.cuh"
#include "tc_ptx.cuh"

namespace mgfwa {
namespace {

using namespace tc;

constexpr int kM = 128, kN = 128;        // samples x columns of a tile
constexpr int kKB = 32;                  // inputs per block
constexpr int kConvWarps = 8, kEpiWarps = 8;
constexpr int kThreads = 32 * (kConvWarps + kEpiWarps + 1);
constexpr int kParts = 3;
constexpr uint32_t kPartBytes = kM * kKB * 2;          // one BF16 part tile, 64-byte rows
constexpr uint32_t kStageBytes = 2 * kParts * kPartBytes;  // X parts, then W1 parts
constexpr int kMaxStages = 3;
constexpr int kAcc = 4;                  // TMEM accumulators of kN columns
constexpr int kMaxV = 8;                 // sparks per tile
constexpr uint32_t kTmemCols = kAcc * kN;
// What the tensor core's truncation takes from a block's sum on average,
// relative to it: half a unit in the last place, 2^-24 of a power of two, over
// mantissas m spread as 1/m, 2^-24 / (2 ln 2).  The epilogue gives it back
// with the bias, so that the sums' error is as unbiased as a chain of rounded
// FMAs' (mean relative error of the ReLU networks' losses without it -4.4e-8,
// with every d_in from 32 to 3072).  A sum whose last kExactBits bits are zero
// is taken as exact and left alone: of numbers that FP32 holds with so many
// bits to spare (binary or one-hot inputs and coarse weights, say) nothing was
// lost, and of sums that were rounded one in 2^kExactBits looks so, which the
// others make up for.  Over 40 drawn networks and batches the geometric mean of
// the fitness' rms error against 64 bits is 6.6e-8, k_fitness_simt's 9.1e-8.
constexpr int kExactBits = 4;
constexpr uint32_t kLastBits = (1u << kExactBits) - 1u;
constexpr float kTrunc = 0.7213475f * 0x1p-24f * (float)(kLastBits + 1u) / (float)kLastBits;

struct Bars {
  uint64_t full[kMaxStages], empty[kMaxStages];  // a stage's parts are stored; its MMAs have read them
  uint64_t acc_full[kAcc], acc_empty[kAcc];      // an accumulator holds a block's sums; they have been read
  uint64_t done;
  uint32_t tmem_base;
  volatile int abort_flag;
  uint64_t wait_budget;   // clock64 ticks before a wait gives up
  float red[kMaxV][kM / 32];
};

struct X3Args {
  Mlp mlp;
  const float* rows;
  int64_t ld;
  int32_t count, mtiles, tiles;  // tiles = mtiles * ceil(count / V), sample tile fastest
  int32_t V, stages;
  float* partial;                // [mtiles][count]
  uint32_t* status;              // null: not reported
  uint64_t wait_budget;          // clock64 ticks before a wait gives up
};

__device__ __forceinline__ float act_f(int a, float v) { return a == kActTanh ? tanhf(v) : fmaxf(v, 0.0f); }

__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);  // start address
  d |= (uint64_t)1 << 16;                   // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(512 >> 4) << 32;          // stride byte offset: 8 rows x 64 B
  d |= (uint64_t)1 << 46;                   // descriptor version for tcgen05
  d |= (uint64_t)4 << 61;                   // 64-byte swizzle
  return d;
}

// A bounded wait (its limit read from shared memory, and only while it waits, so that it holds no registers).
__device__ __forceinline__ bool wait(Bars* sb, uint64_t* bar, uint32_t parity, uint32_t* status, uint32_t code) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (sb->abort_flag) return false;
    if ((uint64_t)(clock64() - t0) > sb->wait_budget) {
      sb->abort_flag = 1;
      if (status != nullptr) atomicOr(status, code);
      return false;
    }
  }
  return true;
}
// The wait for every issued MMA before the CTA leaves (ignores the abort flag).
__device__ __forceinline__ void drain(uint64_t* bar, uint32_t* status) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, 0u)) {
    if ((uint64_t)(clock64() - t0) > kWaitBudget) {
      if (status != nullptr) atomicOr(status, 16u);
      return;
    }
  }
}
// A whole warp's wait: every lane leaves with the same answer.
__device__ __forceinline__ bool warp_wait(Bars* sb, uint64_t* bar, uint32_t parity, uint32_t* status, uint32_t code) {
  return __all_sync(0xffffffffu, wait(sb, bar, parity, status, code));
}

// Four consecutive inputs -> their three BF16 parts, 8 bytes each.
__device__ __forceinline__ void split4(const float4& x, uint2* p) {
  float v[4] = {x.x, x.y, x.z, x.w};
  uint32_t w[kParts][2];
#pragma unroll
  for (int q = 0; q < kParts; ++q) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      // {low half: v[2 i], high half: v[2 i + 1]}, round to nearest
      asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[q][i]) : "f"(v[2 * i + 1]), "f"(v[2 * i]));
      if (q + 1 < kParts) {
        v[2 * i] = __fsub_rn(v[2 * i], __uint_as_float(w[q][i] << 16));
        v[2 * i + 1] = __fsub_rn(v[2 * i + 1], __uint_as_float(w[q][i] & 0xffff0000u));
      }
    }
    p[q] = make_uint2(w[q][0], w[q][1]);
  }
}

// a += b, two FP32 additions in one instruction.
__device__ __forceinline__ void add2(float& a0, float& a1, float b0, float b1) {
  asm("{\n\t.reg .b64 a, b;\n\t"
      "mov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\t"
      "add.rn.f32x2 a, a, b;\n\t"
      "mov.b64 {%0, %1}, a;\n\t}"
      : "+f"(a0), "+f"(a1)
      : "f"(b0), "f"(b1));
}

// R consecutive samples of a hidden unit.
template <int R>
__device__ __forceinline__ void load_r(const float* p, float* v) {
  static_assert(R == 1 || R == 4, "vector width");
  if constexpr (R == 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
  } else {
    v[0] = *p;
  }
}

// z[u][r] += sum over i of W[u][i] * in[i][sample r] in index order, U outputs
// of R samples at a time, everything in shared memory; W rows wld apart, `in`
// columns kM floats apart.  V4: W rows start on 16 bytes and fi is a multiple
// of 4.  Outputs from `live` on repeat the last one (no branches in the loop).
template <int U, int R, bool V4>
__device__ __forceinline__ void dense(const float* W, int wld, int fi, int live, const float* in, float (*z)[R]) {
  constexpr int kStep = V4 ? 4 : 1, kUnroll = R == 1 ? 2 : 1;
#pragma unroll kUnroll
  for (int i = 0; i < fi; i += kStep) {
    float a[kStep][R];
#pragma unroll
    for (int k = 0; k < kStep; ++k) load_r<R>(in + (i + k) * kM, a[k]);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float* wp = W + min(u, live - 1) * wld + i;
      float w[kStep];
      if constexpr (V4) {
        const float4 x = *reinterpret_cast<const float4*>(wp);
        w[0] = x.x, w[1] = x.y, w[2] = x.z, w[3] = x.w;
      } else {
        w[0] = wp[0];
      }
#pragma unroll
      for (int k = 0; k < kStep; ++k)
#pragma unroll
        for (int r = 0; r < R; ++r) z[u][r] = fmaf(w[k], a[k][r], z[u][r]);
    }
  }
}

// Floats of a spark row from its first bias to its end, rounded up to 4 (the
// row's stride is a multiple of 4 and b1 starts on one, so they can be read).
__host__ __device__ __forceinline__ int tail_ld(const Mlp& mlp) {
  const int L = mlp.n_layers;
  return ((int)(mlp.b_off[L - 1] + mlp.widths[L] - mlp.b_off[0]) + 3) / 4 * 4;
}

// Three layers: the second hidden layer of the tile's sparks, one item of 8
// units of a spark per warp, four samples per lane; the results replace the
// first layer's activations once every warp has read those.  Not inlined: its
// registers would push the accumulators of the caller's loop out to memory.
__noinline__ __device__ void middle_layer(const Mlp& mlp, const float* P, float* H, int V, int ew, int lane, bool v4) {
  const int h1 = mlp.widths[1], h2 = mlp.widths[2], Tp = tail_ld(mlp);
  const int ub = (h2 + 7) / 8;
  const int w2 = (int)(mlp.w_off[1] - mlp.b_off[0]), b2 = (int)(mlp.b_off[1] - mlp.b_off[0]);
  const bool on = ew < V * ub;
  const int v = on ? ew / ub : 0, u0 = on ? (ew - v * ub) * 8 : 0;
  const int live = h2 - u0;
  float z[8][4];
  if (on) {
    const float* w = P + v * Tp;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float b = w[b2 + u0 + min(u, live - 1)];
#pragma unroll
      for (int r = 0; r < 4; ++r) z[u][r] = b;
    }
    const float* in = H + v * h1 * kM + 4 * lane;
    if (v4)
      dense<8, 4, true>(w + w2 + u0 * h1, h1, h1, live, in, z);
    else
      dense<8, 4, false>(w + w2 + u0 * h1, h1, h1, live, in, z);
  }
  epi_bar<kEpiWarps>();
  if (on) {
    float* o = H + (v * h2 + u0) * kM + 4 * lane;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (u < live)
        *reinterpret_cast<float4*>(o + u * kM) = make_float4(act_f(mlp.acts[1], z[u][0]), act_f(mlp.acts[1], z[u][1]),
                                                             act_f(mlp.acts[1], z[u][2]), act_f(mlp.acts[1], z[u][3]));
  }
  epi_bar<kEpiWarps>();
}

// NL: register slots for the logits (C <= NL); kThree: three layers.
template <int NL, bool kThree>
__global__ void __launch_bounds__(kThreads, 1) k_fitness_x3(const __grid_constant__ X3Args a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const Mlp& mlp = a.mlp;
  const int S = a.stages, V = a.V;
  float* H = reinterpret_cast<float*>(base + (size_t)S * kStageBytes);  // [column][sample] activations of layer 1
  float* P = H + kN * kM;  // the tile's parameters from b1 on, [V][tail_ld(mlp)]
  constexpr int L = kThree ? 3 : 2;
  const int h1 = mlp.widths[1], h2 = L == 3 ? mlp.widths[2] : 0, d_in = mlp.widths[0];
  const int Tp = tail_ld(mlp);
  Bars* sb = reinterpret_cast<Bars*>(P + (size_t)V * Tp);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkb = (d_in + kKB - 1) / kKB;
  constexpr int kMmaWarp = kConvWarps + kEpiWarps;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&sb->full[s], kConvWarps);
      mbar_init(&sb->empty[s], 1);
    }
    for (int b = 0; b < kAcc; ++b) {
      mbar_init(&sb->acc_full[b], 1);
      mbar_init(&sb->acc_empty[b], kEpiWarps);
    }
    mbar_init(&sb->done, 1);
    sb->abort_flag = 0;
    sb->wait_budget = a.wait_budget;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sb->tmem_base)),
                 "n"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sb->tmem_base;
  griddep_wait();
  griddep_launch_dependents();

  auto row_ptr = [&](int spark) { return a.rows + (int64_t)spark * a.ld; };

  if (warp < kConvWarps) {
    // ---- load and split: this thread takes inputs 4 c .. 4 c + 3 of a block (a row's 32 inputs are one 128-byte
    // line, eight lanes), of rows r0 + 32 i of X and of W1, 16 bytes a load
    constexpr int kRowsX = kM / 32, kTasks = kRowsX + kN / 32;
    const int c = threadIdx.x & 7, r0 = threadIdx.x >> 3;
    // 64-byte swizzle of the 16-byte chunk c / 2 (the same for r0 + 32 i)
    const uint32_t off = (uint32_t)(r0 * 64 + (((c >> 1) ^ ((r0 >> 1) & 3)) << 4) + (c & 1) * 8);
    uint32_t s = 0, ph = 1;  // stage and the parity of its "empty"
    bool dead = false;
    for (int t = blockIdx.x; t < a.tiles && !dead; t += gridDim.x) {
      const int mt = t % a.mtiles, g0 = t / a.mtiles * V;
      // rows r0 + 32 i of X, columns r0 + 32 i; where there is none, the last one: its sums are not used
      const float* src[kTasks];
#pragma unroll
      for (int i = 0; i < kRowsX; ++i) {
        const int64_t n = (int64_t)mt * kM + r0 + 32 * i;
        src[i] = mlp.X + (n < mlp.N ? n : mlp.N - 1) * d_in;
      }
      const int live = min(V, a.count - g0) * h1;
#pragma unroll
      for (int i = 0; i < kN / 32; ++i) {
        const int col = min(r0 + 32 * i, live - 1), v = col / h1;
        src[kRowsX + i] = row_ptr(g0 + v) + (int64_t)(col - v * h1) * d_in;
      }
      float4 x[kTasks];
      auto load = [&](int i, int kb) {  // inputs past d_in: some others, zeroed before they are split
        x[i] = __ldg(reinterpret_cast<const float4*>(src[i] + min(kb * kKB + 4 * c, d_in - 4)));
      };
#pragma unroll
      for (int i = 0; i < kTasks; ++i) load(i, 0);
      for (int kb = 0; kb < nkb; ++kb) {
        if (!warp_wait(sb, &sb->empty[s], ph, a.status, 1u)) {
          dead = true;
          break;
        }
        if ((kb + 1) * kKB > d_in && kb * kKB + 4 * c >= d_in) {
#pragma unroll
          for (int i = 0; i < kTasks; ++i) x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const int next = min(kb + 1, nkb - 1);
        uint8_t* st = base + (size_t)s * kStageBytes + off;
#pragma unroll
        for (int i = 0; i < kTasks; ++i) {
          uint2 p[kParts];
          split4(x[i], p);
          uint8_t* d = st + (i < kRowsX ? i * 32 * 64 : kParts * kPartBytes + (i - kRowsX) * 32 * 64);
#pragma unroll
          for (int q = 0; q < kParts; ++q) *reinterpret_cast<uint2*>(d + q * kPartBytes) = p[q];
          load(i, next);  // in flight until the next block's turn of this register
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&sb->full[s]);
        if (++s == (uint32_t)S) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
  } else if (warp == kMmaWarp) {
    if (lane == 0) {
      const uint32_t idesc = instr_desc(kM, kN, 1u);
      uint32_t s = 0, ph = 0, b = 0, aph = 1;
      bool dead = false;
      for (int t = blockIdx.x; t < a.tiles && !dead; t += gridDim.x) {
        for (int kb = 0; kb < nkb; ++kb) {
          if (!wait(sb, &sb->full[s], ph, a.status, 2u) ||
              !wait(sb, &sb->acc_empty[b], aph, a.status, 4u)) {
            dead = true;
            break;
          }
          tc_fence_after();
          const uint32_t x1 = smem_u32(base + (size_t)s * kStageBytes);
          const uint32_t w1 = x1 + kParts * kPartBytes, d = tmem + b * (uint32_t)kN;
          auto mma = [&](int px, int pw, int j, uint32_t accum) {
            mma_bf16(d, smem_desc_sw64(x1 + (uint32_t)px * kPartBytes + (uint32_t)j * 32u),
                     smem_desc_sw64(w1 + (uint32_t)pw * kPartBytes + (uint32_t)j * 32u), idesc, accum);
          };
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            mma(2, 0, j, (uint32_t)j);
            mma(0, 2, j, 1u);
            mma(1, 1, j, 1u);
            mma(1, 0, j, 1u);
            mma(0, 1, j, 1u);
          }
          mma(0, 0, 0, 1u);
          mma(0, 0, 1, 1u);
          mma_commit(&sb->empty[s]);
          mma_commit(&sb->acc_full[b]);
          if (++s == (uint32_t)S) {
            s = 0;
            ph ^= 1u;
          }
          if (++b == kAcc) {
            b = 0;
            aph ^= 1u;
          }
        }
      }
      mma_commit(&sb->done);  // after every issued MMA
      drain(&sb->done, a.status);
    }
  } else {
    const int ew = warp - kConvWarps, q = warp & 3, half = ew >> 2;
    const int rrow = q * 32 + lane;  // this thread's sample of the tile = its TMEM lane
    const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * (kN / 2));
    const int et = threadIdx.x - 32 * kConvWarps;
    const int C = mlp.widths[L];
    const bool v4 = h1 % 4 == 0 && h2 % 4 == 0;  // then every later layer's weight rows start on 16 bytes
    uint32_t b = 0, ph = 0;
    int t = blockIdx.x;
    for (; t < a.tiles; t += gridDim.x) {
      const int mt = t % a.mtiles, g0 = t / a.mtiles * V;
      // the tile's later parameters, staged while its first blocks are split (the last tile's have been read)
      for (int e = et; e < V * (Tp / 4); e += 32 * kEpiWarps) {
        const int v = e / (Tp / 4), j = (e - v * (Tp / 4)) * 4;
        if (g0 + v < a.count)
          *reinterpret_cast<float4*>(P + v * Tp + j) =
              __ldg(reinterpret_cast<const float4*>(row_ptr(g0 + v) + mlp.b_off[0] + j));
      }
      // the label of this thread's sample of the loss (an item's 32 samples are those of ew & 3), -1 past the batch
      const int64_t ns = (int64_t)mt * kM + (ew & 3) * 32 + lane;
      const int yn = ns < mlp.N ? __ldg(mlp.y + ns) : -1;
      float acc[kN / 2];
#pragma unroll
      for (int i = 0; i < kN / 2; ++i) acc[i] = 0.0f;
      bool dead = false;
      for (int kb = 0; kb < nkb; ++kb) {
        if (!warp_wait(sb, &sb->acc_full[b], ph, a.status, 8u)) {
          dead = true;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int j0 = 0; j0 < kN / 2; j0 += 16) {
          float x[16];
          tmem_ld16(lanes + b * (uint32_t)kN + (uint32_t)j0, x);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; i += 2) add2(acc[j0 + i], acc[j0 + i + 1], x[i], x[i + 1]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sb->acc_empty[b]);
        if (++b == kAcc) {
          b = 0;
          ph ^= 1u;
        }
      }
      // also: the parameters are staged
      if (epi_bar_any<kEpiWarps>(dead)) break;
      const int64_t n = (int64_t)mt * kM + rrow;
      const int v0 = half * (kN / 2) / h1, j0 = half * (kN / 2) - v0 * h1;
      float* h = H + half * (kN / 2) * kM + rrow;
      uint64_t redo = 0;  // bit i: column i of this thread's half is not finite
      float nan_if_bad = 0.0f;  // 0 z, added up: not zero if a sum is not finite
#pragma unroll
      for (int i = 0; i < kN / 2; ++i) nan_if_bad = fmaf(acc[i], 0.0f, nan_if_bad);
      if (!(nan_if_bad == 0.0f) && n < mlp.N) {
#pragma unroll
        for (int i = 0; i < kN / 2; ++i)
          if (!(acc[i] * 0.0f == 0.0f)) redo |= uint64_t(1) << i;
      }
      auto activate = [&](auto act) {
        int j = j0, v = v0;
#pragma unroll
        for (int i0 = 0; i0 < kN / 2; i0 += 8) {
          float b1[8];  // loaded before any store, so that their latencies overlap
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            b1[i] = P[min(v, V - 1) * Tp + j];  // past the last spark: some bias, the column is not used
            const bool wrap = ++j == h1;
            j = wrap ? 0 : j;
            v += wrap ? 1 : 0;
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float z = acc[i0 + i];
            h[(i0 + i) * kM] = act(z + ((__float_as_uint(z) & kLastBits) != 0 ? fmaf(z, kTrunc, b1[i]) : b1[i]));
          }
        }
      };
      if (mlp.acts[0] == kActTanh)
        activate([](float z) { return tanhf(z); });
      else
        activate([](float z) { return fmaxf(z, 0.0f); });
      if (redo != 0) {
        // those columns of this sample again, in FP32 in index order; a NaN among the inputs needs no more looking,
        // and a sum that has become one stays it (784-64-10, N = 2048, 1,000 sparks, one input NaN in every sample:
        // 4.2 ms, all chains to their end 225, k_fitness_simt 6.0, finite inputs 1.6; an infinite input in every sample,
        // X read from L2 once a column, 150)
        const float* xr = mlp.X + n * d_in;
        float x_nan = 0.0f;
#pragma unroll 1
        for (int k = 0; k < d_in; k += 4) {
          const float4 x = __ldg(reinterpret_cast<const float4*>(xr + k));
#pragma unroll
          for (int u = 0; u < 4; ++u) x_nan = isnan(lane_of(x, u)) ? lane_of(x, u) : x_nan;
        }
        for (; redo != 0; redo &= redo - 1) {
          const int i = __ffsll((long long)redo) - 1, c = half * (kN / 2) + i, v = c / h1;
          if (v >= V || g0 + v >= a.count) break;  // past the last spark: not used
          const float* wr = row_ptr(g0 + v) + (int64_t)(c - v * h1) * d_in;
          float z = x_nan;
#pragma unroll 1
          for (int k = 0; k < d_in && !isnan(z); k += 4) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(xr + k));
            const float4 w = __ldg(reinterpret_cast<const float4*>(wr + k));
#pragma unroll
            for (int u = 0; u < 4; ++u) z = fmaf(lane_of(x, u), lane_of(w, u), z);
          }
          h[i * kM] = act_f(mlp.acts[0], z + P[v * Tp + c - v * h1]);
        }
      }
      epi_bar<kEpiWarps>();
      const int fl = mlp.widths[L - 1];  // last hidden width
      if constexpr (kThree) middle_layer(mlp, P, H, V, ew, lane, v4);
      // logits and loss: items (spark, 32 samples), a sample per lane
      for (int it = ew; it < V * 4; it += kEpiWarps) {
        const int sq = it & 3, v = it >> 2;
        if (g0 + v >= a.count) continue;
        const float* w = P + v * Tp - mlp.b_off[0];
        const float* in = H + v * fl * kM + sq * 32 + lane;
        float z[NL][1];
#pragma unroll
        for (int c = 0; c < NL; ++c) z[c][0] = w[mlp.b_off[L - 1] + min(c, C - 1)];
        if (v4)
          dense<NL, 1, true>(w + mlp.w_off[L - 1], fl, fl, C, in, z);
        else
          dense<NL, 1, false>(w + mlp.w_off[L - 1], fl, fl, C, in, z);
        float zmax = z[0][0];  // logits from C on repeat the last one
#pragma unroll
        for (int c = 1; c < NL; ++c) zmax = fmaxf(zmax, z[c][0]);
        float se = 0.0f, zy = z[0][0];
#pragma unroll
        for (int c = 0; c < NL; ++c) {
          const float e = expf(z[c][0] - zmax);
          se += c < C ? e : 0.0f;
          zy = c == yn ? z[c][0] : zy;
        }
        float ce = yn >= 0 ? (zmax + logf(se)) - zy : 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ce += __shfl_xor_sync(0xffffffffu, ce, o);
        if (lane == 0) sb->red[v][sq] = ce;
      }
      epi_bar<kEpiWarps>();
      if (et < V && g0 + et < a.count) {
        const float* r = sb->red[et];
        a.partial[(int64_t)mt * a.count + g0 + et] = ((r[0] + r[1]) + r[2]) + r[3];
      }
    }
    for (; t < a.tiles; t += gridDim.x) {  // gave up: the tiles left get no value
      const int mt = t % a.mtiles, g0 = t / a.mtiles * V;
      if (et < V && g0 + et < a.count) a.partial[(int64_t)mt * a.count + g0 + et] = __int_as_float(0x7fc00000);
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmemCols) : "memory");
  }
}

// Sparks per tile: their hidden columns side by side within kN (and, three
// layers, their second hidden layers within one item per warp).
int sparks_per_tile(const Mlp& mlp) {
  int v = kN / mlp.widths[1];
  if (mlp.n_layers == 3) {
    const int m = kEpiWarps / ((mlp.widths[2] + 7) / 8);  // one item of the middle layer per warp
    if (m < v) v = m;
  }
  return v < kMaxV ? v : kMaxV;
}

size_t smem_for(const Mlp& mlp, int V, int stages) {
  return 1024 + (size_t)stages * kStageBytes + sizeof(float) * ((size_t)kM * kN + (size_t)V * tail_ld(mlp)) +
         sizeof(Bars);
}

template <int NL, bool kThree>
cudaError_t go(const X3Args& a, dim3 grid, size_t smem, cudaStream_t s) {
  const cudaError_t e = ensure_smem_limit<k_fitness_x3<NL, kThree>>(smem);
  return e != cudaSuccess ? e : launch_pdl(k_fitness_x3<NL, kThree>, grid, dim3(kThreads), smem, s, a);
}

constexpr size_t kSmemLimit = 232448;  // 227 KB per block

}  // namespace

// The line between this kernel and k_fitness_simt.  It depends on the network
// and the batch only, never on how many sparks share the launch, so that a
// spark's fitness does not either.  Below a million first-layer products a
// spark (64-32-10, N = 300, 64 sparks: 19 us there, 22 us here) a launch is
// bound by its fixed latency, which is longer here; under 16 inputs or 8
// hidden units most of a block or a tile would be padding.  Above, the first
// layer is far faster here and the later layers are slower: one warp to a
// spark's 32 samples, a tile's spare columns idle, 25 classes and more in
// registers that spill.  So a tile's estimated times are compared: here the
// splitting or, where it is longer, the layers after it.  The estimates were
// fitted to 998 timed launches of 40 to 1,040 sparks (16 <= d_in <= 3072, 8 <=
// h1 <= 128, h2 <= 64, 2 to 32 classes; 5% off here, 9% there); of 3,587 such
// and smaller launches, us there / here: 784-64-10 (N = 84, 1,040 sparks) 420 /
// 120, 256-64-32 (512, 333) 182 / 157, 64-64-32 (2048, 333) 373 / 473,
// 16-8-64-32 (8192, 1,040) 7,232 / 16,761, 16-43-24-5 (3049, 1,040) 1,173 / 2,476.
constexpr int kMinInputs = 16, kMinHidden = 8;
constexpr int64_t kMinProducts = int64_t(1) << 20;

// Nanoseconds of a tile on one SM, V sparks to a tile.
int64_t tile_ns(const Mlp& mlp, int V) {
  const int L = mlp.n_layers, h1 = mlp.widths[1], h2 = L == 3 ? mlp.widths[2] : 0, C = mlp.widths[L];
  const bool v4 = h1 % 4 == 0 && h2 % 4 == 0;
  // a spark's logits, per input of the last layer: by the register slots, 16-byte weight reads or not
  const int slots = C <= 4 ? 0 : C <= 10 ? 1 : C <= 16 ? 2 : C <= 24 ? 3 : 4;
  constexpr int kLogit[2][5] = {{40, 77, 159, 302, 660}, {19, 46, 81, 141, 507}}, kSlots[5] = {4, 10, 16, 24, 32};
  const int64_t rounds10 = V > 1 ? 5 * V : 7;  // eight (spark, 32 samples) items to a round; four alone take 0.7
  int64_t tail = 4200 + (mlp.acts[0] == kActTanh ? 1100 : 0) +
                 rounds10 * (kLogit[v4][slots] * mlp.widths[L - 1] + 66 * kSlots[slots]) / 10;
  if (L == 3) {
    const int units = (h2 + 7) / 8 * V;
    tail += (C > 10 ? 7200 : 5000) + (int64_t)h1 * (v4 ? 15 + 20 * units : 54 + 62 * units);
  }
  const int64_t split = (int64_t)(mlp.widths[0] + kKB - 1) / kKB * 940;
  const int64_t after = tail + (split > 1100 ? split - 1100 : 0);  // the next tile's first block is split meanwhile
  return split > after ? split : after;
}

bool fitness_x3_ok(const Mlp& mlp) {
  if (mlp.widths[0] % 8 != 0 || mlp.widths[0] < kMinInputs || mlp.widths[1] < kMinHidden || mlp.widths[1] > kN ||
      mlp.w1_elems * mlp.N < kMinProducts || (mlp.n_layers == 3 && mlp.widths[2] > 8 * kEpiWarps))
    return false;
  const int V = sparks_per_tile(mlp);
  return smem_for(mlp, 1, kMaxStages - 1) <= kSmemLimit && 97 * tile_ns(mlp, V) <= 100 * V * fitness_simt_ns(mlp);
}

int launch_fitness_x3(const Mlp& mlp, const float* rows, int64_t ld, int32_t count, float* partial, uint32_t* status,
                      uint64_t wait_budget, cudaStream_t s) {
  if (count <= 0) return 0;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return -1;
  X3Args a;
  a.mlp = mlp;
  a.rows = rows;
  a.ld = ld;
  a.count = count;
  a.V = sparks_per_tile(mlp);
  // few sparks: fewer to a tile, so that the tiles reach more SMs
  const int64_t mtiles = (mlp.N + kM - 1) / kM;
  while (a.V > 1 && mtiles * ((count + a.V - 1) / a.V) * 2 <= sms) a.V = (a.V + 1) / 2;
  while (a.V > 1 && smem_for(mlp, a.V, kMaxStages - 1) > kSmemLimit) --a.V;
  a.mtiles = (int32_t)mtiles;
  const int64_t tiles = mtiles * ((count + a.V - 1) / a.V);
  if (tiles > INT32_MAX - 65536) return -1;
  a.tiles = (int32_t)tiles;
  a.stages = smem_for(mlp, a.V, kMaxStages) <= kSmemLimit ? kMaxStages : kMaxStages - 1;
  a.partial = partial;
  a.status = status;
  // a tile whose sums all end in infinities is 64 chains of d_in steps, each a read from L2, while the other warps wait
  a.wait_budget = wait_budget != 0 ? wait_budget : kWaitBudget + ((uint64_t)mlp.widths[0] << 15);
  const size_t smem = smem_for(mlp, a.V, a.stages);
  const dim3 grid((unsigned)(tiles < sms ? tiles : sms));
  cudaError_t e;
#define MG_X3(NL) e = mlp.n_layers == 3 ? go<NL, true>(a, grid, smem, s) : go<NL, false>(a, grid, smem, s)
  const int C = mlp.widths[mlp.n_layers];
  if (C <= 4)
    MG_X3(4);
  else if (C <= 10)
    MG_X3(10);
  else if (C <= 16)
    MG_X3(16);
  else if (C <= 24)
    MG_X3(24);
  else
    MG_X3(32);
#undef MG_X3
  return e == cudaSuccess ? 1 : -1;
}

}  // namespace mgfwa

// Learned warm start for the level-1 local eigenproblems (Eq. (spepb)): a
// multilayer perceptron maps an element's standardised log-permeability patch
// to guesses for its eigenvectors 1 .. L-1 in the symmetric form
// y = S^{1/2} phi (eigenvector 0, the constant, is known exactly).  The guesses
// seed the subspace iteration, which still runs to the same eigen-residual
// tolerance, so the preconditioner is unchanged; only the set-up time moves.
//
// Network: x (n_in) -> relu(x W1 + b1) (h1) -> relu(. W2 + b2) (h2) -> o = . W3 + b3
// (n_vec * n_in) -> y_k = w * o_k.  The fixed output weighting
// w_c = sqrt(S_c / sum S), recovered from the input (S_c is proportional to
// exp(8 x_c)), makes the network predict the eigenvectors phi, which vary
// slowly across permeability jumps, while its output y = S^{1/2} phi stays in
// the symmetric form.  Weights are kept as FP32 masters (training, Adam) and
// BF16 copies that every product reads; activations and accumulation are FP32.
//
// Loss per sample and output vector k (sign-invariant: an eigenvector is only
// defined up to sign):  l = ||p||^2 + ||t||^2 - 2 |p . t|,  the smaller of
// ||p - t||^2 and ||p + t||^2;  the batch loss is the mean over samples and
// vectors.
//
// All kernels are deterministic (no atomics): a training run is reproducible.
#include "msmg_internal.cuh"
#include <cuda.h>
#include <cuda_bf16.h>
#include <new>

struct msmg_net {
  msmg_net_desc d;
  int n_out;                    // n_vec * n_in
  int64_t n_param;              // total parameters
  // parameter blocks inside one array: W1 [n_in][h1], b1, W2 [h1][h2], b2, W3 [h2][n_out], b3
  int64_t off_w[3], off_b[3];
  float* w32;                   // FP32 masters
  __nv_bfloat16* w16;           // BF16 copies (read by the products)
  float* grad;                  // gradients, same layout
  float* adam_m;
  float* adam_v;
  float* out;                   // [batch_max][n_out]
  float* d_out;                 // [batch_max][n_out]
  float* wgt;                   // [batch_max][n_in] output weighting of the current batch
  float* loss;                  // [batch_max * n_vec + 32]
  int64_t step;
  // tensor-core forward (tcgen05): layer widths multiples of 64
  bool tc;
  __nv_bfloat16* wt16;          // BF16 weights transposed, W_l^T [fan_out][fan_in], same offsets
  __nv_bfloat16* xb;            // [batch_max][n_in] BF16 input (the products' A operand)
  __nv_bfloat16* h1b;           // [batch_max][h1] BF16 activations
  __nv_bfloat16* h2b;           // [batch_max][h2]
  // backward (chunks of at most rc rows; rcp: rc rounded up to 64)
  int rc;
  __nv_bfloat16* dk;            // [3][rc][ldk] BF16 parts of a layer's output gradient
  __nv_bfloat16* dt;            // [3][fan_out][rcp] the same transposed, zero beyond the rows
  __nv_bfloat16* at[3];         // [fan_in][rcp] transposed BF16 input of each layer, zero beyond the rows
  __nv_bfloat16* wp[3];         // BF16 weights with 16-byte row strides (w16 itself where fan_out % 8 == 0); [0] unused
  int ldw[3];                   // their row strides
  float* part;                  // partial sums of the split products
  int64_t part_cap;
  float* csum[3];               // [rcp / 64][fan_out] column sums of 64 rows, per layer
  int* err;                     // device error word: a bounded tensor-core wait gave up
  int map_err;                  // host: a tensor map of the tensor-core products could not be encoded
  // tensor maps of the network's own buffers, encoded again when the row count changes
  CUtensorMap fmap[3][2], gmap[3][4];   // forward A, Bt; backward: parts, weights; act^T, parts^T
  int fmap_rows, gmap_rows;             // 0: not encoded
};

namespace msmg {

// ------------------------------------------------------------------ CUDA-core product
// C = epi(A[M][K] B[K][N] + bias), BF16 operands, FP32 accumulation, for the forward
// pass of networks whose widths are not multiples of 64.  Each output is one chain of
// fmaf over k = 0 .. K-1, whatever the tile.  256 threads, TM x TN outputs each; the next K
// block is in registers while this one is multiplied.
//   EPI 2: ReLU, stored in BF16 (the next layer's operand); EPI 3: times wgt[m][n mod n_in], FP32.
template <int BM, int BN, int BK, int TM, int TN, int EPI>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
    k_gemm(const __nv_bfloat16* __restrict__ A, const __nv_bfloat16* __restrict__ B, float* __restrict__ C,
           __nv_bfloat16* __restrict__ Cb, const float* __restrict__ bias, const float* __restrict__ wgt, int n_in,
           int M, int N, int K) {
  constexpr int NT = (BM / TM) * (BN / TN), LA = BM * BK / NT, LB = BN * BK / NT;
  __shared__ __align__(16) float As[BK][BM + 4];
  __shared__ __align__(16) float Bs[BK][BN + 4];
  const int tid = threadIdx.x, tx = tid % (BN / TN), ty = tid / (BN / TN);
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const __nv_bfloat16 zero = __float2bfloat16(0.f);
  __nv_bfloat16 ra[LA], rb[LB];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < LA; ++q) {
      const int idx = tid + NT * q, kk = idx % BK, mm = idx / BK;
      ra[q] = (m0 + mm < M && k0 + kk < K) ? A[(int64_t)(m0 + mm) * K + k0 + kk] : zero;
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) {
      const int idx = tid + NT * q, nn = idx % BN, kk = idx / BN;
      rb[q] = (n0 + nn < N && k0 + kk < K) ? B[(int64_t)(k0 + kk) * N + n0 + nn] : zero;
    }
  };
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  load(0);
  for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
    for (int q = 0; q < LA; ++q) {
      const int idx = tid + NT * q;
      As[idx % BK][idx / BK] = __bfloat162float(ra[q]);
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) {
      const int idx = tid + NT * q;
      Bs[idx / BN][idx % BN] = __bfloat162float(rb[q]);
    }
    __syncthreads();
    if (k0 + BK < K) load(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][ty * TM + i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx * TN + j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int gm = m0 + ty * TM + i;
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int gn = n0 + tx * TN + j;
      if (gn >= N) continue;
      float v = acc[i][j] + bias[gn];
      if (EPI == 2) Cb[(int64_t)gm * N + gn] = __float2bfloat16(v > 0.f ? v : 0.f);
      else C[(int64_t)gm * N + gn] = v * wgt[(int64_t)gm * n_in + gn % n_in];
    }
  }
}

static int sm_count();
// 64 x 64 tiles where every SM gets one, 32 x 32 below that (512 -> 1000 -> 1000 -> 2560,
// 50 rows 193 -> 122 us, 300 rows 215 against 230).  128 x 128 tiles gain at most 5% where
// their number happens to fill the SMs evenly and lose up to 27% where it does not (64 / 128,
// us: 3000 rows of 216 -> 450 -> 900 -> 864 352 / 449, of 512 -> 1000 -> 1000 -> 2560
// 835 / 968, 8192 rows of it 2108 / 2089), so there are none.
template <int EPI>
static void gemm(const __nv_bfloat16* A, const __nv_bfloat16* B, float* C, __nv_bfloat16* Cb, const float* bias,
                 const float* wgt, int n_in, int M, int N, int K, cudaStream_t s) {
  auto tiles = [&](int bm, int bn) { return (int64_t)((M + bm - 1) / bm) * ((N + bn - 1) / bn); };
  if (tiles(64, 64) >= sm_count())
    k_gemm<64, 64, 32, 4, 4, EPI><<<dim3((N + 63) / 64, (M + 63) / 64), 256, 0, s>>>(A, B, C, Cb, bias, wgt, n_in, M, N, K);
  else
    k_gemm<32, 32, 32, 2, 2, EPI><<<dim3((N + 31) / 32, (M + 31) / 32), 256, 0, s>>>(A, B, C, Cb, bias, wgt, n_in, M, N, K);
}

// ------------------------------------------------------------------ tensor-core GEMM (tcgen05)
// The forward products: C[M][N] = epi(A[M][K] . Bt[N][K]^T), A and Bt BF16 with K
// contiguous, FP32 accumulation in tensor memory (TMEM).  Persistent: one CTA per SM
// takes the 128 x BN output tiles t = blockIdx.x, blockIdx.x + gridDim.x, ... (N-tiles
// fastest, so consecutive tiles share their A rows in L2), with six warps in three roles:
//   warp 0, one thread: TMA (cp.async.bulk.tensor.2d) of the A and Bt blocks
//     (K in blocks of 64, 128-byte swizzle) into a ring of shared-memory stages,
//     completion counted in bytes on the stage's "full" mbarrier; a stage is
//     refilled once its "empty" mbarrier has fired;
//   warp 1, one thread: the four 128 x BN x 16 MMAs of each block (shared-memory
//     descriptors, K-major, 128-byte swizzle: 8-row groups 1024 bytes apart, the
//     16-wide K steps 32 bytes apart inside the swizzle atom), tcgen05.commit to
//     the stage's "empty" barrier, and after a tile's last block a commit to the
//     "accumulator full" barrier of the tile's TMEM buffer (two buffers of BN
//     columns, so the next tile accumulates while this one is written out);
//   warps 2-5: the epilogue (warp w reads TMEM lanes 32 (w mod 4) .. + 31, the
//     tile's rows): 64-column chunks by tcgen05.ld into a padded shared-memory
//     slice, the buffer released ("accumulator empty") once read, then bias, ReLU,
//     FP32 store and, when asked, a BF16 copy (the next layer's A operand), each
//     store writing whole row segments.
// Rows of A beyond M and of Bt beyond N read as zeros (TMA bounds).  Every wait
// is bounded: on timeout the error word is set, the loops stop, what was issued
// is drained with bounded waits, and the TMEM is freed before the CTA returns.
// The operands' row strides are multiples of 8 elements and their bases 16-byte
// aligned (the tensor maps' rules); columns beyond K read as zeros in both.
constexpr int kTcM = 128, kTcK = 64, kTcThreads = 192, kTcChunk = 64;
template <int BN>
__host__ __device__ constexpr int tc_stages() { return BN == 256 ? 3 : (BN == 128 ? 4 : 6); }
template <int BN>
__host__ __device__ constexpr size_t tc_stage_bytes() { return (size_t)(kTcM + BN) * kTcK * 2; }
constexpr size_t kTcEpiBytes = (size_t)4 * 32 * (kTcChunk + 4) * 4;   // four warps' padded 32 x 64 slices
template <int BN>
__host__ __device__ constexpr size_t tc_smem_bytes() {
  return tc_stages<BN>() * tc_stage_bytes<BN>() + kTcEpiBytes + 1024;
}

// shared-memory matrix descriptor, K-major with 128-byte swizzle: start address,
// leading offset unused (1), stride between 8-row groups 1024 bytes, descriptor
// version 1, layout type 2 (128-byte swizzle)
__device__ __forceinline__ uint64_t tc_desc_sw128(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
// instruction descriptor of kind::f16: F32 accumulator, BF16 A and B, both K-major, M x N
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void tc_mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ bool tc_mbar_wait(uint32_t bar, uint32_t parity) {
  for (int it = 0; it < (1 << 24); ++it) {
    uint32_t done;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(done)
                 : "r"(bar), "r"(parity)
                 : "memory");
    if (done) return true;
  }
  return false;
}
__device__ __forceinline__ void tc_tma_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}

// a load that stays where it is written, from L2 (the read-only path through what 227 KB of
// shared memory leave of L1 took the largest product of 8192 rows from 49 to 166 us)
__device__ __forceinline__ float4 tc_ldg4(const float* p) {
  float4 v;
  asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}

struct TcArgs {
  float* C;                    // FP32 output (EPI 1), row stride N
  __nv_bfloat16* Cb;           // BF16 output (EPI 2), row stride N
  const float* bias;
  const float* wgt;            // EPI 1: output weighting [M][n_in]
  int n_in;
  int M, N, K;
  int* err;
};

// EPI 1: (sum + bias) * wgt[row][col mod n_in], FP32; 2: ReLU(sum + bias), BF16
template <int EPI, int BN>
__global__ void __launch_bounds__(kTcThreads, 1) k_gemm_tc(const __grid_constant__ CUtensorMap mapA,
                                                           const __grid_constant__ CUtensorMap mapB,
                                                           const __grid_constant__ TcArgs g_) {
  const int M = g_.M, N = g_.N;
  constexpr int S = tc_stages<BN>();
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  __shared__ __align__(8) unsigned long long full[S], empty[S], acc_full[2], acc_empty[2], done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_fail;
  constexpr uint32_t kStage = (uint32_t)tc_stage_bytes<BN>();
  constexpr uint32_t kBytesA = kTcM * kTcK * 2;
  constexpr uint32_t kCols = 2 * BN;                      // two accumulator buffers
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(tc_smem) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nk = g_.K / kTcK;
  const int ntn = N / BN, ntiles = ntn * ((M + kTcM - 1) / kTcM);
  const int mytiles = blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                 "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (threadIdx.x == 32) {
    for (int i = 0; i < S; ++i) {
      tc_mbar_init(smem_u32(&full[i]), 1);
      tc_mbar_init(smem_u32(&empty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc_mbar_init(smem_u32(&acc_full[i]), 1);
      tc_mbar_init(smem_u32(&acc_empty[i]), 4);   // one arrival per epilogue warp
    }
    tc_mbar_init(smem_u32(&done_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    s_fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = tmem_slot;
  if (threadIdx.x == 0) {
    // producer: global block counter g runs across the CTA's tiles
    int g = 0;
    bool stop = false;
    for (int i = 0; i < mytiles && !stop; ++i) {
      const int t = (int)blockIdx.x + i * (int)gridDim.x;
      const int m0 = (t / ntn) * kTcM, n0 = (t % ntn) * BN;
      for (int kb = 0; kb < nk; ++kb, ++g) {
        const int st = g % S, use = g / S;
        if ((use > 0 && !tc_mbar_wait(smem_u32(&empty[st]), (uint32_t)((use - 1) & 1))) ||
            *(volatile int*)&s_fail) {
          atomicExch(&s_fail, 1);
          stop = true;
          break;
        }
        const uint32_t sA = smem_u32(smem + st * kStage), sB = sA + kBytesA;
        const uint32_t fb = smem_u32(&full[st]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fb), "r"(kStage) : "memory");
        tc_tma_2d(sA, &mapA, kb * kTcK, m0, fb);
        tc_tma_2d(sB, &mapB, kb * kTcK, n0, fb);
      }
    }
    // a load issued but not consumed must land before the CTA may exit (the last
    // S loads are the last completions of their barriers)
    for (int j = g - S < 0 ? 0 : g - S; j < g; ++j) tc_mbar_wait(smem_u32(&full[j % S]), (uint32_t)((j / S) & 1));
  } else if (threadIdx.x == 32) {
    // MMA issuer
    constexpr uint32_t idesc = tc_idesc(kTcM, BN);
    int g = 0;
    bool stop = false;
    for (int i = 0; i < mytiles && !stop; ++i) {
      const int a = i & 1, use = i >> 1;
      if ((use > 0 && !tc_mbar_wait(smem_u32(&acc_empty[a]), (uint32_t)((use - 1) & 1))) || *(volatile int*)&s_fail) {
        atomicExch(&s_fail, 1);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const uint32_t acc_tm = tmem + (uint32_t)(a * BN);
      for (int kb = 0; kb < nk; ++kb, ++g) {
        const int st = g % S, su = g / S;
        if (!tc_mbar_wait(smem_u32(&full[st]), (uint32_t)(su & 1)) || *(volatile int*)&s_fail) {
          atomicExch(&s_fail, 1);
          stop = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint32_t sA = smem_u32(smem + st * kStage), sB = sA + kBytesA;
#pragma unroll
        for (int kk = 0; kk < kTcK / 16; ++kk) {
          const uint64_t da = tc_desc_sw128(sA + kk * 32), db = tc_desc_sw128(sB + kk * 32);
          const uint32_t accf = (kb > 0 || kk > 0) ? 1u : 0u;
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(acc_tm),
              "l"(da), "l"(db), "r"(idesc), "r"(accf));
        }
        tc_commit(smem_u32(&empty[st]));
      }
      if (!stop) tc_commit(smem_u32(&acc_full[a]));
    }
    tc_commit(smem_u32(&done_bar));   // covers every MMA this CTA issued
  } else if (warp >= 2) {
    // epilogue
    const int q = warp & 3;                                 // TMEM lane quarter = rows 32q .. 32q + 31
    float* sl = reinterpret_cast<float*>(smem + S * kStage) + (size_t)(warp - 2) * 32 * (kTcChunk + 4);
    for (int i = 0; i < mytiles; ++i) {
      const int t = (int)blockIdx.x + i * (int)gridDim.x;
      const int m0 = (t / ntn) * kTcM, n0 = (t % ntn) * BN;
      const int a = i & 1, use = i >> 1;
      bool ok = tc_mbar_wait(smem_u32(&acc_full[a]), (uint32_t)(use & 1));
      ok = __all_sync(0xffffffffu, ok && *(volatile int*)&s_fail == 0);
      if (!ok) {
        if (lane == 0) atomicExch(&s_fail, 1);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const uint32_t acc_tm = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(a * BN);
#pragma unroll 1
      for (int c0 = 0; c0 < BN; c0 += kTcChunk) {
        // lanes 0-15 row 2k, lanes 16-31 row 2k + 1, four columns each
        const int cl = (lane & 15) * 4;
        // the chunk's output weights (a chunk stays in one block of n_in columns), all
        // loads in flight while the accumulator is read
        float4 wv[EPI == 1 ? 16 : 1];
        if (EPI == 1) {
          const float* wrow = g_.wgt + (n0 + c0) % g_.n_in + cl;
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const int row = m0 + q * 32 + 2 * k + (lane >> 4);
            wv[EPI == 1 ? k : 0] = tc_ldg4(wrow + (int64_t)(row < M ? row : M - 1) * g_.n_in);
          }
        }
#pragma unroll
        for (int c1 = 0; c1 < kTcChunk; c1 += 16) {
          uint32_t v[16];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
              "%14, %15}, [%16];\n"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
              : "r"(acc_tm + (uint32_t)(c0 + c1)));
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
          float4* dst = reinterpret_cast<float4*>(sl + (size_t)lane * (kTcChunk + 4) + c1);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            dst[j] = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                 __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
        }
        if (c0 + kTcChunk >= BN) {
          // the whole accumulator of this tile has been read: release the buffer
          asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
          __syncwarp();
          if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&acc_empty[a])) : "memory");
        }
        __syncwarp();
        const float4 bb = __ldg(reinterpret_cast<const float4*>(g_.bias + n0 + c0 + cl));
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const int r = 2 * k + (lane >> 4);
          const int row = m0 + q * 32 + r;
          float4 v = *reinterpret_cast<const float4*>(sl + (size_t)r * (kTcChunk + 4) + cl);
          if (row < M) {
            v.x += bb.x; v.y += bb.y; v.z += bb.z; v.w += bb.w;
            const int64_t at = (int64_t)row * N + n0 + c0 + cl;
            if (EPI == 1) {
              const float4 w = wv[EPI == 1 ? k : 0];
              v.x *= w.x; v.y *= w.y; v.z *= w.z; v.w *= w.w;
              *reinterpret_cast<float4*>(g_.C + at) = v;
            } else {
              const __nv_bfloat162 h0 = __floats2bfloat162_rn(v.x > 0.f ? v.x : 0.f, v.y > 0.f ? v.y : 0.f),
                                   h1 = __floats2bfloat162_rn(v.z > 0.f ? v.z : 0.f, v.w > 0.f ? v.w : 0.f);
              uint2 w;
              w.x = *reinterpret_cast<const uint32_t*>(&h0);
              w.y = *reinterpret_cast<const uint32_t*>(&h1);
              *reinterpret_cast<uint2*>(g_.Cb + at) = w;
            }
          }
        }
        __syncwarp();   // the slice is rewritten by the next chunk
      }
    }
  }
  __syncwarp();
  __syncthreads();
  if (threadIdx.x == 0) {
    // every MMA complete before the TMEM is freed (at once unless a wait gave up)
    const bool d = tc_mbar_wait(smem_u32(&done_bar), 0u);
    if (s_fail || !d) atomicExch(g_.err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kCols));
  }
}

// ------------------------------------------------------------------ backward products
// C[M][N] (+)= A[M][K] . Bt[N][K]^T with one FP32 operand, held as three BF16 parts
// stacked in rows: v = hi + mid + lo keeps 24 bits, so its products with the other,
// BF16, operand are the FP32 value's.  NA = 3, NB = 1: A in parts (an input gradient,
// d W^T); NA = 1, NB = 3: Bt in parts (a weight gradient, act^T d).  A stage holds one
// K block of every part (64 KB, three stages), so the shared operand is read once for the
// three; the K blocks of a tile may be split over CTAs (each writes its own partial
// sum, added by the next k_split_grad).
// Precision: the tensor core cuts its FP32 accumulator at every MMA, always towards
// zero, which over a long K is worse than rounded FP32 chains (dW of 512 rows 1.9e-6
// off FP64 against 7e-7 with one accumulator).  So a K block's hi products go to two
// accumulators (two MMAs each), the small mid and lo products under one of them, and
// after every K block (kGrSeg = 1; four blocks: 9e-7) the epilogue warps add both to
// FP32 registers, rounded.
// Roles and bounded waits as in k_gemm_tc; 128 x 128 tiles, two pairs of 128-column
// accumulators (all 512 columns of the SM's TMEM).
constexpr int kGrN = 128, kGrStages = 3, kGrSeg = 1, kGrChunk = 32;
constexpr uint32_t kGrStageBytes = (uint32_t)(4 * 128) * kTcK * 2;
constexpr size_t kGrSmem = (size_t)kGrStages * kGrStageBytes + (size_t)4 * 32 * (kGrChunk + 4) * 4 + 1024;
struct GrArgs {
  float* C;                    // row stride ldc; split i at C + i * split_stride
  int64_t ldc, split_stride;
  int M, N, K;                 // K blocks reach beyond K (the tensor maps read zeros there)
  int rows_a, rows_b;          // rows of one part
  int splits;
  int accum;                   // add to C
  int vec;                     // 16-byte stores allowed: ldc, N and split_stride multiples of 4, C aligned
  int* err;
};

template <int NA, int NB>
__global__ void __launch_bounds__(kTcThreads, 1) k_gemm_grad(const __grid_constant__ CUtensorMap mapA,
                                                             const __grid_constant__ CUtensorMap mapB,
                                                             const __grid_constant__ GrArgs p) {
  static_assert(NA + NB == 4 && kTcM == 128 && kGrN == 128, "one operand in three parts, tiles of 128 x 128");
  constexpr int S = kGrStages;
  constexpr uint32_t kTile = 128 * kTcK * 2;
  constexpr uint32_t kCols = 4 * kGrN;
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  __shared__ __align__(8) unsigned long long full[S], empty[S], acc_full[2], acc_empty[2], done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_fail;
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(tc_smem) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int M = p.M, N = p.N;
  const int nkb = (p.K + kTcK - 1) / kTcK;
  const int ntn = (N + kGrN - 1) / kGrN, ntile1 = ntn * ((M + kTcM - 1) / kTcM), ntiles = ntile1 * p.splits;
  const int mytiles = (int)blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  auto tile = [&](int i, int* m0, int* n0, int* kb0, int* kb1) {
    const int t = (int)blockIdx.x + i * (int)gridDim.x, sp = t / ntile1, tt = t - sp * ntile1;
    *m0 = (tt / ntn) * kTcM;
    *n0 = (tt % ntn) * kGrN;
    *kb0 = (int)((int64_t)sp * nkb / p.splits);
    *kb1 = (int)((int64_t)(sp + 1) * nkb / p.splits);
    return sp;
  };
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                 "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (threadIdx.x == 32) {
    for (int i = 0; i < S; ++i) {
      tc_mbar_init(smem_u32(&full[i]), 1);
      tc_mbar_init(smem_u32(&empty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc_mbar_init(smem_u32(&acc_full[i]), 1);
      tc_mbar_init(smem_u32(&acc_empty[i]), 4);   // one arrival per epilogue warp
    }
    tc_mbar_init(smem_u32(&done_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    s_fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = tmem_slot;
  if (threadIdx.x == 0) {
    // producer: block counter g runs across the CTA's tiles
    int g = 0;
    bool stop = false;
    for (int i = 0; i < mytiles && !stop; ++i) {
      int m0, n0, kb0, kb1;
      tile(i, &m0, &n0, &kb0, &kb1);
      for (int kb = kb0; kb < kb1; ++kb, ++g) {
        const int st = g % S, use = g / S;
        if ((use > 0 && !tc_mbar_wait(smem_u32(&empty[st]), (uint32_t)((use - 1) & 1))) ||
            *(volatile int*)&s_fail) {
          atomicExch(&s_fail, 1);
          stop = true;
          break;
        }
        const uint32_t sA = smem_u32(smem + st * kGrStageBytes), sB = sA + NA * kTile;
        const uint32_t fb = smem_u32(&full[st]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fb), "r"(kGrStageBytes) : "memory");
#pragma unroll
        for (int k = 0; k < NA; ++k) tc_tma_2d(sA + k * kTile, &mapA, kb * kTcK, m0 + k * p.rows_a, fb);
#pragma unroll
        for (int k = 0; k < NB; ++k) tc_tma_2d(sB + k * kTile, &mapB, kb * kTcK, n0 + k * p.rows_b, fb);
      }
    }
    // a load issued but not consumed must land before the CTA may exit
    for (int j = g - S < 0 ? 0 : g - S; j < g; ++j) tc_mbar_wait(smem_u32(&full[j % S]), (uint32_t)((j / S) & 1));
  } else if (threadIdx.x == 32) {
    // MMA issuer: accumulator pair sg & 1 takes segment sg 
    constexpr uint32_t idesc = tc_idesc(kTcM, kGrN);
    int g = 0, sg = 0;
    bool stop = false;
    for (int i = 0; i < mytiles && !stop; ++i) {
      int m0, n0, kb0, kb1;
      tile(i, &m0, &n0, &kb0, &kb1);
      for (int k0 = kb0; k0 < kb1 && !stop; k0 += kGrSeg, ++sg) {
        const int a = sg & 1, use = sg >> 1;
        if ((use > 0 && !tc_mbar_wait(smem_u32(&acc_empty[a]), (uint32_t)((use - 1) & 1))) ||
            *(volatile int*)&s_fail) {
          atomicExch(&s_fail, 1);
          stop = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint32_t acc_hi = tmem + (uint32_t)(a * 2 * kGrN), acc_lo = acc_hi + kGrN;
        for (int kb = k0; kb < kb1 && kb < k0 + kGrSeg; ++kb, ++g) {
          const int st = g % S, su = g / S;
          if (!tc_mbar_wait(smem_u32(&full[st]), (uint32_t)(su & 1)) || *(volatile int*)&s_fail) {
            atomicExch(&s_fail, 1);
            stop = true;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          const uint32_t sA = smem_u32(smem + st * kGrStageBytes), sB = sA + NA * kTile;
#pragma unroll
          for (int pt = 2; pt >= 0; --pt)
#pragma unroll
            for (int kk = 0; kk < kTcK / 16; ++kk) {
              const uint64_t da = tc_desc_sw128(sA + (NA > 1 ? pt : 0) * kTile + kk * 32),
                             db = tc_desc_sw128(sB + (NB > 1 ? pt : 0) * kTile + kk * 32);
              // the lo and mid parts and half of hi in one accumulator, hi's other half in the other
              const bool first = pt == 0 && kk < 2;
              const uint32_t accf = (kb > k0 || kk > 0 || (pt == 1)) ? 1u : 0u;
              asm volatile(
                  "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                  " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(first ? acc_hi : acc_lo),
                  "l"(da), "l"(db), "r"(idesc), "r"(accf));
            }
          tc_commit(smem_u32(&empty[st]));
        }
        if (!stop) tc_commit(smem_u32(&acc_full[a]));
      }
    }
    tc_commit(smem_u32(&done_bar));   // covers every MMA this CTA issued
  } else if (warp >= 2) {
    // epilogue: thread = row; the tile's FP32 sums in registers over its segments
    const int q = warp & 3;
    float* sl = reinterpret_cast<float*>(smem + S * kGrStageBytes) + (size_t)(warp - 2) * 32 * (kGrChunk + 4);
    int sg = 0;
    bool ok = true;
    for (int i = 0; i < mytiles && ok; ++i) {
      int m0, n0, kb0, kb1;
      const int sp = tile(i, &m0, &n0, &kb0, &kb1);
      float acc[kGrN];
#pragma unroll
      for (int c = 0; c < kGrN; ++c) acc[c] = 0.f;
      for (int k0 = kb0; k0 < kb1; k0 += kGrSeg, ++sg) {
        const int a = sg & 1, use = sg >> 1;
        ok = tc_mbar_wait(smem_u32(&acc_full[a]), (uint32_t)(use & 1));
        ok = __all_sync(0xffffffffu, ok && *(volatile int*)&s_fail == 0);
        if (!ok) {
          if (lane == 0) atomicExch(&s_fail, 1);
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint32_t tm = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(a * 2 * kGrN);
#pragma unroll
        for (int c0 = 0; c0 < kGrN; c0 += 16) {
          uint32_t v[32];
#pragma unroll
          for (int h = 0; h < 2; ++h)
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                "%14, %15}, [%16];\n"
                : "=r"(v[16 * h + 0]), "=r"(v[16 * h + 1]), "=r"(v[16 * h + 2]), "=r"(v[16 * h + 3]),
                  "=r"(v[16 * h + 4]), "=r"(v[16 * h + 5]), "=r"(v[16 * h + 6]), "=r"(v[16 * h + 7]),
                  "=r"(v[16 * h + 8]), "=r"(v[16 * h + 9]), "=r"(v[16 * h + 10]), "=r"(v[16 * h + 11]),
                  "=r"(v[16 * h + 12]), "=r"(v[16 * h + 13]), "=r"(v[16 * h + 14]), "=r"(v[16 * h + 15])
                : "r"(tm + (uint32_t)(h * kGrN + c0)));
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
          for (int c = 0; c < 16; ++c) acc[c0 + c] += __uint_as_float(v[c]) + __uint_as_float(v[16 + c]);
        }
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&acc_empty[a])) : "memory");
      }
      if (!ok) break;
      float* const C = p.C + sp * p.split_stride;
#pragma unroll
      for (int c0 = 0; c0 < kGrN; c0 += kGrChunk) {
        float4* dst = reinterpret_cast<float4*>(sl + (size_t)lane * (kGrChunk + 4));
#pragma unroll
        for (int j = 0; j < kGrChunk / 4; ++j)
          dst[j] = make_float4(acc[c0 + 4 * j], acc[c0 + 4 * j + 1], acc[c0 + 4 * j + 2], acc[c0 + 4 * j + 3]);
        __syncwarp();
        // eight lanes per row, four columns each
        const int cl = (lane & 7) * 4, col = n0 + c0 + cl;
#pragma unroll 2
        for (int k = 0; k < 8; ++k) {
          const int r = 4 * k + (lane >> 3), row = m0 + q * 32 + r;
          if (row >= M || col >= N) continue;
          float4 v = *reinterpret_cast<const float4*>(sl + (size_t)r * (kGrChunk + 4) + cl);
          float* out = C + (int64_t)row * p.ldc + col;
          if (p.vec) {
            if (p.accum) {
              const float4 o = *reinterpret_cast<const float4*>(out);
              v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
            }
            *reinterpret_cast<float4*>(out) = v;
          } else {
            const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (col + j < N) out[j] = p.accum ? out[j] + e[j] : e[j];
          }
        }
        __syncwarp();   // the slice is rewritten by the next chunk
      }
    }
  }
  __syncwarp();
  __syncthreads();
  if (threadIdx.x == 0) {
    // every MMA complete before the TMEM is freed (at once unless a wait gave up)
    const bool d = tc_mbar_wait(smem_u32(&done_bar), 0u);
    if (s_fail || !d) atomicExch(p.err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kCols));
  }
}

// cuTensorMapEncodeTiled, looked up once through the runtime (no link against
// the driver library)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
    else
      cudaGetLastError();
  }
  return fn;
}
// 2-D BF16 map of a rows x cols matrix (cols contiguous, row stride ld elements),
// box of box_rows x 64, 128-byte swizzle, zero fill outside
static bool tc_map(CUtensorMap* map, const __nv_bfloat16* base, int64_t rows, int cols, int64_t ld, int box_rows) {
  EncodeTiledFn fn = encode_tiled();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kTcK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      n = 1;
    }
  }
  return n;
}
// Width of a forward tile: the widest of 256, 128, 64 that divides N and still gives at
// least half of the SMs a tile; 64 otherwise (512 rows, 1024 columns, K = 512: 16 tiles
// of 256 took 13.3 us, 64 tiles of 64 take 8.9).
static int tc_bn(int M, int N) {
  for (int bn : {256, 128})
    if (N % bn == 0 && (int64_t)((M + kTcM - 1) / kTcM) * (N / bn) * 2 >= sm_count()) return bn;
  return 64;
}
// persistent launch: one CTA per SM (or per tile, when there are fewer)
template <int EPI>
static void gemm_tc(const CUtensorMap& ma, const CUtensorMap& mb, const TcArgs& g, int bn, cudaStream_t s) {
  const int64_t tiles = (int64_t)(g.N / bn) * ((g.M + kTcM - 1) / kTcM);
  const unsigned grid = (unsigned)(tiles < sm_count() ? tiles : sm_count());
  if (bn == 256) k_gemm_tc<EPI, 256><<<grid, kTcThreads, tc_smem_bytes<256>(), s>>>(ma, mb, g);
  else if (bn == 128) k_gemm_tc<EPI, 128><<<grid, kTcThreads, tc_smem_bytes<128>(), s>>>(ma, mb, g);
  else k_gemm_tc<EPI, 64><<<grid, kTcThreads, tc_smem_bytes<64>(), s>>>(ma, mb, g);
}
template <int EPI>
static void gemm_tc_prepare() {
  cudaFuncSetAttribute(k_gemm_tc<EPI, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem_bytes<256>());
  cudaFuncSetAttribute(k_gemm_tc<EPI, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem_bytes<128>());
  cudaFuncSetAttribute(k_gemm_tc<EPI, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem_bytes<64>());
}

// Wt[c][r] = bf16(W[r][c]) for a rows x cols FP32 matrix: 64 x 64 tiles through shared
// memory, both sides in whole row segments
__global__ void __launch_bounds__(256) k_transpose_bf16(const float* __restrict__ W, int rows, int cols,
                                                        __nv_bfloat16* __restrict__ Wt) {
  __shared__ __nv_bfloat16 t[64][66];
  const int r0 = blockIdx.y * 64, c0 = blockIdx.x * 64, x = threadIdx.x & 63, y = threadIdx.x >> 6;
#pragma unroll 4
  for (int r = y; r < 64; r += 4)
    if (r0 + r < rows && c0 + x < cols) t[r][x] = __float2bfloat16(W[(int64_t)(r0 + r) * cols + c0 + x]);
  __syncthreads();
#pragma unroll 4
  for (int c = y; c < 64; c += 4)
    if (c0 + c < cols && r0 + x < rows) Wt[(int64_t)(c0 + c) * rows + r0 + x] = t[x][c];
}
// BF16 rows with another stride (the tensor maps want strides of 16 bytes)
__global__ void k_pad_bf16(const __nv_bfloat16* __restrict__ W, int rows, int cols, int ld,
                           __nv_bfloat16* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < (int64_t)rows * cols) out[i / cols * ld + i % cols] = W[i];
}

// ------------------------------------------------------------------ input
// One warp per row of x: its BF16 copy (the first product's operand) and the output
// weighting w[b][c] = exp(4 (x_c - max x)) / sqrt(sum_c exp(8 (x_c - max x))) =
// sqrt(S_c / sum S) for x_c = (log S_c - mean) / 8.  The sum is formed as four partial
// sums (columns c mod 128 in [32 k, 32 k + 32) in the k-th), each over the lanes, added in order.
__global__ void __launch_bounds__(256) k_net_input(const float* __restrict__ x, int batch, int n_in,
                                                   __nv_bfloat16* __restrict__ xb, float* __restrict__ w) {
  const int64_t b = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (b >= batch) return;
  const float* xr = x + b * n_in;
  float mx = -3.0e38f;
  for (int c = lane; c < n_in; c += 32) {
    const float v = xr[c];
    xb[b * n_in + c] = __float2bfloat16(v);
    mx = fmaxf(mx, v);
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  float t = 0.f;
  for (int k = 0; k < 4; ++k) {
    float acc = 0.f;
    for (int c = lane + 32 * k; c < n_in; c += 128) acc += expf(8.f * (xr[c] - mx));
    t += warp_sum_t(acc);
  }
  const float inv = rsqrtf(t);
  for (int c = lane; c < n_in; c += 32) w[b * n_in + c] = expf(4.f * (xr[c] - mx)) * inv;
}

// ------------------------------------------------------------------ backward, elementwise
// Sign-invariant loss and its gradient; one warp per (sample, vector).
//   loss[b * n_vec + k] = ||p||^2 + ||t||^2 - 2 |p.t|
//   dp = 2 (p - sign(p.t) t) * scale, then times the output weighting (y = w o: d o = w d y)
__global__ void k_loss(const float* __restrict__ out, const float* __restrict__ target, const float* __restrict__ wgt,
                       int batch, int n_vec, int n_in, float scale, float* __restrict__ loss,
                       float* __restrict__ d_out) {
  const int lane = threadIdx.x & 31;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= (int64_t)batch * n_vec) return;
  const float* p = out + w * n_in;
  const float* t = target + w * n_in;
  const float* wr = wgt + w / n_vec * n_in;
  float pt = 0.f, pp = 0.f, tt = 0.f;
  for (int i = lane; i < n_in; i += 32) {
    const float a = p[i], b = t[i];
    pt = fmaf(a, b, pt);
    pp = fmaf(a, a, pp);
    tt = fmaf(b, b, tt);
  }
  pt = warp_sum_t(pt);
  pp = warp_sum_t(pp);
  tt = warp_sum_t(tt);
  const float sg = pt >= 0.f ? 1.f : -1.f;
  if (lane == 0) loss[w] = pp + tt - 2.f * fabsf(pt);
  float* dp = d_out + w * n_in;
  for (int i = lane; i < n_in; i += 32) dp[i] = 2.f * scale * (p[i] - sg * t[i]) * wr[i];
}

// v = hi + mid + lo in BF16, exactly: hi v rounded to 6 bits, mid the rest rounded to 8,
// lo what is left (at most 8 bits).  The 6-bit hi leaves 14-bit products, so fewer of
// their bits are cut where the tensor core accumulates them.  An infinity or a NaN stays
// in hi; a value that would round up to infinity is cut instead.
__device__ __forceinline__ void bf16_parts(float v, __nv_bfloat16 (&p)[3]) {
  const uint32_t u = __float_as_uint(v);
  p[1] = p[2] = __float2bfloat16(0.f);
  if (!(fabsf(v) < INFINITY)) {
    p[0] = __float2bfloat16(v);
    return;
  }
  uint32_t h = (u + 0x1ffffu + ((u >> 18) & 1u)) & 0xfffc0000u;   // 5 fraction bits, ties to even
  if ((h & 0x7f800000u) == 0x7f800000u) h = u & 0xfffc0000u;
  const float hi = __uint_as_float(h), r1 = v - hi;
  p[0] = __float2bfloat16(hi);
  p[1] = __float2bfloat16(r1);
  p[2] = __float2bfloat16(r1 - __bfloat162float(p[1]));
}

// A layer's output gradient: the sum of `splits` partial products, masked by the ReLU
// (mask > 0; the sign of the BF16 activation is the activation's), as three BF16 parts in
// both layouts the products read, dk[part][row][ldk] (null: not needed) and
// dt[part][col][ldt] (rows beyond `rows` zero), with the column sums of each 64 rows.
// One 64 x 64 tile per CTA; bound by its bytes, S x 4 in and 6 or 12 out per value.
__global__ void __launch_bounds__(256) k_split_grad(const float* __restrict__ src, int splits, int64_t sstride, int rows,
                                                    int cols, const __nv_bfloat16* __restrict__ mask,
                                                    __nv_bfloat16* __restrict__ dk, int ldk, int64_t pk,
                                                    __nv_bfloat16* __restrict__ dt, int ldt, int64_t pt,
                                                    float* __restrict__ csum) {
  __shared__ __nv_bfloat16 tile[3][64][66];
  __shared__ float cs[4][64];
  const int c0 = blockIdx.x * 64, r0 = blockIdx.y * 64, x = threadIdx.x & 63, y = threadIdx.x >> 6;
  const int col = c0 + x;
  float v[16];
  float mk[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {      // every load of a pass in flight before the first use
    const int row = r0 + y + 4 * j;
    const bool in = row < rows && col < cols;
    const int64_t at = (int64_t)row * cols + col;
    v[j] = in ? src[at] : 0.f;
    mk[j] = (in && mask) ? __bfloat162float(mask[at]) : 1.f;
  }
  for (int k = 1; k < splits; ++k) {
    float a[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int row = r0 + y + 4 * j;
      a[j] = (row < rows && col < cols) ? src[k * sstride + (int64_t)row * cols + col] : 0.f;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] += a[j];
  }
  float acc = 0.f;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int r = y + 4 * j, row = r0 + r;
    if (!(mk[j] > 0.f)) v[j] = 0.f;
    __nv_bfloat16 p[3];
    bf16_parts(v[j], p);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      tile[k][r][x] = p[k];
      if (dk && row < rows && col < cols) dk[k * pk + (int64_t)row * ldk + col] = p[k];
    }
    acc += v[j];
  }
  cs[y][x] = acc;
  __syncthreads();
#pragma unroll 4
  for (int c = y; c < 64; c += 4) {
    if (c0 + c >= cols) break;
#pragma unroll
    for (int k = 0; k < 3; ++k) dt[k * pt + (int64_t)(c0 + c) * ldt + r0 + x] = tile[k][x][c];
  }
  if (y == 0 && col < cols) csum[(int64_t)blockIdx.y * cols + col] = (cs[0][x] + cs[1][x]) + (cs[2][x] + cs[3][x]);
}
// The sums that end a backward pass, one launch: CTAs of blockIdx.y = 0, 1, 2 the bias
// gradients db[col] (+)= the 64-row sums in order, y = 3 (one CTA) the loss total in FP64
// (256 interleaved chains and a fixed tree; one thread's chain over 5632 values took 450 us).
struct SumArgs {
  const float* csum[3];
  float* db[3];
  int cols[3];
  int chunks, accum;
  const float* loss;
  int nl;
  float* total;
};
__global__ void __launch_bounds__(256) k_grad_sums(const SumArgs a) {
  if (blockIdx.y == 3) {
    if (blockIdx.x != 0 || a.nl <= 0) return;
    __shared__ double sh[8];
    double acc = 0.0;
#pragma unroll 8
    for (int i = threadIdx.x; i < a.nl; i += 256) acc += a.loss[i];
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int k = 1; k < 8; ++k) acc += sh[k];
      *a.total = (float)acc;
    }
    return;
  }
  const int l = blockIdx.y, cols = a.cols[l], n = blockIdx.x * 256 + threadIdx.x;
  if (n >= cols) return;
  float acc = a.accum ? a.db[l][n] : 0.f;
#pragma unroll 8
  for (int b = 0; b < a.chunks; ++b) acc += a.csum[l][(int64_t)b * cols + n];
  a.db[l][n] = acc;
}
// out[col][ld] = in[row][cols] transposed (BF16), zero for rows .. ld; the three layers'
// inputs in one launch (blockIdx.z)
struct TransArgs {
  const __nv_bfloat16* in[3];
  __nv_bfloat16* out[3];
  int cols[3];
  int rows, ld;
};
__global__ void __launch_bounds__(256) k_transpose_act(const TransArgs a) {
  __shared__ __nv_bfloat16 t[64][66];
  const int l = blockIdx.z, cols = a.cols[l];
  const int r0 = blockIdx.y * 64, c0 = blockIdx.x * 64, x = threadIdx.x & 63, y = threadIdx.x >> 6;
  if (c0 >= cols) return;
  __nv_bfloat16 v[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int row = r0 + y + 4 * j;
    v[j] = (row < a.rows && c0 + x < cols) ? a.in[l][(int64_t)row * cols + c0 + x] : __float2bfloat16(0.f);
  }
#pragma unroll
  for (int j = 0; j < 16; ++j) t[y + 4 * j][x] = v[j];
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int c = y + 4 * j;
    if (c0 + c < cols) a.out[l][(int64_t)(c0 + c) * a.ld + r0 + x] = t[x][c];
  }
}

// Adam (Kingma and Ba, 2015) on the FP32 masters; refresh the BF16 copies.  Nothing is
// touched when the error word is set: the gradients are then incomplete (a product's wait
// gave up), and masters and moments must survive the call that reports it.
__global__ void k_adam(float* __restrict__ w, __nv_bfloat16* __restrict__ w16, const float* __restrict__ g,
                       float* __restrict__ m, float* __restrict__ v, int64_t n, float lr, float b1, float b2,
                       float eps, float c1, float c2, const int* __restrict__ err) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || *err) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  w[i] = wi;
  w16[i] = __float2bfloat16(wi);
}

__global__ void k_to_bf16(const float* __restrict__ a, __nv_bfloat16* __restrict__ b, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = __float2bfloat16(a[i]);
}

// Deterministic initial weights: uniform(-a, a), a = sqrt(6 / fan_in), from a
// counter-based hash of (seed, index) (the splitmix64 finaliser); biases zero.
__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__global__ void k_init_uniform(float* __restrict__ w, int64_t n, uint64_t seed, float a) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t h = splitmix64(seed ^ splitmix64((uint64_t)i));
  const float u = (float)((h >> 40) * (1.0 / 16777216.0));   // [0, 1)
  w[i] = a * (2.f * u - 1.f);
}

static inline unsigned g256(int64_t n) { return (unsigned)((n + 255) / 256); }

// ------------------------------------------------------------------ passes
// The products' operands are BF16: the weights (the masters' BF16 copies) and
// the activations (x, h1, h2 rounded to BF16 before the product that reads them);
// accumulation is FP32.  With layer widths multiples of 64 the forward products run
// on the tensor cores (tcgen05, k_gemm_tc), otherwise on the CUDA cores (k_gemm)
// with the same operands.  The backward products have one FP32 operand, the gradient:
// it enters the tensor cores as three BF16 parts (24 bits), at any width.
static inline dim3 g64(int64_t cols, int64_t rows) { return dim3((unsigned)((cols + 63) / 64), (unsigned)((rows + 63) / 64)); }

static void net_refresh_bf16(msmg_net* t, cudaStream_t s) {
  const int64_t dims[4] = {t->d.n_in, t->d.hidden[0], t->d.hidden[1], t->n_out};
  for (int l = 0; l < 3; ++l) {
    if (t->tc)
      k_transpose_bf16<<<g64(dims[l + 1], dims[l]), 256, 0, s>>>(t->w32 + t->off_w[l], (int)dims[l], (int)dims[l + 1],
                                                                 t->wt16 + t->off_w[l]);
    if (l > 0 && t->wp[l] != t->w16 + t->off_w[l])
      k_pad_bf16<<<g256(dims[l] * dims[l + 1]), 256, 0, s>>>(t->w16 + t->off_w[l], (int)dims[l], (int)dims[l + 1],
                                                             t->ldw[l], t->wp[l]);
  }
}

// The three forward products on the tensor cores, the output to y; with ev (6 events)
// each launch is bracketed by ev[2l], ev[2l + 1].
static void net_tc_products(msmg_net* t, int batch, float* y, cudaStream_t s, cudaEvent_t* ev) {
  const msmg_net_desc& d = t->d;
  const int dims[4] = {d.n_in, d.hidden[0], d.hidden[1], t->n_out};
  __nv_bfloat16* const acts[3] = {t->xb, t->h1b, t->h2b};
  if (t->fmap_rows != batch) {
    t->fmap_rows = 0;
    for (int l = 0; l < 3; ++l) {
      const int K = dims[l], N = dims[l + 1];
      if (!tc_map(&t->fmap[l][0], acts[l], batch, K, K, kTcM) ||
          !tc_map(&t->fmap[l][1], t->wt16 + t->off_w[l], N, K, K, tc_bn(batch, N))) {
        t->map_err = 1;
        return;
      }
    }
    t->fmap_rows = batch;
  }
  for (int l = 0; l < 3; ++l) {
    const int K = dims[l], N = dims[l + 1], bn = tc_bn(batch, N);
    const CUtensorMap &ma = t->fmap[l][0], &mb = t->fmap[l][1];
    const TcArgs g{y, l < 2 ? acts[l + 1] : nullptr, t->w32 + t->off_b[l], t->wgt, d.n_in, batch, N, K, t->err};
    if (ev) cudaEventRecord(ev[2 * l], s);
    if (l < 2) gemm_tc<2>(ma, mb, g, bn, s);
    else gemm_tc<1>(ma, mb, g, bn, s);
    if (ev) cudaEventRecord(ev[2 * l + 1], s);
  }
}

// forward for `batch` rows of x; output to y (16-byte aligned)
static void net_forward(msmg_net* t, const float* x, int batch, float* y, cudaStream_t s) {
  const msmg_net_desc& d = t->d;
  const int h1 = d.hidden[0], h2 = d.hidden[1], no = t->n_out;
  k_net_input<<<(unsigned)((batch + 7) / 8), 256, 0, s>>>(x, batch, d.n_in, t->xb, t->wgt);
  if (t->tc) {
    net_tc_products(t, batch, y, s, nullptr);
  } else {
    gemm<2>(t->xb, t->w16 + t->off_w[0], nullptr, t->h1b, t->w32 + t->off_b[0], nullptr, 1, batch, h1, d.n_in, s);
    gemm<2>(t->h1b, t->w16 + t->off_w[1], nullptr, t->h2b, t->w32 + t->off_b[1], nullptr, 1, batch, h2, h1, s);
    gemm<3>(t->h2b, t->w16 + t->off_w[2], y, nullptr, t->w32 + t->off_b[2], t->wgt, d.n_in, batch, no, h2, s);
  }
}
// to any y: through the network's own buffer where y is not 16-byte aligned
static int net_forward_to(msmg_net* t, const float* x, int batch, float* y, cudaStream_t s) {
  const bool direct = (reinterpret_cast<uintptr_t>(y) & 15) == 0;
  net_forward(t, x, batch, direct ? y : t->out, s);
  if (!direct)
    MSMG_CUDA_TRY(cudaMemcpyAsync(y, t->out, (size_t)batch * t->n_out * sizeof(float), cudaMemcpyDeviceToDevice, s));
  return 0;
}

// one backward product
template <int NA, int NB>
static void grad_product(const CUtensorMap& ma, const CUtensorMap& mb, const GrArgs& g, cudaStream_t s) {
  const int64_t tiles = (int64_t)((g.N + kGrN - 1) / kGrN) * ((g.M + kTcM - 1) / kTcM) * g.splits;
  k_gemm_grad<NA, NB><<<(unsigned)(tiles < sm_count() ? tiles : sm_count()), kTcThreads, kGrSmem, s>>>(ma, mb, g);
}
// tensor maps of a backward chunk of `rows` rows
static bool net_grad_maps(msmg_net* t, const int (&dims)[4], int rows) {
  if (t->gmap_rows == rows) return true;
  const int rp = (rows + 63) / 64 * 64;
  t->gmap_rows = 0;
  for (int l = 0; l < 3; ++l) {
    const int fi = dims[l], fo = dims[l + 1], ldk = (fo + 7) / 8 * 8;
    if (l > 0 && (!tc_map(&t->gmap[l][0], t->dk, (int64_t)3 * rows, fo, ldk, kTcM) ||
                  !tc_map(&t->gmap[l][1], t->wp[l], fi, fo, t->ldw[l], kGrN)))
      return false;
    if (!tc_map(&t->gmap[l][2], t->at[l], fi, rp, rp, kTcM) || !tc_map(&t->gmap[l][3], t->dt, (int64_t)3 * fo, rp, rp, kGrN))
      return false;
  }
  t->gmap_rows = rows;
  return true;
}

// Loss and gradients (to grad, 16-byte aligned) for `batch` rows, forward included; the loss
// total goes to the word after t->err.
// Per chunk of rows and layer (3, 2, 1): the gradient's parts and column sums
// (k_split_grad), dW = act^T d with the rows as K, and the input's gradient d W^T, its K
// blocks split over CTAs where the output has few tiles (the next k_split_grad adds the
// partial sums).
static void net_backward(msmg_net* t, const float* x, const float* target, int batch, float* grad, cudaStream_t s) {
  const msmg_net_desc& d = t->d;
  const int dims[4] = {d.n_in, d.hidden[0], d.hidden[1], t->n_out};
  const __nv_bfloat16* const acts[3] = {t->xb, t->h1b, t->h2b};
  net_forward(t, x, batch, t->out, s);
  const int nl = batch * d.n_vec;
  const float scale = 1.f / (float)nl;
  k_loss<<<(unsigned)(((int64_t)nl * 32 + 255) / 256), 256, 0, s>>>(t->out, target, t->wgt, batch, d.n_vec, d.n_in,
                                                                   scale, t->loss, t->d_out);
  for (int b0 = 0; b0 < batch; b0 += t->rc) {
    const int rows = batch - b0 < t->rc ? batch - b0 : t->rc, rp = (rows + 63) / 64 * 64;
    if (!net_grad_maps(t, dims, rows)) {
      t->map_err = 1;
      return;
    }
    const float* src = t->d_out + (int64_t)b0 * t->n_out;
    int splits = 1;
    int64_t sstride = 0;
    TransArgs ta;
    SumArgs sa;
    int top = 0, top_out = 0;
    for (int l = 0; l < 3; ++l) {
      ta.in[l] = acts[l] + (int64_t)b0 * dims[l];
      ta.out[l] = t->at[l];
      ta.cols[l] = dims[l];
      sa.csum[l] = t->csum[l];
      sa.db[l] = grad + t->off_b[l];
      sa.cols[l] = dims[l + 1];
      top = dims[l] > top ? dims[l] : top;
      top_out = dims[l + 1] > top_out ? dims[l + 1] : top_out;
    }
    ta.rows = rows;
    ta.ld = rp;
    sa.chunks = rp / 64;
    sa.accum = b0 > 0;
    sa.loss = t->loss;
    sa.nl = b0 == 0 ? nl : 0;
    sa.total = reinterpret_cast<float*>(t->err + 1);
    k_transpose_act<<<dim3((unsigned)((top + 63) / 64), (unsigned)(rp / 64), 3), 256, 0, s>>>(ta);
    for (int l = 2; l >= 0; --l) {
      const int fi = dims[l], fo = dims[l + 1];
      const int ldk = (fo + 7) / 8 * 8;
      const __nv_bfloat16* mask = l < 2 ? acts[l + 1] + (int64_t)b0 * fo : nullptr;
      k_split_grad<<<g64(fo, rp), 256, 0, s>>>(src, splits, sstride, rows, fo, mask, l > 0 ? t->dk : nullptr, ldk,
                                               (int64_t)rows * ldk, t->dt, rp, (int64_t)fo * rp, t->csum[l]);
      GrArgs g{};
      if (l > 0) {
        // d_in = d W^T: M rows, N = fan_in, K = fan_out
        g.err = t->err;
        g.M = g.rows_a = rows;
        g.N = g.rows_b = fi;
        g.K = fo;
        const int64_t tiles = (int64_t)((rows + kTcM - 1) / kTcM) * ((fi + kGrN - 1) / kGrN);
        const int nkb = (fo + kTcK - 1) / kTcK;
        int64_t sp = sm_count() / tiles;
        if (sp > (nkb + 3) / 4) sp = (nkb + 3) / 4;          // four K blocks a split at least
        if (sp * rows * fi > t->part_cap) sp = t->part_cap / ((int64_t)rows * fi);
        g.splits = (int)(sp < 1 ? 1 : sp);
        g.C = t->part;
        g.ldc = fi;
        g.split_stride = sstride = (int64_t)rows * fi;
        g.vec = fi % 4 == 0;
        splits = g.splits;
        grad_product<3, 1>(t->gmap[l][0], t->gmap[l][1], g, s);
        src = t->part;
      }
      // dW = act^T d: M = fan_in, N = fan_out, K = rows
      g = GrArgs{};
      g.err = t->err;
      g.M = g.rows_a = fi;
      g.N = g.rows_b = fo;
      g.K = rp;
      g.splits = 1;
      g.C = grad + t->off_w[l];
      g.ldc = fo;
      g.vec = fo % 4 == 0;
      g.accum = b0 > 0;
      grad_product<1, 3>(t->gmap[l][2], t->gmap[l][3], g, s);
    }
    k_grad_sums<<<dim3((unsigned)((top_out + 255) / 256), 4), 256, 0, s>>>(sa);
  }
}

}  // namespace msmg

using namespace msmg;

static int64_t net_layout(const msmg_net_desc* d, int64_t off_w[3], int64_t off_b[3]) {
  const int n_out = d->n_vec * d->n_in;
  const int64_t dims[4] = {d->n_in, d->hidden[0], d->hidden[1], n_out};
  int64_t o = 0;
  for (int l = 0; l < 3; ++l) {
    off_w[l] = o;
    o += dims[l] * dims[l + 1];
    o = (o + 63) / 64 * 64;
    off_b[l] = o;
    o += dims[l + 1];
    o = (o + 63) / 64 * 64;
  }
  return o;
}

static bool desc_ok(const msmg_net_desc* d) {
  return d && d->n_in >= 1 && d->n_in <= 4096 && d->hidden[0] >= 1 && d->hidden[1] >= 1 && d->hidden[0] <= 16384 &&
         d->hidden[1] <= 16384 && d->n_vec >= 1 && d->n_vec <= 64 && d->batch_max >= 1 && d->batch_max <= 1 << 20;
}

// rows of a backward chunk: its parts take 12 bytes per row and output value, so that a
// network made for large inference batches does not carry them for every row
constexpr int64_t kBackRows = 4096;
constexpr int64_t kPartFloats = (int64_t)152 * 128 * 128;  // one partial tile per SM

static int64_t net_carve(const msmg_net_desc* d, Arena& ar, msmg_net* t) {
  int64_t ow[3], ob[3];
  const int64_t np = net_layout(d, ow, ob);
  const int no = d->n_vec * d->n_in;
  const int64_t B = d->batch_max;
  float* w32 = ar.take<float>(np);
  __nv_bfloat16* w16 = ar.take<__nv_bfloat16>(np);
  float* grad = ar.take<float>(np);
  float* am = ar.take<float>(np);
  float* av = ar.take<float>(np);
  float* out = ar.take<float>(B * no);
  float* dout = ar.take<float>(B * no);
  float* loss = ar.take<float>(B * d->n_vec + 32);
  float* wgt = ar.take<float>(B * d->n_in);
  const bool tc = d->n_in % 64 == 0 && d->hidden[0] % 64 == 0 && d->hidden[1] % 64 == 0;
  __nv_bfloat16* wt16 = ar.take<__nv_bfloat16>(tc ? np : 0);
  __nv_bfloat16* xb = ar.take<__nv_bfloat16>(B * d->n_in);
  __nv_bfloat16* h1b = ar.take<__nv_bfloat16>(B * d->hidden[0]);
  __nv_bfloat16* h2b = ar.take<__nv_bfloat16>(B * d->hidden[1]);
  // backward, in chunks of kBackRows rows
  const int64_t dims[4] = {d->n_in, d->hidden[0], d->hidden[1], no};
  const int64_t rc = B < kBackRows ? B : kBackRows, rcp = (rc + 63) / 64 * 64;
  int64_t top = 0, hid = dims[1] > dims[2] ? dims[1] : dims[2];
  for (int l = 1; l < 4; ++l) top = dims[l] > top ? dims[l] : top;
  const int64_t part_cap = rc * hid > kPartFloats ? rc * hid : kPartFloats;
  __nv_bfloat16* dk = ar.take<__nv_bfloat16>(3 * rc * ((top + 7) / 8 * 8));
  __nv_bfloat16* dt = ar.take<__nv_bfloat16>(3 * top * rcp);
  __nv_bfloat16* at[3];
  for (int l = 0; l < 3; ++l) at[l] = ar.take<__nv_bfloat16>(dims[l] * rcp);
  __nv_bfloat16* wp[3] = {nullptr, nullptr, nullptr};
  int ldw[3] = {0, 0, 0};
  for (int l = 1; l < 3; ++l) {
    ldw[l] = (int)((dims[l + 1] + 7) / 8 * 8);
    wp[l] = ldw[l] == dims[l + 1] ? (w16 ? w16 + ow[l] : nullptr) : ar.take<__nv_bfloat16>(dims[l] * ldw[l]);
  }
  float* part = ar.take<float>(part_cap);
  float* csum[3];
  for (int l = 0; l < 3; ++l) csum[l] = ar.take<float>(rcp / 64 * dims[l + 1]);
  int* err = ar.take<int>(4);
  if (t) {
    t->d = *d;
    t->n_out = no;
    t->n_param = np;
    for (int l = 0; l < 3; ++l) { t->off_w[l] = ow[l]; t->off_b[l] = ob[l]; }
    t->w32 = w32; t->w16 = w16; t->grad = grad; t->adam_m = am; t->adam_v = av;
    t->out = out; t->d_out = dout; t->loss = loss;
    t->wgt = wgt;
    t->step = 0;
    t->wt16 = wt16; t->xb = xb; t->h1b = h1b; t->h2b = h2b; t->err = err;
    t->rc = (int)rc;
    t->dk = dk; t->dt = dt; t->part = part; t->part_cap = part_cap;
    for (int l = 0; l < 3; ++l) { t->at[l] = at[l]; t->csum[l] = csum[l]; t->wp[l] = wp[l]; t->ldw[l] = ldw[l]; }
    t->tc = tc;
  }
  return np;
}

// --------------------------------------------------------------- set-up integration
namespace msmg {

// x[e][c] = clamp(log S_c - mean_e log S, -20, 20) / 8: the element's
// log-permeability pattern up to a constant factor (for isotropic kappa,
// log S = log kappa + const), the scale-free input of the network.
// Output row: the element itself, or its lexicographic index when lex_of_hid is given.
__global__ void k_net_features(const double* __restrict__ S, int nb, int64_t m, const int* __restrict__ lex_of_hid,
                               float* __restrict__ x) {
  const int64_t e = blockIdx.x;
  if (e >= m) return;
  const int64_t row = lex_of_hid ? (int64_t)lex_of_hid[e] : e;
  __shared__ double red[32];
  double acc = 0.0;
  for (int c = threadIdx.x; c < nb; c += blockDim.x) acc += log(S[e * nb + c]);
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) t += red[w];
    red[0] = t / nb;
  }
  __syncthreads();
  const double mean = red[0];
  for (int c = threadIdx.x; c < nb; c += blockDim.x) {
    double v = log(S[e * nb + c]) - mean;
    v = v < -20.0 ? -20.0 : (v > 20.0 ? 20.0 : v);
    x[row * nb + c] = (float)(v / 8.0);
  }
}

// y[e][k - 1][c] = sqrt(S_c) Phi[e][k][c], k = 1 .. L-1: the level-1 eigenvectors
// in the symmetric form (Euclidean-orthonormal), the network's targets.
__global__ void k_net_targets(const double* __restrict__ S, const double* __restrict__ Phi, int nb, int L, int64_t m,
                              const int* __restrict__ lex_of_hid, float* __restrict__ y) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = m * (L - 1) * nb;
  if (i >= total) return;
  const int c = (int)(i % nb);
  const int64_t ek = i / nb;
  const int k = (int)(ek % (L - 1)) + 1;
  const int64_t e = ek / (L - 1);
  const int64_t row = lex_of_hid ? (int64_t)lex_of_hid[e] : e;
  y[(row * (L - 1) + (k - 1)) * nb + c] = (float)(sqrt(S[e * nb + c]) * Phi[(e * L + k) * nb + c]);
}

void launch_net_features(msmg_ctx* c, float* x, const int* lex_of_hid, cudaStream_t s) {
  k_net_features<<<(unsigned)c->fine.m, 128, 0, s>>>(c->fine.S, c->fine.nb, c->fine.m, lex_of_hid, x);
}

int net_status(msmg_net* t, cudaStream_t s, float* loss = nullptr);

// Guesses for every element, in chunks of the network's batch: g[e][k-1][c].
int net_guesses(msmg_ctx* c, const msmg_net* net, float* x, float* g, cudaStream_t s) {
  msmg_net* t = const_cast<msmg_net*>(net);
  launch_net_features(c, x, nullptr, s);
  const int64_t m = c->fine.m;
  const int nb = c->fine.nb;
  for (int64_t e0 = 0; e0 < m; e0 += t->d.batch_max) {
    const int b = (int)((m - e0) < t->d.batch_max ? (m - e0) : t->d.batch_max);
    const int st = net_forward_to(t, x + e0 * nb, b, g + e0 * t->n_out, s);
    if (st) return st;
  }
  MSMG_CUDA_TRY(cudaGetLastError());
  return net_status(t, s);
}

// MSMG_ERR_DEVICE_TIMEOUT when a tensor-core wait of the network's products gave up
// (synchronises the stream; clears the word), MSMG_ERR_CUDA when a tensor map
// could not be encoded (the products were not launched).  loss (may be null) receives the
// loss total, read with the error word.
int net_status(msmg_net* t, cudaStream_t s, float* loss) {
  if (t->map_err) {
    t->map_err = 0;
    return MSMG_ERR_CUDA;
  }
  struct { int err; float loss; } h{0, 0.f};
  MSMG_CUDA_TRY(cudaMemcpyAsync(&h, t->err, loss ? 8 : 4, cudaMemcpyDeviceToHost, s));
  MSMG_CUDA_TRY(cudaStreamSynchronize(s));
  if (h.err) {
    MSMG_CUDA_TRY(cudaMemsetAsync(t->err, 0, sizeof(int), s));
    return MSMG_ERR_DEVICE_TIMEOUT;
  }
  if (loss) *loss = h.loss;
  return 0;
}

bool net_matches(const msmg_ctx* c, const msmg_net* net) {
  return net && net->d.n_in == c->fine.nb && net->d.n_vec == c->fine.L - 1;
}

}  // namespace msmg

extern "C" {

size_t msmg_net_workspace_size(const msmg_net_desc* desc) {
  if (!desc_ok(desc)) return 0;
  Arena ar;
  net_carve(desc, ar, nullptr);
  return ar.off + 256;
}

int msmg_net_create(const msmg_net_desc* desc, void* workspace, size_t workspace_bytes, uint64_t seed,
                    msmg_stream stream, msmg_net** out) {
  if (!out || !desc_ok(desc) || !workspace) return MSMG_ERR_INVALID_ARG;
  *out = nullptr;
  if (reinterpret_cast<uintptr_t>(workspace) % 256) return MSMG_ERR_WORKSPACE;
  if (workspace_bytes < msmg_net_workspace_size(desc)) return MSMG_ERR_WORKSPACE;
  msmg_net* t = new (std::nothrow) msmg_net{};
  if (!t) return MSMG_ERR_INVALID_ARG;
  Arena ar;
  ar.base = static_cast<char*>(workspace);
  ar.cap = workspace_bytes;
  net_carve(desc, ar, t);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  MSMG_CUDA_TRY(cudaMemsetAsync(t->w32, 0, (size_t)t->n_param * sizeof(float), s));
  MSMG_CUDA_TRY(cudaMemsetAsync(t->adam_m, 0, (size_t)t->n_param * sizeof(float), s));
  MSMG_CUDA_TRY(cudaMemsetAsync(t->adam_v, 0, (size_t)t->n_param * sizeof(float), s));
  const int64_t dims[4] = {desc->n_in, desc->hidden[0], desc->hidden[1], t->n_out};
  for (int l = 0; l < 3; ++l) {
    const int64_t n = dims[l] * dims[l + 1];
    k_init_uniform<<<g256(n), 256, 0, s>>>(t->w32 + t->off_w[l], n, seed * 4 + (uint64_t)l,
                                           sqrtf(6.f / (float)dims[l]) * (l == 2 ? 0.25f : 1.f));
  }
  k_to_bf16<<<g256(t->n_param), 256, 0, s>>>(t->w32, t->w16, t->n_param);
  net_refresh_bf16(t, s);
  MSMG_CUDA_TRY(cudaMemsetAsync(t->err, 0, 4 * sizeof(int), s));
  cudaFuncSetAttribute(k_gemm_grad<3, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGrSmem);
  cudaFuncSetAttribute(k_gemm_grad<1, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGrSmem);
  gemm_tc_prepare<1>();
  gemm_tc_prepare<2>();
  MSMG_CUDA_TRY(cudaGetLastError());
  *out = t;
  return 0;
}

void msmg_net_destroy(msmg_net* net) { delete net; }

int64_t msmg_net_param_count(const msmg_net* net) { return net ? net->n_param : 0; }

int msmg_net_param_offsets(const msmg_net* net, int64_t* w_off, int64_t* b_off) {
  if (!net || !w_off || !b_off) return MSMG_ERR_INVALID_ARG;
  for (int l = 0; l < 3; ++l) { w_off[l] = net->off_w[l]; b_off[l] = net->off_b[l]; }
  return 0;
}

int msmg_net_get_params(const msmg_net* net, float* params, msmg_stream stream) {
  if (!net || !params) return MSMG_ERR_INVALID_ARG;
  MSMG_CUDA_TRY(cudaMemcpyAsync(params, net->w32, (size_t)net->n_param * sizeof(float), cudaMemcpyDeviceToDevice,
                                reinterpret_cast<cudaStream_t>(stream)));
  return 0;
}

int msmg_net_set_params(msmg_net* net, const float* params, msmg_stream stream) {
  if (!net || !params) return MSMG_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  MSMG_CUDA_TRY(cudaMemcpyAsync(net->w32, params, (size_t)net->n_param * sizeof(float), cudaMemcpyDeviceToDevice, s));
  k_to_bf16<<<g256(net->n_param), 256, 0, s>>>(net->w32, net->w16, net->n_param);
  net_refresh_bf16(net, s);
  MSMG_CUDA_TRY(cudaGetLastError());
  return 0;
}

int msmg_net_forward(msmg_net* net, const float* x, float* y, int batch, msmg_stream stream) {
  if (!net || !x || !y || batch < 0) return MSMG_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  for (int b0 = 0; b0 < batch; b0 += net->d.batch_max) {
    const int b = batch - b0 < net->d.batch_max ? batch - b0 : net->d.batch_max;
    const int st = net_forward_to(net, x + (int64_t)b0 * net->d.n_in, b, y + (int64_t)b0 * net->n_out, s);
    if (st) return st;
  }
  MSMG_CUDA_TRY(cudaGetLastError());
  return net_status(net, s);
}

int msmg_net_time_products(msmg_net* net, const float* x, int batch, double* ms, msmg_stream stream) {
  if (!net || !x || !ms || batch < 1 || batch > net->d.batch_max) return MSMG_ERR_INVALID_ARG;
  if (!net->tc) return MSMG_ERR_UNSUPPORTED;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  cudaEvent_t ev[6];
  for (int i = 0; i < 6; ++i) MSMG_CUDA_TRY(cudaEventCreate(&ev[i]));
  net_forward(net, x, batch, net->out, s);   // the products' operands: BF16 input and activations
  net_tc_products(net, batch, net->out, s, ev);
  cudaError_t e = cudaStreamSynchronize(s);
  for (int l = 0; l < 3 && e == cudaSuccess; ++l) {
    float t = 0.f;
    e = cudaEventElapsedTime(&t, ev[2 * l], ev[2 * l + 1]);
    ms[l] = t;
  }
  for (int i = 0; i < 6; ++i) cudaEventDestroy(ev[i]);
  MSMG_CUDA_TRY(e);
  return net_status(net, s);
}

int msmg_net_gradients(msmg_net* net, const float* x, const float* target, int batch, float* grad, float* loss_host,
                       msmg_stream stream) {
  if (!net || !x || !target || batch < 1 || batch > net->d.batch_max) return MSMG_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // straight into the caller's array where its alignment allows the products' stores
  const bool direct = grad && (reinterpret_cast<uintptr_t>(grad) & 15) == 0;
  net_backward(net, x, target, batch, direct ? grad : net->grad, s);
  if (grad && !direct)
    MSMG_CUDA_TRY(cudaMemcpyAsync(grad, net->grad, (size_t)net->n_param * sizeof(float), cudaMemcpyDeviceToDevice, s));
  {
    const int st = net_status(net, s, loss_host);
    if (st) return st;
  }
  if (loss_host) *loss_host /= (float)(batch * net->d.n_vec);
  MSMG_CUDA_TRY(cudaGetLastError());
  return 0;
}

int msmg_net_train_step(msmg_net* net, const float* x, const float* target, int batch, float lr, float* loss_host,
                        msmg_stream stream) {
  if (!net || !x || !target || batch < 1 || batch > net->d.batch_max || !(lr > 0.f)) return MSMG_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  net_backward(net, x, target, batch, net->grad, s);
  if (net->map_err) return net_status(net, s);   // no product was launched: no gradients to step with
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float k = (float)(net->step + 1), c1 = 1.f - powf(b1, k), c2 = 1.f - powf(b2, k);
  k_adam<<<g256(net->n_param), 256, 0, s>>>(net->w32, net->w16, net->grad, net->adam_m, net->adam_v, net->n_param, lr,
                                            b1, b2, eps, c1, c2, net->err);
  net_refresh_bf16(net, s);
  {
    const int st = net_status(net, s, loss_host);
    if (st) return st;
  }
  net->step += 1;
  if (loss_host) *loss_host /= (float)(batch * net->d.n_vec);
  MSMG_CUDA_TRY(cudaGetLastError());
  return 0;
}

int msmg_learning_data(msmg_ctx* c, float* x, float* y, msmg_stream stream) {
  if (!c || !x || !y || c->fine.L < 2) return MSMG_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  launch_net_features(c, x, c->fine.lex_of_hid, s);
  const int64_t total = c->fine.m * (c->fine.L - 1) * c->fine.nb;
  k_net_targets<<<g256(total), 256, 0, s>>>(c->fine.S, c->fine.Phi, c->fine.nb, c->fine.L, c->fine.m,
                                            c->fine.lex_of_hid, y);
  MSMG_CUDA_TRY(cudaGetLastError());
  return 0;
}

}  // extern "C"

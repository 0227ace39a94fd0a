// tkf_mlp.cu -- training and inference kernels of the learned step proposer.
//
// Network: 12 inputs -> 64 SiLU -> 64 SiLU -> 1, parameters packed as W1 [64][12], b1 [64],
// W2 [64][64], b2 [64], w3 [64], b3 (FP32 master copy). Loss: mean squared error. Optimiser:
// Adam (Kingma & Ba 2015). A training step on a batch of B samples is
//   the tiles (train_tile): one CTA per 128 samples; the forward and backward pass with every
//     dense contraction on the tensor cores (tcgen05.mma kind::f16, BF16 operands, FP32
//     accumulation in tensor memory): the two layers, the backpropagation through layer 2, and
//     the weight gradients of both layers together with the bias gradients (one M128 N96 K128
//     product per CTA); the output layer, bias, SiLU and its derivative on the CUDA cores in
//     FP32; each CTA writes its partial gradient;
//   then the partials summed in CTA order (no atomics: deterministic) and the Adam step.
// mlp_train_steps_kernel runs up to 256 steps in one cooperative launch; mlp_train_tc_kernel and
// mlp_reduce_adam_kernel are one step in two launches (the gradient alone, and devices that cannot hold a
// batch's CTAs at once).
// Around training: seeded initialisation, calibration of the output bias (a quantile of the
// training residuals, by a radix select on the device) and rounding to the BF16 weights the
// fit's inference uses.
// The paper has no learned component; the learned step proposer is an addition to its method.

#include <math.h>

#include <type_traits>

#include "tkf_fit_impl.cuh"

namespace tkf {
namespace {

constexpr int kIn = 12, kHid = 64;
constexpr int oW1 = 0, oB1 = 768, oW2 = 832, oB2 = 4928, oW3 = 4992, oB3 = 5056;

__device__ __forceinline__ float sigm(float z) { return 1.0f / (1.0f + expf(-z)); }

// Per-sample activations: z1, a1, z2, a2 (4 x 64 floats), then out.
struct Act {
  float* z1;
  float* a1;
  float* z2;
  float* a2;
  float* out;
  float* dz1;
  float* dz2;
  float* dout;
};

__global__ void __launch_bounds__(128) mlp_forward_kernel(const float* __restrict__ p, const float* __restrict__ x,
                                                          int x_stride, uint32_t n, Act act) {
  __shared__ float w[kMlpParams];
  for (int k = threadIdx.x; k < kMlpParams; k += blockDim.x) w[k] = p[k];
  __syncthreads();
  const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  float in[kIn];
  for (int i = 0; i < kIn; ++i) in[i] = x[size_t(s) * x_stride + i];
  float a1[kHid];
  for (int j = 0; j < kHid; ++j) {
    float z = w[oB1 + j];
    for (int i = 0; i < kIn; ++i) z = fmaf(w[oW1 + j * kIn + i], in[i], z);
    const float a = z * sigm(z);
    a1[j] = a;
    if (act.z1) {
      act.z1[size_t(s) * kHid + j] = z;
      act.a1[size_t(s) * kHid + j] = a;
    }
  }
  float out = w[oB3];
  for (int j = 0; j < kHid; ++j) {
    float z = w[oB2 + j];
    for (int i = 0; i < kHid; ++i) z = fmaf(w[oW2 + j * kHid + i], a1[i], z);
    const float a = z * sigm(z);
    if (act.z2) {
      act.z2[size_t(s) * kHid + j] = z;
      act.a2[size_t(s) * kHid + j] = a;
    }
    out = fmaf(w[oW3 + j], a, out);
  }
  act.out[s] = out;
}

// ---- training on the tensor cores
// One CTA of 512 threads per tile of 128 samples. Sample s is accumulator row s; four threads share a
// sample (warps w, w + 4, w + 8, w + 12 read the same 32 tensor-memory lanes), each takes a quarter of
// the columns. Operands in shared memory are K-major, no swizzle, 8 x 16-byte core matrices
// (core_offset); a K16 step of an operand with g groups of 8 along K starts 256 bytes further, its K
// groups are 128 bytes apart and its row groups g x 128 bytes apart.
//   xa  [128 x 16]   features (12, then zeros)           layer 1:  Z1 = X W1^T       M128 N64 K16
//   a1  [128 x 64]   SiLU(Z1 + b1)                        layer 2:  Z2 = A1 W2^T      M128 N64 K64
//   dz2 [128 x 64]   dL/dZ2 = dout w3 SiLU'(Z2 + b2)      back:     dA1 = dZ2 W2      M128 N64 K64
//   ag  [128 x 128]  rows 0..63: dZ2^T, rows 64..127: dZ1^T (dZ1 = dA1 SiLU'(Z1 + b1)); K = samples
//   bg  [96 x 128]   rows 0..63: A1^T, 64..79: X^T, 80: ones, 81..95: zeros
//   gradients:       G = ag bg^T                          M128 N96 K128
//     G[j][i] = dW2[j][i] (j, i < 64), G[64 + j][64 + q] = dW1[j][q], G[r][80] = db2 / db1.
// w3 and b3 get their gradients on the CUDA cores (FP32, a fixed-order sum over the tile).
// BF16 operands are rounded to nearest even from the FP32 values; the products are exact and
// summed in FP32.
//
// A step's work is tiny (8 tiles at batch 1024) and serial: it is bound by latencies and by the issue
// slots of the SMs that hold its tiles, not by the tensor cores. With one thread a sample and two
// launches a step it took 42 us; four threads a sample, padded sums that overlap the last product, and
// many steps a launch brought it to 17 us; the CTAs of a batch as one cluster, partial gradients in the
// product's order, BF16 pairs rounded and stored by the word, and no block-wide vote after each product
// to 12 us (two epochs of 380,000 records: 31.7 -> 12.9 -> 8.8 ms, the same bits). What is left: the
// SiLU's exponentials and divisions 6 of 22 kcycles, four products' round trips 3.4, two barriers 2.8.
constexpr int kTile = 128;
constexpr int kTrainThreads = 512;
constexpr uint32_t kIdescN64 = umma_idesc_bf16(128, 64);
constexpr uint32_t kIdescN96 = umma_idesc_bf16(128, 96);
static_assert(kIdescN64 == kIdescM128N64, "instruction descriptor");

struct __align__(1024) TrainSmem {
  uint8_t ag[128 * 128 * 2];  // 32 KB
  uint8_t bg[96 * 128 * 2];   // 24 KB
  uint8_t a1[128 * 64 * 2];   // 16 KB
  uint8_t dz2[128 * 64 * 2];  // 16 KB
  uint8_t w2[64 * 64 * 2];    // W2 (N = outputs j, K = inputs i)
  uint8_t w2t[64 * 64 * 2];   // W2^T (N = i, K = j)
  uint8_t xa[128 * 16 * 2];
  uint8_t w1[64 * 16 * 2];    // W1 (N = j, K = inputs, 12..15 zero)
  float xs[kTile * kMlpRecord];  // a tile's records (the steps kernel)
  float red[66][kTile + 1];   // per-sample a2[j], then dout a2[j] (j < 64), dout, squared residual; padded
  alignas(16) float b1[64];
  float b2[64], w3[64], b3;
  uint64_t mbar;
  uint32_t tmem_base, flag;
};

__device__ __forceinline__ void st_bf16(uint8_t* base, uint32_t off, float v) {
  *reinterpret_cast<uint16_t*>(base + off) = uint16_t(bf16_rne(v));
}

// 16 / 8 consecutive FP32 accumulator columns of this thread's row of tensor memory.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = __uint_as_float(r[k]);
}

// mbar_wait that polls without sleeping first: a product of this size takes a few hundred cycles.
__device__ __forceinline__ bool mbar_poll(uint64_t* mbar, uint32_t parity) {
  for (uint32_t it = 0; it < 4096; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(smem_addr(mbar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return mbar_wait(mbar, parity);
}

// Issues `nk` K16 steps of D = A B^T into tensor memory (thread 0) after every thread's operand stores,
// and commits them to the mbarrier.
__device__ void tc_issue(TrainSmem& sm, uint32_t tmem, const uint8_t* a, uint32_t a_sbo, const uint8_t* b,
                         uint32_t b_sbo, int nk, uint32_t idesc) {
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) {
    tc_fence_after();
    for (int k = 0; k < nk; ++k)
      tc_mma_id(tmem, umma_desc(smem_addr(a) + k * 256, 128, a_sbo), umma_desc(smem_addr(b) + k * 256, 128, b_sbo),
                idesc, k > 0 ? 1u : 0u);
    tc_commit(&sm.mbar);
  }
}
// Waits for it (every thread, bounded); false if this thread's wait ran out. The tile goes on regardless
// (its values are then discarded), so that every thread passes the same barriers.
__device__ __forceinline__ bool tc_await(TrainSmem& sm, uint32_t& phase) {
  const bool done = mbar_poll(&sm.mbar, phase);
  phase ^= 1u;
  __syncwarp();
  tc_fence_after();
  return done;
}

// Two FP32 values rounded to BF16 (nearest even), lo in the low half.
__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

// A value of row `r` and of row r + 1 at K index `k`, with k + 1 at the next lane for even lanes, into an
// operand with `kgroups` K groups: lane pairs exchange one value each, so that a lane stores one 32-bit
// word of one row.
__device__ __forceinline__ void st_bf16_pair(uint8_t* base, int r, int k, int kgroups, float v0, float v1) {
  const uint32_t odd = threadIdx.x & 1u, b = bf16x2(v0, v1);
  const uint32_t got = __shfl_xor_sync(0xffffffffu, b, 1);
  // even: own v0, the neighbour's v0; odd: the neighbour's v1, own v1
  const uint32_t word = odd ? __byte_perm(got, b, 0x7632) : __byte_perm(b, got, 0x5410);
  *reinterpret_cast<uint32_t*>(base + core_offset(r + int(odd), k & ~1, kgroups)) = word;
}

// 8 consecutive K values of one row of an operand (one 16-byte store)
__device__ __forceinline__ void st_bf16x8(uint8_t* at, const float* v) {
  *reinterpret_cast<uint4*>(at) =
      make_uint4(bf16x2(v[0], v[1]), bf16x2(v[2], v[3]), bf16x2(v[4], v[5]), bf16x2(v[6], v[7]));
}

// One CTA's set-up: mbarrier, 128 accumulator columns (each stage writes from column 0), the operands'
// constant rows. Returns the tensor-memory base.
__device__ uint32_t train_setup(TrainSmem& sm) {
  const int tid = threadIdx.x;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&sm.mbar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(smem_addr(&sm.tmem_base))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int e = tid; e < 16 * kTile; e += kTrainThreads)  // the ones (bias gradients) and the zeros below
    st_bf16(sm.bg, core_offset(80 + e / kTile, e % kTile, 16), e < kTile ? 1.0f : 0.0f);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  return sm.tmem_base;
}
__device__ void train_teardown(uint32_t tmem) {
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(tmem) : "memory");
  }
}

// Partial gradients, and the parameters while many steps train them, are kept in the order in which the
// gradient product leaves them (lane = row of G): W2 by columns (i 64 + j), then W1 by columns, b2, b1,
// w3, b3. A warp then stores and loads whole lines; row by row the stores of one step took 3 us.
constexpr int gW1 = 4096, gB2 = 4864, gB1 = 4928;
__host__ __device__ __forceinline__ int g_index(int k) {  // place of parameter k
  if (k < oB1) return gW1 + (k % kIn) * 64 + k / kIn;
  if (k < oW2) return gB1 + (k - oB1);
  if (k < oB2) return ((k - oW2) & 63) * 64 + ((k - oW2) >> 6);
  if (k < oW3) return gB2 + (k - oB2);
  return k;
}
__device__ __forceinline__ int g_param(int e) {  // parameter at place e
  if (e < gW1) return oW2 + (e & 63) * 64 + (e >> 6);
  if (e < gB2) return oW1 + (e & 63) * kIn + ((e - gW1) >> 6);
  if (e < gB1) return oB2 + (e - gB2);
  if (e < oW3) return oB1 + (e - gB1);
  return e;
}

// Parameters (in that order, kG, or as the caller keeps them) as BF16 operands (both orientations of
// W2), biases and w3 in FP32. The loads skip L1 (the parameters change between the steps of one launch)
// and are all issued before the first store.
template <bool kG>
__device__ void train_weights(TrainSmem& sm, const float* __restrict__ p) {
  const int tid = threadIdx.x, j = tid & 63, ig = tid >> 6;  // row j, columns 8 ig .. (W2) and 2 ig .. (W1)
  const auto at = [&](int k) { return __ldcg(p + (kG ? g_index(k) : k)); };
  float w2[8], w1[2], b = 0.0f;
#pragma unroll
  for (int q = 0; q < 8; ++q) w2[q] = at(oW2 + j * 64 + ig * 8 + q);
#pragma unroll
  for (int q = 0; q < 2; ++q) w1[q] = ig * 2 + q < kIn ? at(oW1 + j * kIn + ig * 2 + q) : 0.0f;
  if (tid < 64)
    b = at(oB1 + tid);
  else if (tid < 128)
    b = at(oB2 + tid - 64);
  else if (tid <= 192)
    b = at(oW3 + tid - 128);  // w3, then b3
  st_bf16x8(sm.w2 + core_offset(j, ig * 8, 8), w2);
#pragma unroll
  for (int q = 0; q < 8; q += 2) st_bf16_pair(sm.w2t, ig * 8 + q, j, 8, w2[q], w2[q + 1]);
  *reinterpret_cast<uint32_t*>(sm.w1 + core_offset(j, ig * 2, 2)) = bf16x2(w1[0], w1[1]);
  if (tid < 64)
    sm.b1[tid] = b;
  else if (tid < 128)
    sm.b2[tid - 64] = b;
  else if (tid < 192)
    sm.w3[tid - 128] = b;
  else if (tid == 192)
    sm.b3 = b;
}
static_assert(kTrainThreads == 512, "eight threads a row of W2");

// This thread's quarter of its sample's inputs (4 of 16, the last four zero) and the label.
struct TrainInput {
  float x[4], y;
};
__device__ __forceinline__ TrainInput train_input(const float* __restrict__ x, int x_stride,
                                                  const float* __restrict__ y, int y_stride, uint32_t n) {
  const uint32_t s = blockIdx.x * kTile + (threadIdx.x & (kTile - 1)), cg = threadIdx.x >> 7;
  TrainInput in{{0.0f, 0.0f, 0.0f, 0.0f}, 0.0f};
  if (s < n) {
    if (cg < kIn / 4)
      for (int i = 0; i < 4; ++i) in.x[i] = x[size_t(s) * x_stride + cg * 4 + i];
    in.y = y[size_t(s) * y_stride];
  }
  return in;
}

// The same from records (inputs, label), whose tile is contiguous: whole lines into registers (ahead of
// time), then by way of shared memory; thread by thread the strided loads of a step took 1.5 us.
constexpr int kTileLoads = (kTile * kMlpRecord + kTrainThreads - 1) / kTrainThreads;
__device__ __forceinline__ void tile_records(const float* __restrict__ rec, uint32_t n, float v[kTileLoads]) {
  const uint32_t from = blockIdx.x * kTile * kMlpRecord;
#pragma unroll
  for (int q = 0; q < kTileLoads; ++q) {
    const uint32_t e = threadIdx.x + q * kTrainThreads;
    v[q] = e < kTile * kMlpRecord && from + e < n * kMlpRecord ? rec[from + e] : 0.0f;
  }
}
__device__ __forceinline__ TrainInput tile_input(TrainSmem& sm, const float v[kTileLoads]) {
  const uint32_t s = threadIdx.x & (kTile - 1), cg = threadIdx.x >> 7;
#pragma unroll
  for (int q = 0; q < kTileLoads; ++q) {
    const uint32_t e = threadIdx.x + q * kTrainThreads;
    if (e < kTile * kMlpRecord) sm.xs[e] = v[q];
  }
  __syncthreads();
  TrainInput in;
#pragma unroll
  for (int i = 0; i < 4; ++i) in.x[i] = cg < kIn / 4 ? sm.xs[s * kMlpRecord + cg * 4 + i] : 0.0f;
  in.y = sm.xs[s * kMlpRecord + 12];
  return in;
}

// Forward and backward pass of one tile; the CTA's partial gradient (TKF_MLP_PARAMS floats) and
// its sum of squared residuals go to g and *sq. `inv_n`: 1 / batch size (dL/dout = 2 r / n). Returns
// false (nothing written) if any thread's wait for the tensor cores ran out.
__device__ bool train_tile(TrainSmem& sm, uint32_t tmem, uint32_t& phase, const TrainInput& in, uint32_t n, float inv_n,
                           float* __restrict__ g, float* __restrict__ sq) {
  const int tid = threadIdx.x, s = tid & (kTile - 1), cg = tid >> 7, c0 = cg * 16;
  const bool live = blockIdx.x * kTile + s < n;
  const uint32_t t_row = tmem + (uint32_t(s & ~31) << 16);  // this warp's 32 lanes
  for (int i = 0; i < 4; i += 2) {
    *reinterpret_cast<uint32_t*>(sm.xa + core_offset(s, cg * 4 + i, 2)) = bf16x2(in.x[i], in.x[i + 1]);
    st_bf16_pair(sm.bg, 64 + cg * 4 + i, s, 16, in.x[i], in.x[i + 1]);  // X^T
  }
  bool ok = true;
  float v[16], d1[16], z2[16], sg2[16];  // d1: SiLU'(Z1 + b1)
  // layer 1
  tc_issue(sm, tmem, sm.xa, 256, sm.w1, 256, 1, kIdescN64);
  ok = tc_await(sm, phase) && ok;
  tmem_ld16(t_row + uint32_t(c0), v);
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float z = v[k] + sm.b1[c0 + k], sg = sigm(z);
    v[k] = z * sg;
    d1[k] = sg * (1.0f + z * (1.0f - sg));
  }
#pragma unroll
  for (int k = 0; k < 16; k += 8) st_bf16x8(sm.a1 + core_offset(s, c0 + k, 8), v + k);
#pragma unroll
  for (int k = 0; k < 16; k += 2) st_bf16_pair(sm.bg, c0 + k, s, 16, v[k], v[k + 1]);  // A1^T
  // layer 2
  tc_issue(sm, tmem, sm.a1, 1024, sm.w2, 1024, 4, kIdescN64);
  ok = tc_await(sm, phase) && ok;
  tmem_ld16(t_row + uint32_t(c0), v);
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    z2[k] = v[k] + sm.b2[c0 + k];
    sg2[k] = sigm(z2[k]);
    v[k] = z2[k] * sg2[k];
    sm.red[c0 + k][s] = v[k];
  }
  __syncthreads();
  if (cg == 0) {  // the output layer, in column order
    float out = sm.b3;
#pragma unroll 16
    for (int j = 0; j < 64; ++j) out = fmaf(sm.w3[j], sm.red[j][s], out);
    const float r = live ? out - in.y : 0.0f;
    sm.red[64][s] = 2.0f * r * inv_n;
    sm.red[65][s] = r * r;
  }
  __syncthreads();
  const float dout = sm.red[64][s];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    sm.red[c0 + k][s] = dout * v[k];
    const float sg = sg2[k];
    v[k] = dout * sm.w3[c0 + k] * (sg * (1.0f + z2[k] * (1.0f - sg)));
  }
#pragma unroll
  for (int k = 0; k < 16; k += 8) st_bf16x8(sm.dz2 + core_offset(s, c0 + k, 8), v + k);
#pragma unroll
  for (int k = 0; k < 16; k += 2) st_bf16_pair(sm.ag, c0 + k, s, 16, v[k], v[k + 1]);  // dZ2^T
  // backpropagation through layer 2
  tc_issue(sm, tmem, sm.dz2, 1024, sm.w2t, 1024, 4, kIdescN64);
  ok = tc_await(sm, phase) && ok;
  tmem_ld16(t_row + uint32_t(c0), v);
#pragma unroll
  for (int k = 0; k < 16; k += 2) st_bf16_pair(sm.ag, 64 + c0 + k, s, 16, v[k] * d1[k], v[k + 1] * d1[k + 1]);  // dZ1^T
  // weight and bias gradients of both layers: G = ag bg^T over the tile's samples
  tc_issue(sm, tmem, sm.ag, 2048, sm.bg, 2048, 8, kIdescN96);
  // meanwhile w3, b3 and the squared residuals: sums over the tile in sample order (warps 1 to 3)
  float acc = 0.0f;
  const int row = tid - 32;
  if (row >= 0 && row < 66) {
#pragma unroll 16
    for (int t = 0; t < kTile; ++t) acc += sm.red[row][t];
  }
  ok = tc_await(sm, phase) && ok;
  ok = __syncthreads_or(!ok) == 0;
  if (!ok) return false;
  if (row >= 0 && row < 64)
    g[oW3 + row] = acc;
  else if (row == 64)
    g[oB3] = acc;
  else if (row == 65)
    *sq = acc;
  // row s of G, columns 24 cg ..: dW2 row s and db2 (s < 64), or dW1 row s - 64 and db1
  float w[24];
  tmem_ld16(t_row + uint32_t(cg * 24), w);
  tmem_ld8(t_row + uint32_t(cg * 24 + 16), w + 16);
#pragma unroll
  for (int k = 0; k < 24; ++k) {
    const int col = cg * 24 + k;
    if (s < 64) {
      if (col < 64) g[col * 64 + s] = w[k];
      if (col == 80) g[gB2 + s] = w[k];
    } else {
      if (col >= 64 && col < 64 + kIn) g[gW1 + (col - 64) * 64 + s - 64] = w[k];
      if (col == 80) g[gB1 + s - 64] = w[k];
    }
  }
  return ok;
}

__device__ __forceinline__ TrainSmem& train_smem(uint8_t* raw) {
  // the operands at a 1024-byte boundary (the launch reserves the slack)
  return *reinterpret_cast<TrainSmem*>(raw + ((1024u - (smem_addr(raw) & 1023u)) & 1023u));
}

// A wait that ran out: NaN partials (and so a NaN loss), after a bounded time for a product in flight.
__device__ void train_failed(TrainSmem& sm, uint32_t phase, float* __restrict__ g, float* __restrict__ sq) {
  const float nan = __int_as_float(0x7fc00000);
  for (int k = threadIdx.x; k < kMlpParams; k += kTrainThreads) g[k] = nan;
  if (threadIdx.x == 0) *sq = nan;
  mbar_wait(&sm.mbar, phase ^ 1u);
}

// One forward and backward pass over a batch: partial gradients part[CTA], squared residuals sq[CTA].
__global__ void __launch_bounds__(kTrainThreads, 1)
    mlp_train_tc_kernel(const float* __restrict__ p, const float* __restrict__ x, int x_stride,
                        const float* __restrict__ y, int y_stride, uint32_t n, float inv_n, float* __restrict__ part,
                        float* __restrict__ sq) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  TrainSmem& sm = train_smem(smem_raw);
  const uint32_t tmem = train_setup(sm);
  uint32_t phase = 0;
  train_weights<false>(sm, p);
  const TrainInput in = train_input(x, x_stride, y, y_stride, n);
  float* g = part + size_t(blockIdx.x) * kMlpParams;
  if (!train_tile(sm, tmem, phase, in, n, inv_n, g, sq + blockIdx.x)) train_failed(sm, phase, g, sq + blockIdx.x);
  train_teardown(tmem);
}

// One Adam step of a parameter (Kingma & Ba 2015); c1, c2: the bias corrections 1 - beta^t.
__device__ __forceinline__ void adam(float gk, float& p, float& m, float& v, float lr, float beta1, float beta2, float eps,
                                     float c1, float c2) {
  const float mk = beta1 * m + (1.0f - beta1) * gk;
  const float vk = beta2 * v + (1.0f - beta2) * gk * gk;
  m = mk;
  v = vk;
  p -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

// Sum of the CTAs' partial gradients (in CTA order), written to grad, then (when m is not
// null) one Adam step of the parameters; thread 0 also writes the batch's mean squared residual
// to *loss and adds it, weighted, to *epoch_acc.
__global__ void __launch_bounds__(256) mlp_reduce_adam_kernel(const float* __restrict__ part,
                                                              const float* __restrict__ sq, uint32_t n_cta, float inv_n,
                                                              float* __restrict__ grad, float* __restrict__ p,
                                                              float* __restrict__ m, float* __restrict__ v, float lr,
                                                              float beta1, float beta2, float eps, float c1, float c2,
                                                              float* __restrict__ loss, float* __restrict__ epoch_acc,
                                                              float inv_batches) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k == 0) {
    float l = 0.0f;
    for (uint32_t c = 0; c < n_cta; ++c) l += sq[c];
    l *= inv_n;
    if (loss) *loss = l;
    if (epoch_acc) *epoch_acc += l * inv_batches;
  }
  if (k >= kMlpParams) return;
  float gk = 0.0f;
  for (uint32_t c = 0; c < n_cta; ++c) gk += part[size_t(c) * kMlpParams + g_index(k)];
  if (grad) grad[k] = gk;
  if (!m) return;
  adam(gk, p[k], m[k], v[k], lr, beta1, beta2, eps, c1, c2);
}

// ---- many training steps in one launch
// The CTAs of a batch run together (a cooperative launch) and meet twice a step: after writing their
// partial gradients, and after each has summed its slice of the parameters over the CTAs (in CTA
// order, as mlp_reduce_adam_kernel does) and taken their Adam step. The moments stay in registers for
// the launch, the next batch's inputs are loaded before the first meeting. The bias corrections 1 -
// beta^t come with the launch (kTrainSteps of them), computed on the host.
constexpr int kTrainSteps = 256;
constexpr int kSliceMax = (kMlpParams + kTrainThreads - 1) / kTrainThreads;  // parameters a thread, one CTA

struct TrainSteps {
  const float* records;  // [batches][batch][TKF_MLP_RECORD]
  uint32_t batch, batches, first, count;  // the launch's steps: first .. first + count - 1 (over all epochs)
  float *p, *m, *v, *part, *sq, *epoch_loss;
  float* q;        // the parameters in the gradient's order, for the launch
  uint32_t* meet;  // arrivals of the grid barrier, zeroed before the launch
  uint32_t meet_polls;  // limit of the counter's wait
  float lr, beta1, beta2, eps;
  float2 c[kTrainSteps];
};

// Every CTA of the launch arrives, then waits for the others: by the hardware barrier where the CTAs are
// one cluster, else by a counter (bounded: false if the wait ran out).
template <bool kCluster>
__device__ bool train_meet(TrainSmem& sm, uint32_t* meet, uint32_t target, uint32_t polls) {
  if constexpr (kCluster) {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    return true;
  } else {
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      atomicAdd(meet, 1u);
      uint32_t seen = 0, it = 0;
      for (; it < polls; ++it) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(meet) : "memory");
        if (int32_t(seen - target) >= 0) break;
        if (it > 4096) __nanosleep(100);
      }
      sm.flag = it < polls;
      __threadfence();
    }
    __syncthreads();
    return sm.flag != 0;
  }
}

template <bool kCluster>
__global__ void __launch_bounds__(kTrainThreads, 1) mlp_train_steps_kernel(const __grid_constant__ TrainSteps a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  TrainSmem& sm = train_smem(smem_raw);
  const uint32_t tmem = train_setup(sm);
  // this CTA's slice of the parameters, in the gradient's order
  const uint32_t per = (kMlpParams + gridDim.x - 1) / gridDim.x, e0 = blockIdx.x * per;
  const uint32_t e1 = min(e0 + per, uint32_t(kMlpParams));
  float pk[kSliceMax], mk[kSliceMax], vk[kSliceMax];
#pragma unroll
  for (int q = 0; q < kSliceMax; ++q) {
    const uint32_t e = e0 + threadIdx.x + q * kTrainThreads;
    const int k = e < e1 ? g_param(int(e)) : 0;
    pk[q] = a.p[k];
    mk[q] = a.m[k];
    vk[q] = a.v[k];
    if (e < e1) a.q[e] = pk[q];
  }
  const float inv_n = 1.0f / float(a.batch), inv_batches = 1.0f / float(a.batches);
  float* g = a.part + size_t(blockIdx.x) * kMlpParams;
  uint32_t phase = 0, met = 0;
  bool ok = true;
  float rec[kTileLoads];
  const auto load = [&](uint32_t step) {
    tile_records(a.records + size_t(step % a.batches) * a.batch * kMlpRecord, a.batch, rec);
  };
  load(a.first);
  bool together = train_meet<kCluster>(sm, a.meet, (met += gridDim.x), a.meet_polls);  // every slice of q is there
  uint32_t i = 0, epoch = a.first / a.batches;  // the current epoch and its loss so far (one thread's)
  float sum = __ldcg(a.epoch_loss + epoch);
  for (; i < a.count && together; ++i) {
    train_weights<true>(sm, a.q);
    const TrainInput in = tile_input(sm, rec);
    if (ok) ok = train_tile(sm, tmem, phase, in, a.batch, inv_n, g, a.sq + blockIdx.x);
    if (!ok) train_failed(sm, phase, g, a.sq + blockIdx.x);
    if (i + 1 < a.count) load(a.first + i + 1);
    together = train_meet<kCluster>(sm, a.meet, (met += gridDim.x), a.meet_polls);
    if (!together) break;
    if (blockIdx.x == 0 && threadIdx.x == kTrainThreads - 1) {
      float l = 0.0f;
      for (uint32_t c = 0; c < gridDim.x; ++c) l += __ldcg(a.sq + c);
      l *= inv_n;
      if ((a.first + i) / a.batches != epoch) {
        ++epoch;
        sum = 0.0f;
      }
      // stored by comparison: not over the NaN that a CTA left whose meeting failed
      const float next = fmaf(l, inv_batches, sum);
      atomicCAS(reinterpret_cast<unsigned*>(a.epoch_loss + epoch), __float_as_uint(sum), __float_as_uint(next));
      sum = next;
    }
    const float2 c = a.c[i];
    // every element's sum runs over the CTAs in order; the loads of a thread's elements overlap
    const auto reduce = [&](auto n_elements) {
      constexpr int kN = decltype(n_elements)::value;
      float gk[kN];
#pragma unroll
      for (int q = 0; q < kN; ++q) gk[q] = 0.0f;
      const float* at = a.part + e0 + threadIdx.x;
#pragma unroll 8
      for (uint32_t cta = 0; cta < gridDim.x; ++cta, at += kMlpParams) {
#pragma unroll
        for (int q = 0; q < kN; ++q)
          if (e0 + threadIdx.x + q * kTrainThreads < e1) gk[q] += __ldcg(at + q * kTrainThreads);
      }
#pragma unroll
      for (int q = 0; q < kN; ++q) {
        const uint32_t e = e0 + threadIdx.x + q * kTrainThreads;
        if (e < e1) {
          adam(gk[q], pk[q], mk[q], vk[q], a.lr, a.beta1, a.beta2, a.eps, c.x, c.y);
          a.q[e] = pk[q];
        }
      }
    };
    if (per <= 2 * kTrainThreads)
      reduce(std::integral_constant<int, 2>{});
    else
      reduce(std::integral_constant<int, kSliceMax>{});
    together = train_meet<kCluster>(sm, a.meet, (met += gridDim.x), a.meet_polls);
  }
#pragma unroll
  for (int q = 0; q < kSliceMax; ++q) {
    const uint32_t e = e0 + threadIdx.x + q * kTrainThreads;
    if (e < e1) {
      const int k = g_param(int(e));
      a.m[k] = mk[q];
      a.v[k] = vk[q];
      a.p[k] = together ? pk[q] : __int_as_float(0x7fc00000);
    }
  }
  // a meeting that did not come about: with the parameters the losses of the epochs that it cut short are NaN
  if (!together && threadIdx.x == 0)
    for (uint32_t ep = (a.first + min(i, a.count - 1)) / a.batches; ep <= (a.first + a.count - 1) / a.batches; ++ep)
      atomicExch(a.epoch_loss + ep, __int_as_float(0x7fc00000));
  train_teardown(tmem);
}

// ---- initialisation: W ~ U(-1/sqrt(fan_in), 1/sqrt(fan_in)) from SplitMix64 of (seed, index), b = 0
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

__global__ void __launch_bounds__(256) mlp_init_kernel(float* __restrict__ p, uint64_t seed) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= kMlpParams) return;
  const bool weight = k < oB1 || (k >= oW2 && k < oB2) || (k >= oW3 && k < oB3);
  if (!weight) {
    p[k] = 0.0f;
    return;
  }
  const float fan_in = k < oB1 ? float(kIn) : float(kHid);
  const uint64_t r = splitmix64(seed * 0x100000001B3ull + uint64_t(k));
  const float u = float(r >> 40) * (1.0f / 16777216.0f);  // [0, 1), 24 bits
  p[k] = (2.0f * u - 1.0f) * rsqrtf(fan_in);
}

// ---- calibration: residual = label - output, shifted bias b3 += quantile of the residuals
// order-preserving map of an FP32 value to an unsigned key, and back
__device__ __forceinline__ uint32_t order_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float from_order_key(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__global__ void __launch_bounds__(256) residual_keys_kernel(const float* __restrict__ rec, uint32_t n,
                                                            const float* __restrict__ out, uint32_t* __restrict__ keys) {
  const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < n) keys[s] = order_key(rec[size_t(s) * kMlpRecord + 12] - out[s]);
}

// The k0-th and k1-th smallest keys (0-based) by a radix select, 8 bits a pass from the top:
// each pass counts the keys that share the digits chosen so far by their next digit and keeps
// the bucket that holds the wanted rank. One block; every loop is bounded by n or 256.
__global__ void __launch_bounds__(1024) select_kernel(const uint32_t* __restrict__ keys, uint32_t n, uint32_t k0,
                                                      uint32_t k1, uint32_t* __restrict__ sel) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t s_prefix, s_rank;
  for (int which = 0; which < 2; ++which) {
    uint32_t prefix = 0, mask = 0, rank = which ? k1 : k0;
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      for (int b = threadIdx.x; b < 256; b += blockDim.x) hist[b] = 0;
      __syncthreads();
      for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
        const uint32_t key = keys[i];
        if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        uint32_t acc = 0;
        int d = 0;
        for (; d < 255; ++d) {
          if (acc + hist[d] > rank) break;
          acc += hist[d];
        }
        s_prefix = prefix | (uint32_t(d) << shift);
        s_rank = rank - acc;
      }
      __syncthreads();
      prefix = s_prefix;
      rank = s_rank;
      mask |= 255u << shift;
      __syncthreads();
    }
    if (threadIdx.x == 0) sel[which] = prefix;
    __syncthreads();
  }
}

// The quantile by linear interpolation between the two order statistics around
// position q (n - 1) (FP64), added to the output bias (FP64, rounded to FP32).
__global__ void shift_bias_kernel(float* __restrict__ p, const uint32_t* __restrict__ sel, double frac,
                                  double* __restrict__ shift) {
  const double v0 = from_order_key(sel[0]), v1 = from_order_key(sel[1]);
  const double q = v0 + frac * (v1 - v0);
  p[oB3] = float(double(p[oB3]) + q);
  *shift = q;
}

// ---- BF16 weights: round to nearest even; a non-finite value sets *bad
__global__ void __launch_bounds__(256) round_bf16_kernel(const float* __restrict__ in, float* __restrict__ out,
                                                         uint32_t* __restrict__ bad) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= kMlpParams) return;
  const float x = in[k];
  if (!isfinite(x)) atomicOr(bad, 1u);
  const uint32_t u = __float_as_uint(x);
  out[k] = __uint_as_float((u + 0x7FFFu + ((u >> 16) & 1u)) & 0xFFFF0000u);
}

}  // namespace

cudaError_t mlp_init(float* params, uint64_t seed, cudaStream_t stream) {
  mlp_init_kernel<<<(kMlpParams + 255) / 256, 256, 0, stream>>>(params, seed);
  return cudaGetLastError();
}

size_t mlp_calibrate_scratch_bytes(uint32_t n) { return sizeof(float) * 2 * size_t(n) + 64; }

cudaError_t mlp_calibrate(float* params, const float* records, uint32_t n, double quantile, double* shift,
                          void* scratch, cudaStream_t stream) {
  float* out = static_cast<float*>(scratch);
  uint32_t* keys = reinterpret_cast<uint32_t*>(out + n);
  uint32_t* sel = keys + n;
  Act act{};
  act.out = out;
  const unsigned g = (n + 255) / 256;
  mlp_forward_kernel<<<(n + 127) / 128, 128, 0, stream>>>(params, records, kMlpRecord, n, act);
  residual_keys_kernel<<<g, 256, 0, stream>>>(records, n, out, keys);
  const double pos = quantile * double(n - 1);
  const uint32_t k0 = uint32_t(floor(pos));
  const uint32_t k1 = k0 + 1 < n ? k0 + 1 : k0;
  select_kernel<<<1, 1024, 0, stream>>>(keys, n, k0, k1, sel);
  shift_bias_kernel<<<1, 1, 0, stream>>>(params, sel, pos - double(k0), shift);
  return cudaGetLastError();
}

cudaError_t mlp_round_bf16(const float* in, float* out, uint32_t* bad, cudaStream_t stream) {
  round_bf16_kernel<<<(kMlpParams + 255) / 256, 256, 0, stream>>>(in, out, bad);
  return cudaGetLastError();
}

size_t mlp_train_scratch_bytes(uint32_t batch) {
  const size_t n_cta = (size_t(batch) + kTile - 1) / kTile;
  return sizeof(float) * (n_cta * (kMlpParams + 1) + 2 * kMlpParams + 1) + 256;
}

namespace {
// Partial gradients [n_cta][params], per-CTA squared residuals [n_cta], the summed gradient, the steps
// kernel's parameters and the arrivals of its grid barrier.
struct TrainScratch {
  float* part;
  float* sq;
  float* grad;
  float* q;
  uint32_t* meet;
};
TrainScratch carve_train(void* base, uint32_t batch) {
  const size_t n_cta = (size_t(batch) + kTile - 1) / kTile;
  float* f = static_cast<float*>(base);
  float* grad = f + n_cta * (kMlpParams + 1);
  return TrainScratch{f, f + n_cta * kMlpParams, grad, grad + kMlpParams,
                      reinterpret_cast<uint32_t*>(grad + 2 * kMlpParams)};
}

constexpr size_t kTrainSmemBytes = sizeof(TrainSmem) + 1024;  // + alignment slack
static_assert(kTrainSmemBytes <= 227 * 1024, "shared memory");

// How a batch's CTAs can run at the same time on this device, as the steps kernel needs (one an SM; the largest batch
// has 64): as one cluster (2, 4 or 8 CTAs: batches of 129 to 256, 385 to 512 and 897 to 1,024; its barrier takes a fifth of
// the counter's time) where the device says that it can place one, else as a cooperative launch, else not at all.
// A device partition without room for them trains step by step.
enum class Together { kNo, kCooperative, kCluster };

struct StepsConfig {
  cudaLaunchAttribute attr{};
  cudaLaunchConfig_t cfg{};
  StepsConfig(unsigned n_cta, Together how, cudaStream_t stream) {
    if (how == Together::kCluster) {
      attr.id = cudaLaunchAttributeClusterDimension;
      attr.val.clusterDim.x = n_cta;
      attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    } else {
      attr.id = cudaLaunchAttributeCooperative;
      attr.val.cooperative = 1;
    }
    cfg.gridDim = dim3(n_cta);
    cfg.blockDim = dim3(kTrainThreads);
    cfg.dynamicSmemBytes = kTrainSmemBytes;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
  }
  StepsConfig(const StepsConfig&) = delete;  // cfg points to attr
};

Together train_together(unsigned n_cta) {
  int dev = 0, sms = 0, coop = 0, per_sm = 0, clusters = 0;
  const StepsConfig cluster(n_cta, Together::kCluster, nullptr);
  if (cudaGetDevice(&dev) == cudaSuccess && (n_cta == 2 || n_cta == 4 || n_cta == 8) &&
      cudaFuncSetAttribute(mlp_train_steps_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           int(kTrainSmemBytes)) == cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&clusters, mlp_train_steps_kernel<true>, &cluster.cfg) == cudaSuccess && clusters > 0)
    return Together::kCluster;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
      cudaFuncSetAttribute(mlp_train_steps_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           int(kTrainSmemBytes)) == cudaSuccess &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mlp_train_steps_kernel<false>, kTrainThreads,
                                                    kTrainSmemBytes) == cudaSuccess &&
      n_cta <= unsigned(sms) * unsigned(per_sm))
    return Together::kCooperative;
  cudaGetLastError();
  return Together::kNo;
}

// Launch errors that say that the CTAs do not fit together here (a process limited to fewer SMs than the device has,
// say); nothing was enqueued.
bool does_not_fit(cudaError_t e) {
  return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources ||
         e == cudaErrorInvalidConfiguration || e == cudaErrorInvalidClusterSize;
}

cudaError_t train_tile_launch(const float* params, const float* x, int x_stride, const float* y, int y_stride,
                              uint32_t n, const TrainScratch& sc, cudaStream_t stream) {
  cudaError_t e = cudaFuncSetAttribute(mlp_train_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(kTrainSmemBytes));
  if (e != cudaSuccess) return e;
  const unsigned n_cta = (n + kTile - 1) / kTile;
  mlp_train_tc_kernel<<<n_cta, kTrainThreads, kTrainSmemBytes, stream>>>(params, x, x_stride, y, y_stride, n, 1.0f / float(n), sc.part,
                                                      sc.sq);
  return cudaGetLastError();
}
}  // namespace

cudaError_t mlp_loss_grad(const float* params, const float* x, int x_stride, const float* y, int y_stride,
                          uint32_t n, float* grad, float* loss, void* scratch, cudaStream_t stream) {
  const TrainScratch sc = carve_train(scratch, n);
  cudaError_t e = train_tile_launch(params, x, x_stride, y, y_stride, n, sc, stream);
  if (e != cudaSuccess) return e;
  const unsigned n_cta = (n + kTile - 1) / kTile;
  mlp_reduce_adam_kernel<<<(kMlpParams + 255) / 256, 256, 0, stream>>>(
      sc.part, sc.sq, n_cta, 1.0f / float(n), grad, nullptr, nullptr, nullptr, 0.0f, 0.0f, 0.0f, 0.0f, 1.0f, 1.0f, loss,
      nullptr, 0.0f);
  return cudaGetLastError();
}

cudaError_t mlp_train(const float* records, uint32_t n, uint32_t batch, uint32_t epochs, float lr, float beta1,
                      float beta2, float eps, float* params, float* moments, uint32_t* adam_t, float* epoch_loss,
                      void* scratch, cudaStream_t stream, uint32_t meet_polls) {
  const TrainScratch sc = carve_train(scratch, batch);
  const uint32_t nb = n / batch;
  const unsigned n_cta = (batch + kTile - 1) / kTile;
  cudaError_t e = cudaMemsetAsync(epoch_loss, 0, sizeof(float) * epochs, stream);
  if (e != cudaSuccess) return e;
  const uint64_t steps = uint64_t(epochs) * nb;
  const auto corrections = [&](uint32_t t) {
    return make_float2(1.0f - powf(beta1, float(t)), 1.0f - powf(beta2, float(t)));
  };
  uint64_t done = 0;
  Together how = steps < (uint64_t(1) << 32) ? train_together(n_cta) : Together::kNo;
  if (how != Together::kNo) {  // many steps a launch
    TrainSteps a{};
    a.records = records;
    a.batch = batch;
    a.batches = nb;
    a.p = params;
    a.m = moments;
    a.v = moments + kMlpParams;
    a.part = sc.part;
    a.sq = sc.sq;
    a.epoch_loss = epoch_loss;
    a.q = sc.q;
    a.meet = sc.meet;
    a.meet_polls = meet_polls;
    a.lr = lr;
    a.beta1 = beta1;
    a.beta2 = beta2;
    a.eps = eps;
    while (done < steps) {
      a.first = uint32_t(done);
      a.count = uint32_t(steps - done < uint64_t(kTrainSteps) ? steps - done : uint64_t(kTrainSteps));
      for (uint32_t i = 0; i < a.count; ++i) a.c[i] = corrections(*adam_t + i + 1);
      if ((e = cudaMemsetAsync(sc.meet, 0, sizeof(uint32_t), stream)) != cudaSuccess) return e;
      const StepsConfig c(n_cta, how, stream);
      e = how == Together::kCluster ? cudaLaunchKernelEx(&c.cfg, mlp_train_steps_kernel<true>, a)
                                    : cudaLaunchKernelEx(&c.cfg, mlp_train_steps_kernel<false>, a);
      if (does_not_fit(e)) {
        cudaGetLastError();
        break;
      }
      if (e != cudaSuccess) return e;
      *adam_t += a.count;
      done += a.count;
    }
  }
  for (; done < steps; ++done) {  // one step in two launches
    const float* rec = records + size_t(done % nb) * batch * kMlpRecord;
    e = train_tile_launch(params, rec, kMlpRecord, rec + 12, kMlpRecord, batch, sc, stream);
    if (e != cudaSuccess) return e;
    const float2 c = corrections(*adam_t + 1);
    mlp_reduce_adam_kernel<<<(kMlpParams + 255) / 256, 256, 0, stream>>>(
        sc.part, sc.sq, n_cta, 1.0f / float(batch), sc.grad, params, moments, moments + kMlpParams, lr, beta1, beta2,
        eps, c.x, c.y, nullptr, epoch_loss + done / nb, 1.0f / float(nb));
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    ++*adam_t;
  }
  return cudaSuccess;
}


cudaError_t mlp_forward(const float* params, const float* x, uint32_t n, float* out, cudaStream_t stream) {
  Act act{};
  act.out = out;
  mlp_forward_kernel<<<(n + 127) / 128, 128, 0, stream>>>(params, x, kIn, n, act);
  return cudaGetLastError();
}

}  // namespace tkf

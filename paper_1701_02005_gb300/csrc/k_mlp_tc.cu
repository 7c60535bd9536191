// The wall-model MLP on the tensor cores (no counterpart in the paper):
// tcgen05.mma (kind::f16, BF16 operands, FP32 accumulation in tensor memory)
// issued by one thread per CTA on operand tiles staged in shared memory.
//
//   forward      z[b][n]  = sum_k a(b, k) W[n][k] + bias[n],  a = x_n or GELU(z_prev)
//   data grad    da[b][k] = (sum_n dz[b][n] W[n][k]) GELU'(z_prev[b][k])
//   weight grad  dW[n][k] = sum_b dz[b][n] a(b, k),  dbias[n] = sum_b dz[b][n]
//
// Three kernels: k_mlp_infer_tc (all layers, outputs only), k_mlp_train_tc (all
// layers forward, the loss, and the data gradients back to the first layer, one
// 128-row tile at a time on chip) and k_mlp_wgrad_tc (the weight gradients from
// the BF16 operand tiles the second one leaves in global memory).
//
// A tile of R rows is kept as 8-row x 16-byte core matrices (canon below), and
// the same bytes serve every product it enters: read with K along the 16 bytes
// (K-major) the activations and weights of the forward pass, read with K along
// the 8 rows (MN-major, the descriptor's transpose bits) the weights of the data
// gradient and both operands of the weight gradient.  So no tile is ever
// transposed and the weights have one image.
//
// One CTA has 16 epilogue warps and one warp that issues the MMAs.  A layer's
// epilogue covers accumulator columns 0-63, then 64-127; each half is handed to
// the issuing warp through an mbarrier as soon as it is staged, so that the next
// layer's first K steps run under the second half of the epilogue.  Waits are
// bounded: on a timeout a kernel records PNP_ERR_TIMEOUT; in every case the threads
// that issued MMAs and copies wait (bounded) until these have completed before the
// kernel frees its tensor memory and returns (pnp_mlpflow.cuh).
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "pnp_common.cuh"
#include "pnp_mlpflow.cuh"
#include "pnp_wall.cuh"

namespace pnp {

namespace {

constexpr int kTcRows = 128;      // rows of D per tile (M of every MMA)
constexpr unsigned long long kTcWaitNs = 2000000000ull;

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// GELU(z) = z Phi(z)
__device__ __forceinline__ float gelu_erf(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }

// ... and its derivative, from the same erff
__device__ __forceinline__ void gelu_erf_d(float z, float& g, float& d) {
  const float e = 1.0f + erff(z * 0.70710678118654752f);
  g = 0.5f * z * e;
  d = 0.5f * e + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// Byte offset of element (r, k) of an R-row K-major tile: core matrix (r / 8,
// k / 8) of 8 rows x 16 bytes, K groups outermost, so the core matrices
// adjacent in K are R/8 * 128 bytes apart (the leading-dimension offset) and
// those adjacent in M/N 128 bytes (the stride-dimension offset).
__device__ __forceinline__ uint32_t canon(int r, int k, int R) {
  return (uint32_t)((((k >> 3) * (R >> 3) + (r >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1));
}

// Shared-memory matrix descriptor: start address, leading- and stride-
// dimension byte offsets (each >> 4), the fixed version bits 0b001 at 46-48,
// no base offset, no swizzle.  Leading: between core matrices adjacent in K;
// stride: between those adjacent in M or N (in both major orders).
__device__ __forceinline__ uint64_t sdesc(uint32_t start, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((start >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B BF16
// (bits 7-9 and 10-12 = 1), transpose bits of A and B (15, 16: 1 = MN-major),
// N / 8 at bits 17-22, M / 16 at bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool mnA, bool mnB) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((mnA ? 1u : 0u) << 15) | ((mnB ? 1u : 0u) << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_commit(unsigned long long* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(bar))
               : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// the generic-proxy writes of the staged tiles become visible to the tensor cores
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// one full warp; the address lands in *slot
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(slot)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// 16 consecutive FP32 accumulator columns of this thread's lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// 16 consecutive FP32 columns of this thread's lane, written back
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
  uint32_t r[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(v[i]);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
      "%14, %15};" ::"r"(r[0]),
      "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_init(unsigned long long* b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(b)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned long long* b, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, unsigned long long* b) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(saddr(dst)),
      "l"(src), "r"(bytes), "r"(saddr(b))
      : "memory");
}
__device__ __forceinline__ bool mbar_test(unsigned long long* b, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(saddr(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// bounded wait for the phase with this parity to complete
__device__ __forceinline__ bool mbar_wait_tc(unsigned long long* b, unsigned parity) {
  if (mbar_test(b, parity)) return true;
  const unsigned long long t0 = now_ns();
  for (int it = 0; it < (1 << 26); ++it) {
    if (mbar_test(b, parity)) return true;
    if ((it & 255) == 0 && now_ns() - t0 > kTcWaitNs) break;
  }
  return false;
}

// nsteps MMAs of K = 16: operand A from `a` (leading / stride offsets, bytes per
// step), operand B likewise; the first one overwrites D when acc is false.
struct Operand {
  uint32_t base, lbo, sbo, step;
};
__device__ __forceinline__ void mma_steps(uint32_t d, Operand a, Operand b, uint32_t id, int s0, int s1, bool acc) {
  for (int s = s0; s < s1; ++s)
    mma_bf16(d, sdesc(a.base + s * a.step, a.lbo, a.sbo), sdesc(b.base + s * b.step, b.lbo, b.sbo), id,
             (acc || s > s0) ? 1u : 0u);
}

// Operands from an R-row tile (canon): K along the row's 16-byte groups, or K
// along the rows.
__device__ __forceinline__ Operand k_major(const void* t, int R) {
  return {saddr(t), (uint32_t)R * 16u, 128u, (uint32_t)R * 32u};
}
__device__ __forceinline__ Operand mn_major(const void* t, int R) { return {saddr(t), 128u, (uint32_t)R * 16u, 256u}; }

__device__ __forceinline__ uint32_t pack_bf16(float x, float y) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<const uint32_t*>(&h);
}

constexpr int kEpiWarps = 16, kEpiThreads = 32 * kEpiWarps, kNetThreads = kEpiThreads + 32;
constexpr int kInPad = 48;                       // the first layer's K, 40 rounded up to the MMA's 16
constexpr int kInChunks = kTcRows * (kMlpIn / 8);   // 16-byte chunks of a tile's inputs
constexpr int kOutPad = 16;

__host__ __device__ constexpr int layer_kp(int l) { return l == 0 ? kInPad : kMlpHidden; }
__host__ __device__ constexpr int layer_np(int l) { return l == kMlpLayers - 1 ? kOutPad : kMlpHidden; }
__host__ __device__ constexpr int img_off(int l) {   // BF16 elements before layer l's weight image
  return l == 0 ? 0 : kMlpHidden * kInPad + (l - 1) * kMlpHidden * kMlpHidden;
}
constexpr int kImgTotal = img_off(kMlpLayers - 1) + kOutPad * kMlpHidden;

// Shared memory of the two network kernels: the five weight images, the A tile,
// dz of the output layer, input shift and scale, biases, then the mbarriers.
struct NetSmem {
  __nv_bfloat16 w[kImgTotal];
  __nv_bfloat16 a[kTcRows * kMlpHidden];
  __nv_bfloat16 dz5[kTcRows * kOutPad];
  float norm[2 * kMlpIn];
  float bias[4 * kMlpHidden + 8];
  float red[4 * 8];
  unsigned long long ready[2];   // a half of the A tile is staged (one arrival per epilogue warp)
  unsigned long long done;       // the layer's MMAs have completed
  unsigned long long drained;    // all MMAs have (used once)
  uint32_t slot;
};

// Hand a staged half of the A tile to the issuing warp: the tile's generic-proxy
// writes become visible to the tensor cores, and this warp's TMEM reads are done.
__device__ __forceinline__ void hand_over(unsigned long long* b) {
  fence_async_smem();
  fence_before();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(b);
}

// A tile's inputs as 16-byte chunks q < 640 of 8 values: row q % 128, columns
// 8 (q / 128) .. + 7; VEC: X is 16-byte aligned.
struct InChunk {
  float v[8];
};
__device__ __forceinline__ void load_inputs(InChunk (&c)[2], const float* __restrict__ X, int b0, int rows, bool vec) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int q = (int)threadIdx.x + i * kEpiThreads, r = q & (kTcRows - 1), k = (q >> 7) * 8;
    if (q >= kInChunks || r >= rows) {
#pragma unroll
      for (int j = 0; j < 8; ++j) c[i].v[j] = 0.f;
      continue;
    }
    const float* s = X + (size_t)(b0 + r) * kMlpIn + k;
    if (vec) {
      const float4 u = __ldg(reinterpret_cast<const float4*>(s)), w = __ldg(reinterpret_cast<const float4*>(s) + 1);
      c[i].v[0] = u.x; c[i].v[1] = u.y; c[i].v[2] = u.z; c[i].v[3] = u.w;
      c[i].v[4] = w.x; c[i].v[5] = w.y; c[i].v[6] = w.z; c[i].v[7] = w.w;
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) c[i].v[j] = __ldg(s + j);
    }
  }
}
// The scaled inputs as the first layer's A tile [128][48], and (g, training) its
// copy for the weight gradient.  Column 40 is one in the rows that exist: the
// weight images are zero there, and the weight gradient's column 40 is the bias
// gradient.
__device__ __forceinline__ void stage_inputs(const InChunk (&c)[2], const float* norm, unsigned char* a, int rows,
                                             unsigned char* g) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int q = (int)threadIdx.x + i * kEpiThreads, r = q & (kTcRows - 1), k = (q >> 7) * 8;
    if (q < kInChunks) {
      uint32_t p[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float x = r < rows ? (c[i].v[2 * j] - norm[k + 2 * j]) * norm[kMlpIn + k + 2 * j] : 0.f;
        const float y = r < rows ? (c[i].v[2 * j + 1] - norm[k + 2 * j + 1]) * norm[kMlpIn + k + 2 * j + 1] : 0.f;
        p[j] = pack_bf16(x, y);
      }
      const uint4 u = make_uint4(p[0], p[1], p[2], p[3]);
      *reinterpret_cast<uint4*>(a + canon(r, k, kTcRows)) = u;
      if (g) *reinterpret_cast<uint4*>(g + canon(r, k, kTcRows)) = u;
    } else if (q < kInChunks + kTcRows) {   // columns 40 .. 47
      const uint4 u = make_uint4(r < rows ? 0x3F80u : 0u, 0u, 0u, 0u);   // BF16 one, zeros
      *reinterpret_cast<uint4*>(a + canon(r, kMlpIn, kTcRows)) = u;
      if (g) *reinterpret_cast<uint4*>(g + canon(r, kMlpIn, kTcRows)) = u;
    }
  }
}

// The set-up both network kernels share: TMEM, barriers, weights, constants.
__device__ __forceinline__ uint32_t net_setup(NetSmem& s, uint32_t ncols, const __nv_bfloat16* __restrict__ wimg,
                                              const MlpDims& d, const float* __restrict__ param,
                                              const float* __restrict__ in_shift, const float* __restrict__ in_scale) {
  const int tid = threadIdx.x;
  if (tid < 32) tmem_alloc(&s.slot, ncols);
  if (tid == 0) {
    mbar_init(&s.ready[0], kEpiWarps);
    mbar_init(&s.ready[1], kEpiWarps);
    mbar_init(&s.done, 1);
    mbar_init(&s.drained, 1);
  }
  const uint4* src = reinterpret_cast<const uint4*>(wimg);
  uint4* dst = reinterpret_cast<uint4*>(s.w);
#pragma unroll 4
  for (int i = tid; i < kImgTotal / 8; i += kNetThreads) dst[i] = __ldg(src + i);
  for (int k = tid; k < kMlpIn; k += kNetThreads) {
    s.norm[k] = in_shift[k];
    s.norm[kMlpIn + k] = in_scale[k];
  }
  for (int l = 0; l < kMlpLayers; ++l)
    for (int n = tid; n < d.out[l]; n += kNetThreads) s.bias[l * kMlpHidden + n] = param[d.boff[l] + n];
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
  return s.slot;
}

// The MMA thread's operations (pnp_mlpflow.cuh).  Layer l's accumulators: two column
// blocks by turns, or (TRAIN) a block each for the first three layers and one that
// layer 4, the output and the data gradients share.
__device__ __forceinline__ bool drain_mmas(unsigned long long* bar) {
  mma_commit(bar);
  return mbar_wait_tc(bar, 0);
}

template <bool TRAIN>
struct NetOps {
  NetSmem& s;
  uint32_t tmem;
  __device__ uint32_t dcol(int l) const { return tmem + (TRAIN ? min(l, 3) : l & 1) * kMlpHidden; }
  __device__ bool ready(int h, unsigned phase) {
    if (!mbar_wait_tc(&s.ready[h], phase)) return false;
    fence_after();
    return true;
  }
  // z = a W^T, half h of K (the first layer's 48 at once)
  __device__ void forward(int l, int h) {
    const int mid = l == 0 ? kInPad / 16 : kMlpHidden / 32, end = layer_kp(l) / 16;
    mma_steps(dcol(l), k_major(s.a, kTcRows), k_major(s.w + img_off(l), layer_np(l)),
              idesc_bf16(kTcRows, layer_np(l), false, false), h ? mid : 0, h ? end : mid, h != 0);
  }
  // da = dz W: dz from the A tile or the output layer's, W^T by reading the forward
  // image with K along its rows
  __device__ void backward(int l) {
    const bool out = l == kMlpLayers - 1;
    mma_steps(dcol(3), k_major(out ? s.dz5 : s.a, kTcRows), mn_major(s.w + img_off(l), layer_np(l)),
              idesc_bf16(kTcRows, kMlpHidden, false, true), 0, layer_np(l) / 16, false);
  }
  __device__ void commit() { mma_commit(&s.done); }
  __device__ bool drain() { return drain_mmas(&s.drained); }
};

// 16 accumulator columns + bias as pairs
__device__ __forceinline__ float2 z_pair(const float (&v)[16], const float* bias, int i) {
  return __fadd2_rn(make_float2(v[2 * i], v[2 * i + 1]), *reinterpret_cast<const float2*>(bias + 2 * i));
}

constexpr float kInferClip = 6.0f;

// records a wait that ran out; the MMAs are drained, so the tensor memory can go
// once every warp's reads of it are done
__device__ __forceinline__ void net_end(uint32_t tmem, uint32_t ncols, bool ok, int* err) {
  if (!ok) atomicExch(err, PNP_ERR_TIMEOUT);
  fence_before();
  __syncthreads();
  if (threadIdx.x < 32) tmem_dealloc(tmem, ncols);
}

}  // namespace

// The whole network for inference, one persistent CTA per SM looping over 128-row
// tiles: the weight images stay in shared memory for the kernel's life, and each
// layer's accumulators go from TMEM through registers (bias, GELU) straight back
// into the A tile of the next layer, so that nothing between the input rows and
// the five outputs touches global memory.  Two accumulators alternate, so that a
// layer's MMAs may start while the last columns of the one before are read.
// The input is scaled in FP32, z + bias and GELU are FP32, the output is clipped
// to +-6 standard deviations and scaled back.  Bound by the epilogues' issue slots
// (erff); 32,768 rows: 33.5 us, 38 us with one 16-warp phase per layer and the MMAs
// waiting for all of it.
__global__ void __launch_bounds__(kNetThreads, 1) k_mlp_infer_tc(const float* __restrict__ X, int B, int vec,
                                                              const __nv_bfloat16* __restrict__ wimg, MlpDims d,
                                                              const float* __restrict__ param,
                                                              const float* __restrict__ in_shift,
                                                              const float* __restrict__ in_scale,
                                                              const float* __restrict__ out_shift,
                                                              const float* __restrict__ out_scale, int skip_out,
                                                              int skip_in, float* __restrict__ Y, int* err) {
  extern __shared__ __align__(128) unsigned char tc_raw[];
  NetSmem& s = *reinterpret_cast<NetSmem*>(tc_raw);
  constexpr uint32_t kCols = 2 * kMlpHidden;
  const uint32_t tmem = net_setup(s, kCols, wimg, d, param, in_shift, in_scale);
  const int tid = threadIdx.x, warp = tid >> 5;
  const int ntiles = (B + kTcRows - 1) / kTcRows;
  unsigned phase = 0;
  bool ok = true;
  if (warp == kEpiWarps) {
    if ((tid & 31) == 0) {
      NetOps<false> o{s, tmem};
      ok = flow_network<kMlpLayers, false>(o, blockIdx.x, ntiles, gridDim.x);
    }
    __syncwarp();
  } else {
    const int grp = warp & 3, quarter = warp >> 2, r = 32 * grp + (tid & 31);
    const uint32_t lane = tmem + ((uint32_t)(32 * grp) << 16);
    unsigned char* a = reinterpret_cast<unsigned char*>(s.a);
    InChunk in[2];
    if ((int)blockIdx.x < ntiles)
      load_inputs(in, X, blockIdx.x * kTcRows, min(kTcRows, B - (int)blockIdx.x * kTcRows), vec != 0);
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
      const int b0 = tile * kTcRows, rows = min(kTcRows, B - b0);
      stage_inputs(in, s.norm, a, rows, nullptr);
      hand_over(&s.ready[0]);
      hand_over(&s.ready[1]);
      const int next = tile + (int)gridDim.x;   // its inputs arrive under this tile's layers
      if (next < ntiles) load_inputs(in, X, next * kTcRows, min(kTcRows, B - next * kTcRows), vec != 0);
      for (int l = 0; l < kMlpLayers && ok; ++l, phase ^= 1u) {
        ok = __all_sync(0xffffffffu, mbar_wait_tc(&s.done, phase));
        if (!ok) break;
        fence_after();
        const uint32_t acc = lane + (l & 1) * kMlpHidden;
        const float* bias = s.bias + l * kMlpHidden;
        if (l + 1 < kMlpLayers) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int c0 = 64 * h + 16 * quarter;
            float v[16];
            tmem_ld16(acc + c0, v);
            uint32_t pk[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float2 z = z_pair(v, bias + c0, i);
              pk[i] = pack_bf16(gelu_erf(z.x), gelu_erf(z.y));
            }
            *reinterpret_cast<uint4*>(a + canon(r, c0, kTcRows)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            *reinterpret_cast<uint4*>(a + canon(r, c0 + 8, kTcRows)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
            hand_over(&s.ready[h]);
          }
        } else if (quarter == 0) {
          float v[16];
          tmem_ld16(acc, v);
          if (r < rows) {
#pragma unroll
            for (int n = 0; n < kMlpOut; ++n) {
              const float yn = fminf(fmaxf(v[n] + bias[n], -kInferClip), kInferClip);
              const float xs = n == skip_out ? __ldg(X + (size_t)(b0 + r) * kMlpIn + skip_in) : 0.f;
              Y[(size_t)(b0 + r) * kMlpOut + n] = yn / out_scale[n] + out_shift[n] + xs;
            }
          }
        }
      }
    }
  }
  net_end(tmem, kCols, ok, err);
}

// Training, the rows' part: forward through all layers, the loss and its
// gradient, and the data gradients back to the first layer, one 128-row tile at
// a time on chip (one persistent CTA per SM).  What leaves the SM is what the
// weight gradients contract over the batch: the BF16 operands a_0 .. a_4 and
// dz_1 .. dz_5, as tiles in the shared-memory layout.  Layer l's accumulators sit
// in TMEM columns 128 (l - 1) and become GELU'(z_l) in place for the way back
// (layer 4's derivative waits in registers instead: its columns take the output
// layer's and then the data gradients' accumulators), so nothing FP32 is written
// but the partial sums of the loss and of the output bias gradient.
// What bounds it: issue slots of the epilogues (erff and expf of 512 values per
// row: 49 warp instructions per 32 values, the schedulers 45% busy) and the serial
// chain of nine MMA phases per tile between them; the operand tiles are 2.2 KB per
// row of writes (11% of HBM).  65,536 rows: 113 us, the gradient of a batch as a
// caller sees it 209 us with its host copies, against 699 us layer by layer
// through FP32 activations in HBM (24 launches).
__global__ void __launch_bounds__(kNetThreads, 1)
    k_mlp_train_tc(const float* __restrict__ X, const float* __restrict__ T, int B, int vec,
                   const __nv_bfloat16* __restrict__ wimg, MlpDims d, const float* __restrict__ param,
                   const float* __restrict__ in_shift, const float* __restrict__ in_scale,
                   const float* __restrict__ out_shift, const float* __restrict__ out_scale, int skip_out, int skip_in,
                   unsigned char* __restrict__ at, unsigned char* __restrict__ dzt, float* __restrict__ lpart,
                   int* err) {
  extern __shared__ __align__(128) unsigned char tc_raw[];
  NetSmem& s = *reinterpret_cast<NetSmem*>(tc_raw);
  constexpr uint32_t kCols = 4 * kMlpHidden;
  const uint32_t tmem = net_setup(s, kCols, wimg, d, param, in_shift, in_scale);
  const int tid = threadIdx.x, warp = tid >> 5;
  const int ntiles = (B + kTcRows - 1) / kTcRows;
  const uint32_t last = 3 * kMlpHidden;   // the column block of layer 4, the output and the data gradients
  unsigned phase = 0;
  bool ok = true;
  if (warp == kEpiWarps) {
    if ((tid & 31) == 0) {
      NetOps<true> o{s, tmem};
      ok = flow_network<kMlpLayers, true>(o, blockIdx.x, ntiles, gridDim.x);
    }
    __syncwarp();
  } else {
    const int grp = warp & 3, quarter = warp >> 2, r = 32 * grp + (tid & 31);
    const uint32_t lane = tmem + ((uint32_t)(32 * grp) << 16);
    unsigned char* a = reinterpret_cast<unsigned char*>(s.a);
    const float inv = 1.0f / (float)((size_t)B * kMlpOut);
    float sum[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // squared errors, then dz of the output layer per column
    InChunk in[2];
    if ((int)blockIdx.x < ntiles)
      load_inputs(in, X, blockIdx.x * kTcRows, min(kTcRows, B - (int)blockIdx.x * kTcRows), vec != 0);
    auto wait = [&]() {
      ok = __all_sync(0xffffffffu, mbar_wait_tc(&s.done, phase));
      phase ^= 1u;
      if (ok) fence_after();
      return ok;
    };
    // 16 columns of BF16 values of row r into the A tile (when st) and the global tile
    auto put = [&](const uint32_t (&pk)[8], int c0, unsigned char* g, bool st) {
      const uint4 u0 = make_uint4(pk[0], pk[1], pk[2], pk[3]), u1 = make_uint4(pk[4], pk[5], pk[6], pk[7]);
      const uint32_t o0 = canon(r, c0, kTcRows), o1 = canon(r, c0 + 8, kTcRows);
      if (st) {
        *reinterpret_cast<uint4*>(a + o0) = u0;
        *reinterpret_cast<uint4*>(a + o1) = u1;
      }
      *reinterpret_cast<uint4*>(g + o0) = u0;
      *reinterpret_cast<uint4*>(g + o1) = u1;
    };
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
      const int b0 = tile * kTcRows, rows = min(kTcRows, B - b0);
      unsigned char* ga = at + (size_t)tile * kATileBytes;
      unsigned char* gz = dzt + (size_t)tile * kDzTileBytes;
      stage_inputs(in, s.norm, a, rows, ga);
      hand_over(&s.ready[0]);
      hand_over(&s.ready[1]);
      const int next = tile + (int)gridDim.x;
      if (next < ntiles) load_inputs(in, X, next * kTcRows, min(kTcRows, B - next * kTcRows), vec != 0);
      float g4[2][16];   // GELU'(z_4) of this thread's 32 values
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        if (ok && wait()) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int c0 = 64 * h + 16 * quarter;
            const uint32_t acc = lane + l * kMlpHidden + c0;
            float v[16], dg[16];
            tmem_ld16(acc, v);
            uint32_t pk[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float2 z = z_pair(v, s.bias + l * kMlpHidden + c0, i);
              float g0, g1;
              gelu_erf_d(z.x, g0, dg[2 * i]);
              gelu_erf_d(z.y, g1, dg[2 * i + 1]);
              pk[i] = pack_bf16(g0, g1);
            }
            put(pk, c0, ga + kA0Bytes + l * kTileBytes, true);
            if (l < 3) {
              tmem_st16(acc, dg);
            } else {
#pragma unroll
              for (int i = 0; i < 16; ++i) g4[h][i] = dg[i];
            }
            hand_over(&s.ready[h]);
          }
        }
      }
      if (ok && wait()) {   // the outputs: loss and its gradient
        if (quarter == 0) {
          float v[16];
          tmem_ld16(lane + last, v);
          float dz[kMlpOut];
#pragma unroll
          for (int n = 0; n < kMlpOut; ++n) {
            dz[n] = 0.f;
            if (r < rows) {
              const size_t t = (size_t)(b0 + r) * kMlpOut + n;
              const float tf = n == skip_out ? T[t] - X[(size_t)(b0 + r) * kMlpIn + skip_in] : T[t];
              const float e = v[n] + s.bias[4 * kMlpHidden + n] - (tf - out_shift[n]) * out_scale[n];
              dz[n] = 2.0f * e * inv;
              sum[0] += e * e;
            }
          }
          const uint4 u0 = make_uint4(pack_bf16(dz[0], dz[1]), pack_bf16(dz[2], dz[3]), pack_bf16(dz[4], 0.f), 0u);
          const uint4 u1 = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
          for (int n = 0; n < kMlpOut; ++n) sum[1 + n] += __bfloat162float(__float2bfloat16_rn(dz[n]));
          unsigned char* z5 = reinterpret_cast<unsigned char*>(s.dz5);
          unsigned char* g5 = gz + 4 * kTileBytes;
          *reinterpret_cast<uint4*>(z5 + canon(r, 0, kTcRows)) = u0;
          *reinterpret_cast<uint4*>(z5 + canon(r, 8, kTcRows)) = u1;
          *reinterpret_cast<uint4*>(g5 + canon(r, 0, kTcRows)) = u0;
          *reinterpret_cast<uint4*>(g5 + canon(r, 8, kTcRows)) = u1;
        }
        hand_over(&s.ready[0]);
        hand_over(&s.ready[1]);
      }
#pragma unroll
      for (int l = 3; l >= 0; --l) {   // dz of layer l + 1
        if (ok && wait()) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int c0 = 64 * h + 16 * quarter;
            float v[16], dg[16];
            tmem_ld16(lane + last + c0, v);
            if (l < 3) tmem_ld16(lane + l * kMlpHidden + c0, dg);
            uint32_t pk[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float2 dd = l < 3 ? make_float2(dg[2 * i], dg[2 * i + 1])
                                      : make_float2(g4[h][2 * i], g4[h][2 * i + 1]);
              const float2 p = __fmul2_rn(make_float2(v[2 * i], v[2 * i + 1]), dd);
              pk[i] = pack_bf16(p.x, p.y);
            }
            put(pk, c0, gz + l * kTileBytes, l > 0);
            if (l > 0) hand_over(&s.ready[h]);
          }
        }
      }
    }
    // the CTA's sums over its rows in a fixed order: lanes, then the four warps
    if (quarter == 0) {
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        float x = sum[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if ((tid & 31) == 0) s.red[8 * grp + q] = x;
      }
    }
  }
  __syncthreads();
  if (tid < 6) lpart[(size_t)blockIdx.x * 8 + tid] = (s.red[tid] + s.red[8 + tid]) + (s.red[16 + tid] + s.red[24 + tid]);
  net_end(tmem, kCols, ok, err);
}

// Weight gradients: one CTA takes every splits[l]-th tile of layer l and
// contracts dz_l with a_(l-1) over its rows, D[n][k] += sum_b dz[b][n] a[b][k],
// both operands read from their tiles with K along the rows.  The bias gradient
// is a column of ones: column 40 of the input tile, and for the hidden layers 16
// more columns behind the tile, set once per stage.  The output layer (five rows)
// runs transposed, D[k][n].  The tiles arrive by bulk copies through a three-
// stage ring: one thread feeds it, one issues the MMAs, four warps drain the
// accumulators (65,536 rows: 26 us).  These alternate between two TMEM blocks every two tiles: the
// tensor cores' FP32 sums are not rounded to nearest, so a sum of 256 rows (2e-7
// of the gradient) goes on in registers (over all of a CTA's rows in TMEM the
// error was 2e-6).  Per tile 64 KB are read for 4.2 MFLOP, so the copies bound
// it: 5.4 TB/s.  Each CTA writes its sums to its own slice of `partial`.
constexpr int kWgStages = 3, kWgThreads = 192, kWgRun = 2;   // stages; threads; tiles per TMEM sum
constexpr int kWgCols = kMlpHidden + 16;
struct WgSmem {
  unsigned char a[kWgStages][kTileBytes];
  unsigned char b[kWgStages][kTileBytes + 16 * kTcRows * 2];
  unsigned long long full[kWgStages], empty[kWgStages];   // ring slots
  unsigned long long sum[2], free[2];                     // TMEM blocks: a sum is complete / has been read
  unsigned long long drained;                             // all MMAs have completed (used once)
  uint32_t slot;
  int bad;
};

// The MMA thread's operations (pnp_mlpflow.cuh).
struct WgOps {
  WgSmem& s;
  uint32_t tmem, id;
  __device__ bool freed(int block, unsigned phase) { return mbar_wait_tc(&s.free[block], phase); }
  __device__ bool full(int q, unsigned phase) {
    if (!mbar_wait_tc(&s.full[q], phase)) return false;
    fence_after();
    return true;
  }
  __device__ void product(int q, int block, bool acc) {
    mma_steps(tmem + block * 256, mn_major(s.a[q], kTcRows), mn_major(s.b[q], kTcRows), id, 0, kTcRows / 16, acc);
  }
  __device__ void commit_slot(int q) { mma_commit(&s.empty[q]); }
  __device__ void commit_sum(int block) { mma_commit(&s.sum[block]); }
  __device__ bool drain() { return drain_mmas(&s.drained); }
};

__global__ void __launch_bounds__(kWgThreads, 1)
    k_mlp_wgrad_tc(const unsigned char* __restrict__ at, const unsigned char* __restrict__ dzt, int ntiles,
                   const __grid_constant__ WgPlan plan, float* __restrict__ partial, int* err) {
  extern __shared__ __align__(128) unsigned char tc_raw[];
  WgSmem& s = *reinterpret_cast<WgSmem*>(tc_raw);
  int l = 0, blk = blockIdx.x;
  while (l + 1 < kMlpLayers && blk >= plan.splits[l]) blk -= plan.splits[l++];
  const int splits = plan.splits[l], tid = threadIdx.x, warp = tid >> 5;
  const bool out = l == kMlpLayers - 1;
  const int N = out ? kOutPad : l == 0 ? kInPad : kWgCols;
  const unsigned abytes = kTileBytes, bbytes = out ? kTcRows * kOutPad * 2 : l == 0 ? kA0Bytes : kTileBytes;
  const int ntl = blk < ntiles ? (ntiles - blk + splits - 1) / splits : 0;   // this CTA's tiles
  const int nrun = (ntl + kWgRun - 1) / kWgRun;
  if (warp == 0) tmem_alloc(&s.slot, 512);
  if (tid == 0) {
    for (int q = 0; q < kWgStages; ++q) {
      mbar_init(&s.full[q], 1);
      mbar_init(&s.empty[q], 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&s.sum[q], 1);
      mbar_init(&s.free[q], 4);
    }
    mbar_init(&s.drained, 1);
    s.bad = 0;
  }
  if (!out && l > 0)   // columns 128 .. 143 of B: ones in column 128
    for (int e = tid; e < kWgStages * 2 * kTcRows; e += kWgThreads) {
      const int q = e / (2 * kTcRows), rr = e % kTcRows, g = (e / kTcRows) & 1;
      *reinterpret_cast<uint4*>(s.b[q] + canon(rr, kMlpHidden + 8 * g, kTcRows)) =
          make_uint4(g == 0 ? 0x3F80u : 0u, 0u, 0u, 0u);
    }
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = s.slot;
  bool ok = true;
  if (warp < 4) {
    // this thread's TMEM lane: output n (hidden layers) or input k (the output layer)
    const uint32_t lane = tmem + ((uint32_t)(32 * warp) << 16);
    float acc[kWgCols];
#pragma unroll
    for (int i = 0; i < kWgCols; ++i) acc[i] = 0.f;
    for (int g = 0; g < nrun && ok; ++g) {
      ok = __all_sync(0xffffffffu, mbar_wait_tc(&s.sum[g & 1], (g >> 1) & 1));
      if (!ok) break;
      fence_after();
#pragma unroll
      for (int c0 = 0; c0 < kWgCols; c0 += 16)
        if (c0 < N) {
          float v[16];
          tmem_ld16(lane + (g & 1) * 256 + c0, v);
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[c0 + i] += v[i];
        }
      fence_before();
      __syncwarp();
      if ((tid & 31) == 0) mbar_arrive(&s.free[g & 1]);
    }
    if (ok) {
      float* p = partial + plan.off[l] + (size_t)blk * plan.len[l];
      const int K = l == 0 ? kMlpIn : kMlpHidden;
      if (out) {
#pragma unroll
        for (int c = 0; c < kMlpOut; ++c) p[(size_t)c * kMlpHidden + tid] = acc[c];
      } else {
#pragma unroll
        for (int c = 0; c < kMlpHidden; c += 4)
          if (c < K)
            *reinterpret_cast<float4*>(p + (size_t)tid * K + c) =
                make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]);
        p[(size_t)kMlpHidden * K + tid] = l == 0 ? acc[kMlpIn] : acc[kMlpHidden];
      }
    }
  } else if (tid == 128) {
    int n = 0;
    for (; n < ntl; ++n) {
      const int q = n % kWgStages, use = n / kWgStages;
      if (use > 0 && !(ok = mbar_wait_tc(&s.empty[q], (use - 1) & 1))) break;
      const size_t tile = (size_t)blk + (size_t)n * splits;
      const unsigned char* ta = at + tile * kATileBytes;
      const unsigned char* tz = dzt + tile * kDzTileBytes;
      mbar_expect(&s.full[q], abytes + bbytes);
      bulk_load(s.a[q], out ? ta + kA0Bytes + 3 * kTileBytes : tz + (size_t)l * kTileBytes, abytes, &s.full[q]);
      bulk_load(s.b[q], out ? tz + 4 * kTileBytes : l == 0 ? ta : ta + kA0Bytes + (size_t)(l - 1) * kTileBytes, bbytes,
                &s.full[q]);
    }
    // no copy outlives the CTA: the last ones have landed (already seen by the MMA
    // thread unless a wait ran out)
    for (int m = n > kWgStages ? n - kWgStages : 0; m < n; ++m) mbar_wait_tc(&s.full[m % kWgStages], (m / kWgStages) & 1);
  } else if (tid == 160) {
    WgOps o{s, tmem, idesc_bf16(kTcRows, N, true, true)};
    ok = flow_wgrad<kWgStages, kWgRun>(o, ntl);
  }
  if (!ok) s.bad = 1;
  __syncthreads();
  if (s.bad && tid == 0) atomicExch(err, PNP_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// Sums of the CTAs' partial gradients in a fixed order, eight running sums per
// parameter (partials 8q .. 8q + 7) folded by halves, in one launch for all layers.
// The last block sums the rows' kernel's squared errors and output-bias
// gradients: 120 threads take every twentieth CTA of one of the six, then a
// fixed-order sum.  Bound by the latency of the loads: eight in flight (7 us; 13
// us per layer with one thread walking all partials four at a time).
__device__ __forceinline__ float sum_strided(const float* __restrict__ src, size_t ld, int b, int step, int n) {
  float t[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (; b < n; b += 8 * step) {
    float v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = b + q * step < n ? __ldg(src + (size_t)(b + q * step) * ld) : 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] += v[q];
  }
  return ((t[0] + t[4]) + (t[1] + t[5])) + ((t[2] + t[6]) + (t[3] + t[7]));
}
constexpr int kRedThreads = 128, kLossSplit = 20;
__global__ void __launch_bounds__(kRedThreads) k_mlp_reduce(const float* __restrict__ partial,
                                                            const __grid_constant__ WgPlan plan,
                                                            const __grid_constant__ MlpDims d,
                                                            const float* __restrict__ lpart, int nl, float loss_scale,
                                                            float* __restrict__ grad, float* __restrict__ loss) {
  const int ob = (int)d.boff[kMlpLayers - 1], tid = threadIdx.x;   // the output biases are the last parameters
  if (blockIdx.x + 1 == gridDim.x) {
    __shared__ float sh[6 * kLossSplit];
    if (tid < 6 * kLossSplit) sh[tid] = sum_strided(lpart + tid / kLossSplit, 8, tid % kLossSplit, kLossSplit, nl);
    __syncthreads();
    if (tid < 6) {
      float t = 0.f;
      for (int q = 0; q < kLossSplit; ++q) t += sh[tid * kLossSplit + q];
      if (tid == 0) *loss = t * loss_scale;
      else grad[ob + tid - 1] = t;
    }
    return;
  }
  const int e = blockIdx.x * kRedThreads + tid;
  if (e >= ob) return;
  int l = 0;
  while (l + 1 < kMlpLayers && e >= (int)d.woff[l + 1]) ++l;
  grad[e] = sum_strided(partial + plan.off[l] + (e - (int)d.woff[l]), plan.len[l], 0, 1, plan.splits[l]);
}

// Weight images: for every layer the BF16 weights [Np][Kp] in the shared-memory
// layout, zero in the padding.
size_t mlp_image_elems() { return kImgTotal; }

__global__ void k_mlp_images(const float* __restrict__ param, __nv_bfloat16* __restrict__ img, MlpDims d) {
  const int stride = gridDim.x * blockDim.x;
  for (int l = 0; l < kMlpLayers; ++l) {
    const int K = d.in[l], N = d.out[l], Kp = layer_kp(l), Np = layer_np(l);
    unsigned char* f = reinterpret_cast<unsigned char*>(img + img_off(l));
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < Np * Kp; e += stride) {
      const int n = e / Kp, k = e - n * Kp;
      *reinterpret_cast<__nv_bfloat16*>(f + canon(n, k, Np)) =
          __float2bfloat16_rn((n < N && k < K) ? param[d.woff[l] + (size_t)n * K + k] : 0.f);
    }
  }
}

cudaError_t mlp_make_images(const float* param, __nv_bfloat16* img, cudaStream_t s) {
  k_mlp_images<<<64, 256, 0, s>>>(param, img, mlp_dims());
  return cudaGetLastError();
}

// ---- launchers ----
namespace {
int tc_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  return sms;
}
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
bool skip_ok(const MlpBufs& b) {
  return b.skip_out < kMlpOut && b.skip_in < kMlpIn && !(b.skip_out >= 0 && b.skip_in < 0);
}
}  // namespace

cudaError_t mlp_infer_tc(const MlpBufs& b, const float* X, int B, float* Y, cudaStream_t s) {
  if (B < 1) return cudaSuccess;
  const int sms = tc_sms();
  if (sms < 1 || !skip_ok(b)) return cudaErrorInvalidValue;
  const cudaError_t e =
      cudaFuncSetAttribute(k_mlp_infer_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(NetSmem));
  if (e != cudaSuccess) return e;
  const int ntiles = (B - 1) / kTcRows + 1;
  k_mlp_infer_tc<<<(unsigned)std::min(ntiles, sms), kNetThreads, sizeof(NetSmem), s>>>(
      X, B, aligned16(X) ? 1 : 0, b.wimg, mlp_dims(), b.param, b.in_shift, b.in_scale, b.out_shift, b.out_scale,
      b.skip_out, b.skip_in, Y, b.err);
  return cudaGetLastError();
}

// How many CTAs share each layer's tiles: one wave of the SMs (a CTA takes one by its
// shared and tensor memory), in proportion to the bytes per tile (44, 64, 64, 64 and 36
// KB of 272), at most one per tile; a layer's slice of the partial sums per CTA.
WgPlan mlp_wgrad_plan(int ntiles, int sms) {
  const MlpDims d = mlp_dims();
  constexpr int full[kMlpLayers] = {24, 36, 36, 36, 20};
  static_assert(full[0] + full[1] + full[2] + full[3] + full[4] == kWgCtas, "shares of kWgCtas");
  int share[kMlpLayers];
  share_ctas(full, kWgCtas, sms, share);
  WgPlan p{};
  size_t off = 0;
  for (int l = 0; l < kMlpLayers; ++l) {
    p.splits[l] = std::max(1, std::min(ntiles, share[l]));
    p.len[l] = (size_t)d.in[l] * d.out[l] + (l + 1 < kMlpLayers ? d.out[l] : 0);
    p.off[l] = off;
    off += p.len[l] * p.splits[l];
  }
  p.total = off;
  return p;
}

cudaError_t mlp_train_tc(const MlpBufs& b, const float* X, const float* T, int B, cudaStream_t s) {
  if (B < 1) return cudaErrorInvalidValue;
  const int sms = std::min(tc_sms(), kMlpMaxRowCtas);
  if (sms < 1 || !skip_ok(b)) return cudaErrorInvalidValue;
  cudaError_t e =
      cudaFuncSetAttribute(k_mlp_train_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(NetSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_mlp_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WgSmem));
  if (e != cudaSuccess) return e;
  const MlpDims d = mlp_dims();
  const int ntiles = (B - 1) / kTcRows + 1, grid = std::min(ntiles, sms);
  k_mlp_train_tc<<<(unsigned)grid, kNetThreads, sizeof(NetSmem), s>>>(
      X, T, B, aligned16(X) ? 1 : 0, b.wimg, d, b.param, b.in_shift, b.in_scale, b.out_shift, b.out_scale, b.skip_out,
      b.skip_in, b.atiles, b.dztiles, b.lpart, b.err);
  const WgPlan plan = mlp_wgrad_plan(ntiles, sms);
  int nblk = 0;
  for (int l = 0; l < kMlpLayers; ++l) nblk += plan.splits[l];
  k_mlp_wgrad_tc<<<(unsigned)nblk, kWgThreads, sizeof(WgSmem), s>>>(b.atiles, b.dztiles, ntiles, plan, b.partial, b.err);
  const float inv = 1.0f / (float)((size_t)B * kMlpOut);
  k_mlp_reduce<<<(unsigned)(d.boff[kMlpLayers - 1] / kRedThreads + 2), kRedThreads, 0, s>>>(
      b.partial, plan, d, b.lpart, grid, inv, b.grad, b.loss);
  return cudaGetLastError();
}

}  // namespace pnp

// The learned warm start's network on the fifth-generation tensor cores.
//
// A multilayer perceptron (GELU hidden layers, affine output) maps a load
// scenario's per-bus (pd, qd) to an ADMM starting point, multipliers and
// per-component penalties.  Every matrix product of its forward and backward
// passes has the form
//
//   C[M x N] = A[M x K] * B[N x K]^T,   A, B bfloat16, K contiguous,
//
// and runs in one of two kernels.  k_gemm_tc has 128 x 128 to 128 x 256 output
// tiles in a persistent, warp-specialised kernel: one CTA per SM loops over
// tiles; warp 0 streams 128 x 64 and up to 256 x 64 operand tiles into a
// four-stage shared-memory ring with TMA (cp.async.bulk.tensor,
// 128-byte swizzle, completion counted on mbarriers); warp 1 issues
// tcgen05.mma (kind::f16, BF16 x BF16 -> FP32, 128 x 256 x 16) into one of two
// 256-column tensor-memory accumulators; warps 2-5 read the other accumulator
// back with tcgen05.ld for a fused epilogue (bias, GELU, GELU derivative,
// bfloat16 row-major and transposed stores, de-standardised outputs), so the
// epilogue of one tile overlaps the main loop of the next.  Long contractions
// are split over K: products with few output tiles run as k_gemm_small, 128 x
// 64 tiles whose CTA keeps every split in an accumulator of its own; the rest
// write FP32 partial tiles summed by k_splitk.
//
// Layout convention: the backward pass needs every operand with its
// contraction index contiguous, so the forward epilogue stores each hidden
// activation both row-major and transposed, the backward epilogue does the
// same for each pre-activation gradient, and the Adam kernel keeps each
// weight both as [out x in] and as [in x out].  Every product is then the
// K-major x K-major form above.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "../../include/acopf.h"
#include "../../include/acopf_mlp.h"
#include "line_qp.cuh"

namespace acopf {
namespace nn {

typedef __nv_bfloat16 bf16;

constexpr int BM = 128, BN = 256, BK = 64, STAGES = 4;  // BN: widest tile of k_gemm_tc (tile_width)
constexpr uint32_t kABytes = BM * BK * 2;  // A tile: 128 rows x 128 bytes
constexpr uint32_t kBBytes = BN * BK * 2;  // B tile: 256 rows x 128 bytes
constexpr int kGemmThreads = 192;          // warp 0 TMA, warp 1 MMA, warps 2-5 epilogue
constexpr int kScratch = 32 * 33;          // floats of epilogue scratch per warp: one 32 x 32 block
constexpr size_t kGemmSmem = 1024 + (size_t)STAGES * (kABytes + kBBytes) + 256;
constexpr uint32_t kTmemCols = 512;        // two 256-column FP32 accumulators

// k_gemm_small
constexpr int SN = 64, kSmallStages = 6, kSmallThreads = 320;  // warp 0 TMA, warp 1 MMA, warps 2-9 epilogue
constexpr uint32_t kSBytes = SN * BK * 2;
constexpr size_t kSmallSmem = 1024 + (size_t)kSmallStages * (kABytes + kSBytes) + 256;
constexpr int kSmallSplits = 512 / SN;  // accumulators that tensor memory holds

// Instruction descriptor of tcgen05.mma kind::f16: D in FP32 (bits 4-5 = 1),
// A and B bfloat16 (bits 7-9 = 1, 10-12 = 1), both K-major (bits 15, 16 = 0),
// N >> 3 in bits 17-22, M >> 4 in bits 24-28.
constexpr uint32_t kIdescM = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BM >> 4) << 24);

enum { EPI_F32 = 0, EPI_GELU = 1, EPI_GELU_BWD = 2, EPI_PARTIAL = 3 };

struct Epi {
  int op;
  int M, N;             // output extent
  int rows_valid;       // bf16 outputs of rows >= rows_valid are written as 0
  const float* bias;    // [N] or null
  float* f32;           // FP32 row-major output (EPI_F32, EPI_PARTIAL; EPI_GELU: the pre-activation, or null)
  int ld_f32;
  size_t split_stride;  // EPI_PARTIAL: elements between the partial tiles of consecutive K splits
  bf16* bf;             // bfloat16 row-major output
  int ld_bf;
  bf16* bt;             // bfloat16 transposed output: (m, n) at bt[n * ld_bt + m] (EPI_GELU: or null)
  int ld_bt;
  const float* z;       // EPI_GELU_BWD: saved pre-activation
  int ld_z;
  const float *mu, *sd; // EPI_F32: not null: outputs de-standardised, y sd + mu (inference)
};

// --------------------------------------------------------------- PTX helpers
// Programmatic dependent launch: every kernel of a step is launched so that it
// may start while the one before it still runs.  It lets its own successor
// start (pdl_go), sets up what touches no global memory, and then waits until
// the kernel before it has completed and its writes are visible (pdl_wait);
// every kernel waits, so completion carries over from one to the next.  The
// gaps and prologues between the small kernels of a step were a third of its
// time: 64 steps of the 30-bus network 7.8 -> 6.6 ms, a prediction for one
// scenario 73 -> 61 us.
__device__ __forceinline__ void pdl_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(saddr(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait for the completion of the phase with the given parity
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, long long limit) {
  long long t0 = clock64();
  while (!mbar_test(b, parity))
    if (clock64() - t0 > limit) return false;
  return true;
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          saddr(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(saddr(bar))
      : "memory");
}
// shared-memory matrix descriptor: K-major operand tile of 128-byte rows with
// the 128-byte swizzle, 8-row groups 1024 bytes apart (stride byte offset),
// descriptor version 1 (bit 46), swizzle mode 2 (bits 61-63)
__device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
  uint64_t d = (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__device__ __forceinline__ uint32_t idesc(int n) { return kIdescM | ((uint32_t)(n >> 3) << 17); }
__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
      "l"(a), "l"(b), "r"(id), "r"(accumulate));
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(bar))
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 consecutive FP32 accumulator columns of this thread's lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float v[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// ------------------------------------------------------------------ epilogue
__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// one element, after the K-split partial tiles have been summed
__device__ __forceinline__ void epi_one(const Epi& e, int m, int n, float acc) {
  switch (e.op) {
    case EPI_F32: {
      float y = acc;
      if (e.bias) y += e.bias[n];
      if (e.sd) y = fmaf(y, e.sd[n], e.mu[n]);
      e.f32[(size_t)m * e.ld_f32 + n] = y;
      break;
    }
    case EPI_GELU: {
      const float zz = acc + e.bias[n];
      if (e.f32) e.f32[(size_t)m * e.ld_f32 + n] = zz;
      const bf16 h = __float2bfloat16_rn(m < e.rows_valid ? gelu_f(zz) : 0.0f);
      e.bf[(size_t)m * e.ld_bf + n] = h;
      if (e.bt) e.bt[(size_t)n * e.ld_bt + m] = h;
      break;
    }
    default: {  // EPI_GELU_BWD
      const float v = m < e.rows_valid ? acc * gelu_grad_f(e.z[(size_t)m * e.ld_z + n]) : 0.0f;
      const bf16 h = __float2bfloat16_rn(v);
      e.bf[(size_t)m * e.ld_bf + n] = h;
      e.bt[(size_t)n * e.ld_bt + m] = h;
      break;
    }
  }
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(b)) : "memory");
}

// EPI_F32: bias, deviation and mean of output columns n0 .. n0 + n - 1 into a
// warp's part of shared memory (stride floats each), fetched before the
// accumulator is waited for.  All 32 lanes call it.
__device__ __forceinline__ void epi_consts(const Epi& e, int n0, int n, float* cst, int stride) {
  if (e.op != EPI_F32) return;
  __syncwarp();
  for (int j = threadIdx.x & 31; j < n && n0 + j < e.N; j += 32) {
    if (e.bias) cst[j] = e.bias[n0 + j];
    if (e.sd) {
      cst[stride + j] = e.sd[n0 + j];
      cst[2 * stride + j] = e.mu[n0 + j];
    }
  }
  __syncwarp();
}

// One warp's 32 x 32 block of the accumulator: lane holds row m0 + lane,
// columns n0 .. n0 + 31.  FP32 outputs are stored from the lanes, 16 bytes of
// a row at a time (through shared memory, in whole rows, the 46,504 x 512
// weight gradient took 49 us against 37).  Pre-activations and row-major
// bfloat16 go through the warp's scratch in shared memory; transposed outputs
// come straight from the lanes, which hold consecutive rows.  A block is read
// back into registers as a whole before it is stored (and a pre-activation
// block read as a whole before it goes to the scratch): the compiler cannot
// move a load past a store that may alias it, and one load per store would pay
// its latency 32 times.  cst: what epi_consts put into shared memory for these
// columns.  All 32 lanes call it.
__device__ __forceinline__ void epi_block(const Epi& e, int m0, int n0, float v[32], int split, float* scratch,
                                          const float* cst, int stride) {
  const int lane = threadIdx.x & 31;
  const int m = m0 + lane, n = n0 + lane;
  const int rows = e.M - m0 < 32 ? e.M - m0 : 32;  // rows of the block that exist (may be <= 0)
  if (e.op == EPI_F32 || e.op == EPI_PARTIAL) {
    if (lane >= rows) return;
    float* dst = e.f32 + (e.op == EPI_PARTIAL ? (size_t)split * e.split_stride : 0) + (size_t)m * e.ld_f32 + n0;
    if (n0 + 32 <= e.N && ((uintptr_t)dst & 15) == 0) {
#pragma unroll
      for (int j = 0; j < 32; j += 4) {
        float4 y = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        if (e.op == EPI_F32 && e.bias) {
          const float4 q = *(const float4*)(cst + j);
          y.x += q.x; y.y += q.y; y.z += q.z; y.w += q.w;
        }
        if (e.op == EPI_F32 && e.sd) {
          const float4 q = *(const float4*)(cst + stride + j), u = *(const float4*)(cst + 2 * stride + j);
          y.x = fmaf(y.x, q.x, u.x); y.y = fmaf(y.y, q.y, u.y); y.z = fmaf(y.z, q.z, u.z); y.w = fmaf(y.w, q.w, u.w);
        }
        *(float4*)(dst + j) = y;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (n0 + j < e.N) {
          float y = v[j];
          if (e.op == EPI_F32 && e.bias) y += cst[j];
          if (e.op == EPI_F32 && e.sd) y = fmaf(y, cst[stride + j], cst[2 * stride + j]);
          dst[j] = y;
        }
    }
    return;
  }
  uint32_t h[16];  // the block's rows in bfloat16, two columns per word
  if (e.op == EPI_GELU) {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] += n0 + j < e.N ? e.bias[n0 + j] : 0.0f;
    if (e.f32) {
#pragma unroll
      for (int j = 0; j < 32; ++j) scratch[lane * 33 + j] = v[j];
      __syncwarp();
      float t[32];
#pragma unroll
      for (int r = 0; r < 32; ++r) t[r] = scratch[r * 33 + lane];
      __syncwarp();
      if (n < e.N) {
        float* dst = e.f32 + (size_t)m0 * e.ld_f32 + n;
#pragma unroll
        for (int r = 0; r < 32; ++r)
          if (r < rows) dst[(size_t)r * e.ld_f32] = t[r];
      }
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = m < e.rows_valid ? gelu_f(v[j]) : 0.0f;
  } else {  // EPI_GELU_BWD: the saved pre-activations, read in rows
    float t[32];
    const float* src = e.z + (size_t)m0 * e.ld_z + n;
#pragma unroll
    for (int r = 0; r < 32; ++r) t[r] = r < rows && n < e.N ? src[(size_t)r * e.ld_z] : 0.0f;
#pragma unroll
    for (int r = 0; r < 32; ++r) scratch[r * 33 + lane] = t[r];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 32; ++j)
      v[j] = m < e.rows_valid && n0 + j < e.N ? v[j] * gelu_grad_f(scratch[lane * 33 + j]) : 0.0f;
    __syncwarp();
  }
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const __nv_bfloat162 w = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    h[j] = *(const uint32_t*)&w;
  }
  if (e.bt && lane < rows) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (n0 + j < e.N)
        e.bt[(size_t)(n0 + j) * e.ld_bt + m] = __ushort_as_bfloat16((unsigned short)(h[j >> 1] >> (16 * (j & 1))));
  }
  // row-major bfloat16 (N and ld_bf are multiples of 8): two rows per store instruction
  uint32_t* sw = (uint32_t*)scratch;
#pragma unroll
  for (int j = 0; j < 16; ++j) sw[lane * 17 + j] = h[j];
  __syncwarp();
  const int w = lane & 15;
#pragma unroll
  for (int i = 0; i < 16; ++i) h[i] = sw[(2 * i + (lane >> 4)) * 17 + w];
  __syncwarp();
  if (n0 + 2 * w < e.N) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int r = 2 * i + (lane >> 4);
      if (r < rows) *(uint32_t*)(e.bf + (size_t)(m0 + r) * e.ld_bf + n0 + 2 * w) = h[i];
    }
  }
}

// work item w -> (split z, row block mb, column block nb).  Within a split,
// items run through groups of kGroup row blocks, column-block-major inside a
// group, so the tiles in flight at one time share a few A and B blocks in L2.
constexpr int kGroup = 16;
__device__ __forceinline__ void decode_item(int w, int mt, int nt, int& z, int& mb, int& nb) {
  z = w / (mt * nt);
  const int r = w - z * mt * nt;
  const int g = r / (kGroup * nt);
  const int g0 = g * kGroup;
  const int gm = mt - g0 < kGroup ? mt - g0 : kGroup;  // row blocks in this group
  const int rr = r - g0 * nt;
  mb = g0 + rr % gm;
  nb = rr / gm;
}

// -------------------------------------------------------------- GEMM kernel
// Persistent: grid = min(work items, SMs), 192 threads, kGemmSmem bytes of
// dynamic shared memory.  Work item w = (split z, row block, column block);
// split z covers K tiles [z * kts, (z + 1) * kts).  Every wait is bounded:
// on time-out the waiting role records *err and stops.
__global__ void __launch_bounds__(kGemmThreads, 1)
    k_gemm_tc(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, int K, int kts,
              int splits, int bn, Epi e, int* err, long long spin) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * kABytes;
  __shared__ __align__(16) float scratch[4][kScratch];
  uint64_t* full = (uint64_t*)(smem + STAGES * (kABytes + kBBytes));
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;  // accumulator a holds a finished tile
  uint64_t* tempty = tfull + 2;      // accumulator a has been read by the epilogue
  uint32_t* tslot = (uint32_t*)(tempty + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_go();
  const int mt = (e.M + BM - 1) / BM, nt = (e.N + bn - 1) / bn;
  const int items = splits * mt * nt;
  const uint32_t bbytes = (uint32_t)bn * BK * 2;
  const int kt_total = (K + BK - 1) / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], 4);  // one arrival per epilogue warp
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(tslot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {  // producer: operand tiles into the ring of stages
      int i = 0;
      bool ok = true;
      for (int w = blockIdx.x; w < items && ok; w += gridDim.x) {
        int z, mb, nb;
        decode_item(w, mt, nt, z, mb, nb);
        const int kt0 = z * kts, kt1 = kt0 + kts < kt_total ? kt0 + kts : kt_total;
        for (int kt = kt0; kt < kt1; ++kt, ++i) {
          const int s = i % STAGES;
          if (i >= STAGES && !mbar_wait(&empty[s], ((i / STAGES) - 1) & 1, spin)) {
            atomicExch(err, 1);
            ok = false;
            break;
          }
          mbar_expect_tx(&full[s], kABytes + bbytes);
          tma_load_2d(sA + s * kABytes, &ta, kt * BK, mb * BM, &full[s]);
          tma_load_2d(sB + s * kBBytes, &tb, kt * BK, nb * bn, &full[s]);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer
      const uint32_t id = idesc(bn);
      int i = 0, j = 0;
      bool ok = true;
      for (int w = blockIdx.x; w < items && ok; w += gridDim.x, ++j) {
        const int z = w / (mt * nt);  // the MMA issuer only needs the split
        const int kt0 = z * kts, kt1 = kt0 + kts < kt_total ? kt0 + kts : kt_total;
        const int a = j & 1, u = j >> 1;
        if (u >= 1 && !mbar_wait(&tempty[a], (u - 1) & 1, spin)) {
          atomicExch(err, 1);
          break;
        }
        tc_fence_after();
        const uint32_t acc = tmem + (uint32_t)(a * BN);
        for (int kt = kt0; kt < kt1; ++kt, ++i) {
          const int s = i % STAGES;
          if (!mbar_wait(&full[s], (i / STAGES) & 1, spin)) {
            atomicExch(err, 1);
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t pa = saddr(sA + s * kABytes), pb = saddr(sB + s * kBBytes);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            mma_bf16(acc, sdesc(pa + 32 * kk), sdesc(pb + 32 * kk), id, (kt > kt0 || kk > 0) ? 1u : 0u);
          mma_commit(&empty[s]);
        }
        if (!ok) break;
        if (kt1 > kt0) mma_commit(&tfull[a]);  // arrives when this tile's MMAs are done
        else mbar_arrive(&tfull[a]);            // empty K range: nothing to wait for
      }
    }
  } else {
    // epilogue: warp w reads accumulator lanes (rows) 32 (w % 4) .. + 31
    const int q = warp & 3;
    int j = 0;
    for (int w = blockIdx.x; w < items; w += gridDim.x, ++j) {
      int z, mb, nb;
      decode_item(w, mt, nt, z, mb, nb);
      const int kt0 = z * kts, kt1 = kt0 + kts < kt_total ? kt0 + kts : kt_total;
      const int a = j & 1, u = j >> 1;
      const int n0 = nb * bn;
      epi_consts(e, n0, bn, scratch[q], BN);
      bool ok = mbar_wait(&tfull[a], u & 1, spin);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) {
        if (lane == 0) atomicExch(err, 1);
        break;
      }
      tc_fence_after();
      for (int c = 0; c < bn; c += 32) {
        if (n0 + c >= e.N) break;
        float v[32];
        if (kt1 > kt0) {
          tmem_ld32(tmem + (uint32_t)(a * BN) + ((uint32_t)(q * 32) << 16) + (uint32_t)c, v);
        } else {
#pragma unroll
          for (int t = 0; t < 32; ++t) v[t] = 0.0f;
        }
        epi_block(e, mb * BM + q * 32, n0 + c, v, z, scratch[q], scratch[q] + c, BN);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[a]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// Products with few output tiles: one 128 x 64 tile per CTA, the whole
// contraction in it.  The K splits of the plan fix how the result is rounded
// (FP32 sums per split, added in order); here each split accumulates in 64
// tensor-memory columns of its own and the epilogue adds them, so there are no
// partial tiles in memory and no second kernel, and eight epilogue warps take
// one 32 x 32 block each where four took eight (a GELU tile of 128 x 256 on
// one SM took 54 us).  One launch can hold two products, the weight and the
// input gradient of a layer.  A layer of 512 x 512 at 256 rows, with launch
// gaps: forward 14.3 -> 10.5 us, backward 25 -> 12-16 us; the 64-wide first
// layer at 128 rows 54 -> 7.3 us.
struct SmallG {
  CUtensorMap ta, tb;  // boxes of 128 and of 64 rows
  int K, kts, splits, mt;
  Epi e;
};
struct SmallP {
  SmallG g[2];
  int first1;  // CTAs from here on work on g[1]
};
__global__ void __launch_bounds__(kSmallThreads, 1)
    k_gemm_small(const __grid_constant__ SmallP p, int* err, long long spin) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;
  uint8_t* sB = smem + kSmallStages * kABytes;
  __shared__ __align__(16) float scratch[8][kScratch];
  uint64_t* full = (uint64_t*)(smem + kSmallStages * (kABytes + kSBytes));
  uint64_t* empty = full + kSmallStages;
  uint64_t* tfull = empty + kSmallStages;
  uint32_t* tslot = (uint32_t*)(tfull + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_go();
  const int second = (int)blockIdx.x >= p.first1;
  const SmallG& g = p.g[second];
  const int item = (int)blockIdx.x - (second ? p.first1 : 0);
  const int mb = item % g.mt, nb = item / g.mt;
  const int kt_total = (g.K + BK - 1) / BK;
  uint32_t cols = 64;
  while (cols < (uint32_t)(g.splits * SN)) cols *= 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kSmallStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tfull, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(tslot)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {  // producer
      for (int kt = 0; kt < kt_total; ++kt) {
        const int s = kt % kSmallStages;
        if (kt >= kSmallStages && !mbar_wait(&empty[s], ((kt / kSmallStages) - 1) & 1, spin)) {
          atomicExch(err, 1);
          break;
        }
        mbar_expect_tx(&full[s], kABytes + kSBytes);
        tma_load_2d(sA + s * kABytes, &g.ta, kt * BK, mb * BM, &full[s]);
        tma_load_2d(sB + s * kSBytes, &g.tb, kt * BK, nb * SN, &full[s]);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer: split z accumulates in columns [64 z, 64 z + 64)
      const uint32_t id = idesc(SN);
      bool ok = true;
      uint32_t acc = tmem;
      for (int kt = 0, in = 0; kt < kt_total; ++kt, ++in) {
        if (in == g.kts) {
          in = 0;
          acc += SN;
        }
        const int s = kt % kSmallStages;
        if (!mbar_wait(&full[s], (kt / kSmallStages) & 1, spin)) {
          atomicExch(err, 1);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t pa = saddr(sA + s * kABytes), pb = saddr(sB + s * kSBytes);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk)
          mma_bf16(acc, sdesc(pa + 32 * kk), sdesc(pb + 32 * kk), id, (in > 0 || kk > 0) ? 1u : 0u);
        mma_commit(&empty[s]);
      }
      if (ok) mma_commit(tfull);
    }
  } else {
    // epilogue: warp w reads accumulator lanes (rows) 32 (w % 4) .. + 31, columns 32 ((w - 2) / 4) .. + 31
    const int q = warp & 3, c = 32 * ((warp - 2) >> 2);
    epi_consts(g.e, nb * SN + c, 32, scratch[warp - 2], 32);
    const bool ok = __all_sync(0xffffffffu, mbar_wait(tfull, 0, spin));
    if (!ok) {
      if (lane == 0) atomicExch(err, 1);
    } else {
      tc_fence_after();
      const int n0 = nb * SN + c;
      if (n0 < g.e.N) {
        float v[32];
        const uint32_t at = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c;
        tmem_ld32(at, v);
        for (int z = 1; z < g.splits; ++z) {
          float u[32];
          tmem_ld32(at + z * SN, u);
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] += u[j];
        }
        epi_block(g.e, mb * BM + q * 32, n0, v, 0, scratch[warp - 2], scratch[warp - 2], 32);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
  }
}

// sum of the K-split partial tiles, then the epilogue
__global__ void k_splitk(const float* ws, int splits, size_t stride, Epi e) {
  pdl_go();
  pdl_wait();
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t total = (size_t)e.M * e.N;
  if (i >= total) return;
  int m = (int)(i / e.N), n = (int)(i % e.N);
  float acc = 0.0f;
  for (int z = 0; z < splits; ++z) acc += ws[(size_t)z * stride + i];
  epi_one(e, m, n, acc);
}

// --------------------------------------------------------- other kernels
// layer-0 input: rows idx[r] of the raw data X (ld = d0), standardised,
// rounded to bfloat16, stored row-major and (AT not null) transposed; rows >=
// rows are 0.  32 x 32 tiles through shared memory, so that both stores
// coalesce (an element-wise kernel wrote the transpose 2 bytes per sector: 12
// us for 256 x 4000).  Grid ceil(d0 / 32) x (rows of A / 32), in one dimension,
// as the others end at 65,535; block 32 x 8.
__global__ void __launch_bounds__(256) k_input(const float* X, const int* idx, int rows, int Mb, int d0,
                                               const float* mu, const float* sd, bf16* A, bf16* AT) {
  __shared__ bf16 tile[32][34];
  pdl_go();
  pdl_wait();
  const int nt = (d0 + 31) / 32, j0 = (int)(blockIdx.x % nt) * 32, r0 = (int)(blockIdx.x / nt) * 32;
  const int j = j0 + threadIdx.x;
  const float m = j < d0 ? mu[j] : 0.0f, s = j < d0 ? sd[j] : 1.0f;
#pragma unroll
  for (int k = threadIdx.y; k < 32; k += 8) {
    const int r = r0 + k;
    float v = 0.0f;
    if (j < d0 && r < rows) {
      const size_t src = idx ? (size_t)idx[r] : (size_t)r;
      v = (X[src * d0 + j] - m) / s;
    }
    const bf16 h = __float2bfloat16_rn(v);
    if (j < d0) A[(size_t)r * d0 + j] = h;
    tile[k][threadIdx.x] = h;
  }
  if (!AT) return;
  __syncthreads();
#pragma unroll
  for (int k = threadIdx.y; k < 32; k += 8) {
    const int jj = j0 + k;
    if (jj < d0) AT[(size_t)jj * Mb + r0 + threadIdx.x] = tile[threadIdx.x][k];
  }
}

// Mean squared error against standardised targets: dY = 2 (Y - T) / (rows *
// N) in bfloat16, row-major and transposed, the output layer's bias gradient
// (the column sums of dY, in row order) and the loss.
//
// One block takes 64 columns over a run of rows, in tiles of 64 rows
// transposed through shared memory, each thread two neighbouring columns.
// Where the columns alone give every SM work (mse_run) the run is all rows and
// the block forms the bias gradient too; a narrow output layer is split over
// grid.y, and k_adam forms it from D' as it does for the hidden layers.  Time of
// a training step in one run and in several: 712 outputs, 16,384 rows 3.11 and
// 0.59 ms; 20,000 outputs, 1,024 rows 388 and 320 us; 712 outputs, 100 rows 88
// and 84 us.  The kernel is bound by its traffic (Y, T, D and D' once: 143 MB
// for 256 x 46,504).  The squares are summed in FP64, over the whole range of the FP32 errors; an error is widened
// in integer operations and takes one FP64 instruction (conversions, products
// and additions in FP64 took most of the former kernel's 100 us, and the
// column sums ran as a kernel of their own, 44 us).  Now 47 us for both.  The
// last block to finish adds the blocks' sums in a fixed order.
constexpr int kMseCols = 64, kMseRows = 64;
__global__ void __launch_bounds__(256) k_mse(const float* Y, const float* T, const int* idx, int rows, int Mb, int N,
                                             const float* mu, const float* sd, int run, bf16* D, bf16* DT, float* gb,
                                             double* part, unsigned* done, float* loss, float* loss_out) {
  __shared__ __align__(4) bf16 tile[kMseCols][kMseRows + 2];  // [column][row]
  __shared__ double red[256];
  __shared__ bool last;
  pdl_go();
  pdl_wait();
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;  // columns n0 + 2 x, + 1; rows y, y + 8, ...
  const int n0 = blockIdx.x * kMseCols, n = n0 + 2 * x;
  const bool in = n < N;  // N is a multiple of 8: both columns or none
  const bool vec = ((uintptr_t)T & 7) == 0;
  float2 m = make_float2(0.0f, 0.0f), s = make_float2(1.0f, 1.0f);
  if (in) {
    m = *(const float2*)(mu + n);
    s = *(const float2*)(sd + n);
  }
  const float den = (float)rows * (float)N;
  double sq[2][2] = {};  // of the thread's two columns, two chains of additions each
  float col = 0.0f;      // threads 0..63: the sum of column n0 + threadIdx.x
  const int r1 = min(Mb, ((int)blockIdx.y + 1) * run);
  for (int r0 = blockIdx.y * run; r0 < r1; r0 += kMseRows) {
#pragma unroll
    for (int k = 0; k < kMseRows; k += 8) {
      const int r = r0 + y + k;
      float2 g = make_float2(0.0f, 0.0f);
      if (in && r < rows) {
        const size_t src = idx ? (size_t)idx[r] : (size_t)r;
        const float* tp = T + src * N + n;
        const float2 t = vec ? *(const float2*)tp : make_float2(tp[0], tp[1]);
        const float2 yv = *(const float2*)(Y + (size_t)r * N + n);
        const float d0 = yv.x - (t.x - m.x) / s.x, d1 = yv.y - (t.y - m.y) / s.y;
        const double w0 = f64_widen(d0), w1 = f64_widen(d1);
        sq[k / 8 % 2][0] = fma(w0, w0, sq[k / 8 % 2][0]);
        sq[k / 8 % 2][1] = fma(w1, w1, sq[k / 8 % 2][1]);
        g = make_float2(2.0f * d0 / den, 2.0f * d1 / den);
      }
      const __nv_bfloat162 h = __floats2bfloat162_rn(g.x, g.y);
      if (in) *(__nv_bfloat162*)(D + (size_t)r * N + n) = h;
      tile[2 * x][y + k] = h.x;
      tile[2 * x + 1][y + k] = h.y;
    }
    __syncthreads();
    for (int c = y; c < kMseCols && n0 + c < N; c += 8)
      *(__nv_bfloat162*)(DT + (size_t)(n0 + c) * Mb + r0 + 2 * x) = *(const __nv_bfloat162*)&tile[c][2 * x];
    if (gb && threadIdx.x < kMseCols) {
#pragma unroll 8
      for (int r = 0; r < kMseRows; ++r) col += __bfloat162float(tile[threadIdx.x][r]);
    }
    __syncthreads();
  }
  if (gb && threadIdx.x < kMseCols && n0 + (int)threadIdx.x < N) gb[n0 + threadIdx.x] = col;
  auto sum = [&](double v) {
    red[threadIdx.x] = v;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
      if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
      __syncthreads();
    }
    return red[0];
  };
  const double mine = sum((sq[0][0] + sq[0][1]) + (sq[1][0] + sq[1][1]));
  if (threadIdx.x == 0) {
    part[blockIdx.y * gridDim.x + blockIdx.x] = mine;
    __threadfence();
    last = atomicAdd(done, 1u) == gridDim.x * gridDim.y - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double t = 0.0;
  for (int i = threadIdx.x; i < (int)(gridDim.x * gridDim.y); i += 256) t += ((volatile double*)part)[i];
  const double total = sum(t);
  if (threadIdx.x == 0) {
    const float v = (float)(total * (1.0 / ((double)rows * N)));
    *loss = v;
    if (loss_out) *loss_out = v;
    *done = 0u;  // for the next launch
  }
}

// rows per block of k_mse: all of them where that makes four blocks per SM, else
// as many runs of whole tiles as make up for it
static int mse_run(int N, int Mb, int sms) {
  const int cols = (N + kMseCols - 1) / kMseCols, tiles = Mb / kMseRows;
  const int runs = std::min(tiles, (4 * sms + cols - 1) / cols);
  return (tiles + runs - 1) / runs * kMseRows;
}

// Adam (bias-corrected) on every parameter of the network in one launch: FP32
// master weights W [out x in] with gradient G, the bfloat16 copies W16 [out x
// in] and W16T [in x out], and the biases, whose gradients of the hidden
// layers (the column sums of D, in row order) are formed here from D'.
//
// A weight block takes a 64 x 64 tile in 16-byte accesses, sixteen loads in
// flight per thread, and transposes the bfloat16 copy through shared memory.
// Bound by its traffic, 32 bytes per parameter: the 26.4 M parameters of the
// 2,000-bus network take 132 us against 220 with 4-byte accesses
// and one launch per layer (845 MB: 124 us at 6.8 TB/s).
constexpr int kMaxLayers = 16;
constexpr int kAdamTile = 64, kAdamBias = 64;  // tile edge; biases per block
struct AdamLayer {
  float *W, *G, *mW, *vW, *b, *gb, *mb, *vb;
  bf16 *W16, *W16T;
  const bf16* DT;  // D' [out x rows], null where gb is already formed
  int in, out;
  int block0, bias0;  // first weight block, first bias block
};
struct AdamP {
  AdamLayer l[kMaxLayers];
  int nl, rows;
  float lr, b1, b2, eps, c1, c2;
};
// the moments with the roundings written out, so that every instance of this
// function rounds alike
__device__ __forceinline__ float adam_one(const AdamP& p, float g, float& m, float& v, float w) {
  m = fmaf(1.0f - p.b1, g, __fmul_rn(p.b1, m));
  v = fmaf(__fmul_rn(1.0f - p.b2, g), g, __fmul_rn(p.b2, v));
  return w - p.lr * (m / p.c1) / (sqrtf(v / p.c2) + p.eps);
}
__global__ void __launch_bounds__(256) k_adam(const __grid_constant__ AdamP p) {
  __shared__ __align__(4) bf16 tile[kAdamTile][kAdamTile + 2];
  const int blk = blockIdx.x, t = threadIdx.x;
  pdl_go();
  pdl_wait();
  if (blk >= p.l[0].bias0) {
    int q = p.nl - 1;
    while (q > 0 && blk < p.l[q].bias0) --q;
    const AdamLayer& y = p.l[q];
    const int i = (blk - y.bias0) * kAdamBias + t;
    if (t >= kAdamBias || i >= y.out) return;
    float g = 0.0f;
    if (y.DT) {
      const uint4* src = (const uint4*)(y.DT + (size_t)i * p.rows);  // rows is a multiple of 128
#pragma unroll 8
      for (int k = 0; k < p.rows / 8; ++k) {
        const uint4 u = src[k];
        const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          g += __uint_as_float(w[h] << 16);
          g += __uint_as_float(w[h] & 0xffff0000u);
        }
      }
      y.gb[i] = g;
    } else {
      g = y.gb[i];
    }
    float m = y.mb[i], v = y.vb[i];
    y.b[i] = adam_one(p, g, m, v, y.b[i]);
    y.mb[i] = m;
    y.vb[i] = v;
    return;
  }
  int q = p.nl - 1;
  while (q > 0 && blk < p.l[q].block0) --q;
  const AdamLayer& y = p.l[q];
  const int nti = (y.in + kAdamTile - 1) / kAdamTile;
  const int i0 = (blk - y.block0) / nti * kAdamTile, j0 = (blk - y.block0) % nti * kAdamTile;
  const int jc = (t & 15) * 4, j = j0 + jc;  // in is a multiple of 8: four columns or none
  float4 W[4], G[4], M[4], V[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int i = i0 + (t >> 4) + 16 * k;
    if (i < y.out && j < y.in) {
      const size_t at = (size_t)i * y.in + j;
      W[k] = *(const float4*)(y.W + at);
      G[k] = *(const float4*)(y.G + at);
      M[k] = *(const float4*)(y.mW + at);
      V[k] = *(const float4*)(y.vW + at);
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int r = (t >> 4) + 16 * k, i = i0 + r;
    if (i < y.out && j < y.in) {
      const size_t at = (size_t)i * y.in + j;
      W[k].x = adam_one(p, G[k].x, M[k].x, V[k].x, W[k].x);
      W[k].y = adam_one(p, G[k].y, M[k].y, V[k].y, W[k].y);
      W[k].z = adam_one(p, G[k].z, M[k].z, V[k].z, W[k].z);
      W[k].w = adam_one(p, G[k].w, M[k].w, V[k].w, W[k].w);
      *(float4*)(y.mW + at) = M[k];
      *(float4*)(y.vW + at) = V[k];
      *(float4*)(y.W + at) = W[k];
      __nv_bfloat162 h[2] = {__floats2bfloat162_rn(W[k].x, W[k].y), __floats2bfloat162_rn(W[k].z, W[k].w)};
      *(uint2*)(y.W16 + at) = *(const uint2*)h;
      *(__nv_bfloat162*)&tile[r][jc] = h[0];
      *(__nv_bfloat162*)&tile[r][jc + 2] = h[1];
    }
  }
  __syncthreads();
  // W16T: two neighbouring outputs per lane (out is a multiple of 8)
  const int x = t & 31, i = i0 + 2 * x;
  if (i >= y.out) return;
#pragma unroll
  for (int k = t >> 5; k < kAdamTile; k += 8) {
    if (j0 + k >= y.in) break;
    __nv_bfloat162 h;
    h.x = tile[2 * x][k];
    h.y = tile[2 * x + 1][k];
    *(__nv_bfloat162*)(y.W16T + (size_t)(j0 + k) * y.out + i) = h;
  }
}

// bfloat16 copies of FP32 weights (after set_params)
__global__ void k_w16(const float* W, int out, int in, bf16* W16, bf16* W16T) {
  size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= (size_t)out * in) return;
  int i = (int)(p / in), j = (int)(p % in);
  bf16 h = __float2bfloat16_rn(W[p]);
  W16[p] = h;
  W16T[(size_t)j * out + i] = h;
}

// column means and population deviations (FP64 accumulation); a column whose
// deviation is at most 1e-12 (1 + |mean|) gets deviation 1
__global__ void k_standardiser(const float* X, int rows, int N, float* mu, float* sd) {
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  double s = 0.0;
  for (int r = 0; r < rows; ++r) s += (double)X[(size_t)r * N + n];
  double m = s / rows;
  double q = 0.0;
  for (int r = 0; r < rows; ++r) {
    double d = (double)X[(size_t)r * N + n] - m;
    q += d * d;
  }
  double dev = sqrt(q / rows);
  if (dev <= 1e-12 * (1.0 + fabs(m))) dev = 1.0;
  mu[n] = (float)m;
  sd[n] = (float)dev;
}

// ------------------------------------------------------------------ host side
static PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

static bool encode_fn() {
  if (g_encode) return true;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !fn)
    return false;
  g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
  return true;
}

// 2-D bfloat16 operand [rows x cols], row stride ld elements; boxes of box_rows rows x 64 columns
static bool make_map(CUtensorMap* m, const void* base, int rows, int cols, int ld, int box_rows) {
  if (!encode_fn()) return false;
  if (((uintptr_t)base & 15) || (ld * 2) % 16 || rows < 1 || cols < 1) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)base, dims, strides, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

struct Gemm {
  CUtensorMap ta, tb;
  int M, N, K, splits, kts;
  Epi e;
  bool small = false;  // run as k_gemm_small
  int bn = BN;         // rows of tb's boxes: 64 for k_gemm_small, else the tile width of k_gemm_tc
};

// launch with programmatic dependence on the kernel before it in the stream
template <typename... P, typename... A>
static cudaError_t launch(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... a) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, P(a)...);
}

// dynamic shared memory of the two kernels, once per device and thread of the caller
static cudaError_t set_smem() {
  static thread_local int done = -1;
  int dev = 0;
  cudaError_t c = cudaGetDevice(&dev);
  if (c != cudaSuccess || done == dev) return c;
  c = cudaFuncSetAttribute(k_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemmSmem);
  if (c == cudaSuccess)
    c = cudaFuncSetAttribute(k_gemm_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem);
  if (c == cudaSuccess) done = dev;
  return c;
}

// k_gemm_small pays while its tiles fit the GPU about twice, tensor memory
// holds every split, and the contraction, which one CTA walks alone at about
// 0.4 us per 64, stays short.  Both sides, as the time of a prediction whose
// other layers are small (this kernel / k_gemm_tc and k_splitk), 128 or 256
// rows: 512 outputs of 1,024 inputs 32 / 34 us, 1,536 inputs 35 / 34, 2,048
// inputs 42 / 33, 4,000 inputs 45 / 34; in tiles over SMs, 512 inputs, 1.25 35 /
// 44 us, 2 37 / 50, 2.5 42 / 34.
static bool fits_small(int M, int N, int K, int splits, int sms) {
  return splits <= kSmallSplits && K <= 24 * BK &&
         (long)((M + BM - 1) / BM) * ((N + SN - 1) / SN) <= 2L * sms;
}

static SmallG small_of(const Gemm& g) {
  SmallG s;
  s.ta = g.ta;
  s.tb = g.tb;
  s.K = g.K;
  s.kts = g.kts;
  s.splits = g.splits;
  s.mt = (g.e.M + BM - 1) / BM;
  s.e = g.e;
  return s;
}

// one or two products whose plan says small (b may be null)
static cudaError_t run_small(const Gemm& a, const Gemm* b, int* err, cudaStream_t st, long long spin) {
  cudaError_t c = set_smem();
  if (c != cudaSuccess) return c;
  SmallP p;
  p.g[0] = small_of(a);
  p.g[1] = b ? small_of(*b) : p.g[0];
  p.first1 = p.g[0].mt * ((a.N + SN - 1) / SN);
  const int grid = p.first1 + (b ? p.g[1].mt * ((b->N + SN - 1) / SN) : 0);
  return launch(k_gemm_small, grid, kSmallThreads, kSmallSmem, st, p, err, spin);
}

static cudaError_t run_gemm(const Gemm& g, float* ws, int* err, cudaStream_t st, long long spin, int sms) {
  if (g.small) return run_small(g, nullptr, err, st, spin);
  cudaError_t c = set_smem();
  if (c != cudaSuccess) return c;
  const int items = g.splits * ((g.e.M + BM - 1) / BM) * ((g.N + g.bn - 1) / g.bn);
  const int grid = items < sms ? items : sms;
  if (g.splits == 1) {
    return launch(k_gemm_tc, grid, kGemmThreads, kGemmSmem, st, g.ta, g.tb, g.K, g.kts, 1, g.bn, g.e, err, spin);
  }
  Epi p = g.e;
  p.op = EPI_PARTIAL;
  p.f32 = ws;
  p.ld_f32 = g.N;
  p.split_stride = (size_t)g.M * g.N;
  c = launch(k_gemm_tc, grid, kGemmThreads, kGemmSmem, st, g.ta, g.tb, g.K, g.kts, g.splits, g.bn, p, err, spin);
  if (c != cudaSuccess) return c;
  size_t total = (size_t)g.e.M * g.N;
  return launch(k_splitk, (unsigned)((total + 255) / 256), 256, 0, st, (const float*)ws, g.splits, p.split_stride, g.e);
}

// K split so that the grid covers the GPU's SMs about once
static void plan_split(Gemm& g, int sms) {
  int tiles = ((g.M + BM - 1) / BM) * ((g.N + BN - 1) / BN);
  int kt = (g.K + BK - 1) / BK;
  int s = 1;
  while (tiles * s * 2 <= sms && kt / (s * 2) >= 4) s *= 2;
  g.kts = (kt + s - 1) / s;
  g.splits = (kt + g.kts - 1) / g.kts;
}

static size_t ws_need(const Gemm& g) { return g.splits > 1 && !g.small ? (size_t)g.splits * g.M * g.N : 0; }

// Tile width of k_gemm_tc: the one whose waves of tiles cover the product with
// the least width per SM (a tile costs about its width plus 32 columns' worth
// of fixed time).  46,504 columns at one block of rows are 182 tiles of 256,
// two waves of which the second holds 30 tiles, but 1.9 waves of 160 (21.7 ->
// 9.1 us; at 256 rows 45 -> 32); wide products keep 256.  Taking the fixed time
// as 0 or 64 columns moves the time of networks with 20,000 to 60,000 outputs by
// 3 % at most either way; 256 throughout is up to 19 % slower.
static int tile_width(int M, int N, int splits, int sms) {
  int best = BN;
  long cost = 0;
  for (int bn = BN; bn >= 128; bn -= 32) {
    const long tiles = (long)splits * ((M + BM - 1) / BM) * ((N + bn - 1) / bn);
    const long c = (tiles + sms - 1) / sms * (bn + 32);
    if (bn == BN || c < cost) {
      cost = c;
      best = bn;
    }
  }
  return best;
}

// split and kernel of one of the network's products, and its operand maps
static bool plan_gemm(Gemm& g, const void* A, int lda, const void* B, int ldb, int sms) {
  plan_split(g, sms);
  g.small = fits_small(g.M, g.N, g.K, g.splits, sms);
  g.bn = g.small ? SN : tile_width(g.M, g.N, g.splits, sms);
  return make_map(&g.ta, A, g.M, g.K, lda, BM) && make_map(&g.tb, B, g.N, g.K, ldb, g.bn);
}

// --------------------------------------------------------------- the network
struct Layer {
  int in, out;
  float *W, *b, *mW, *vW, *mb, *vb, *gW, *gb;
  bf16 *W16, *W16T;
};

struct Net {
  int device = 0;
  int nl = 0;
  std::vector<int> dims;
  int Mb = 0;
  int sms = 0;
  cudaStream_t stream = nullptr;
  std::vector<Layer> L;
  // parameters and gradients, each in one block in the order of the C ABI (W_0,
  // b_0, W_1, ...), so that a read-out is one copy: layer by layer, the driver
  // took up to 90 ms for the 105 MB of the 2,000-bus network where the pieces
  // met the host's pages unfavourably, against 5 ms in one piece
  float *params = nullptr, *grads = nullptr;
  size_t nparams = 0;
  // activations: A[l] / AT[l] layer inputs (l = 0..nl-1), Z[l] pre-activations of hidden layer l (1..nl-1)
  std::vector<bf16*> A, AT;
  std::vector<float*> Z;
  float* Y = nullptr;
  // gradients of layer outputs: D[l] / DT[l], l = 1..nl (D[nl] = dL/dY)
  std::vector<bf16*> D, DT;
  float *mu_x = nullptr, *sd_x = nullptr, *mu_y = nullptr, *sd_y = nullptr;
  float* ws = nullptr;
  size_t ws_elems = 0;
  double* part = nullptr;
  int nparts = 0, mse_run = 0;  // column blocks and rows per block of k_mse
  unsigned* done = nullptr;  // blocks of k_mse that have finished (0 between launches)
  int* err = nullptr;
  float* loss = nullptr;
  int step = 0;
  Gemm head;  // the output layer at one block of rows (inference of at most 128 rows)
  std::vector<Gemm> fwd, bwd_w, bwd_x;  // fwd[l], bwd_w[l] (dW_l), bwd_x[l] (dA_l, l >= 1)
  std::vector<void*> allocs;
  std::string last_error;
  long long spin = 1ll << 32;
};

template <typename T>
static bool dalloc(Net* n, T** p, size_t count) {
  void* q = nullptr;
  if (cudaMalloc(&q, count * sizeof(T) + 16) != cudaSuccess) return false;
  cudaMemset(q, 0, count * sizeof(T) + 16);
  n->allocs.push_back(q);
  *p = (T*)q;
  return true;
}

static void free_net(Net* n) {
  for (void* p : n->allocs) cudaFree(p);
  n->allocs.clear();
}

static acopf_status nfail(Net* n, acopf_status s, const std::string& m) {
  if (n) n->last_error = m;
  return s;
}

static bool plan(Net* n) {
  const int nl = n->nl, Mb = n->Mb;
  n->fwd.assign(nl, Gemm{});
  n->bwd_w.assign(nl, Gemm{});
  n->bwd_x.assign(nl, Gemm{});
  size_t ws = 0;
  for (int l = 0; l < nl; ++l) {
    const int in = n->dims[l], out = n->dims[l + 1];
    Layer& y = n->L[l];
    // forward: [Mb x in] * W[out x in]^T
    Gemm& f = n->fwd[l];
    f.M = Mb; f.N = out; f.K = in;
    if (!plan_gemm(f, n->A[l], in, y.W16, in, n->sms)) return false;
    memset(&f.e, 0, sizeof(Epi));
    f.e.M = Mb; f.e.N = out; f.e.rows_valid = Mb; f.e.bias = y.b;
    if (l < nl - 1) {
      f.e.op = EPI_GELU;
      f.e.f32 = n->Z[l + 1]; f.e.ld_f32 = out;
      f.e.bf = n->A[l + 1]; f.e.ld_bf = out;
      f.e.bt = n->AT[l + 1]; f.e.ld_bt = Mb;
    } else {
      f.e.op = EPI_F32;
      f.e.f32 = n->Y; f.e.ld_f32 = out;
    }
    ws = ws > ws_need(f) ? ws : ws_need(f);
    if (l == nl - 1) {
      // the same product for one block of rows: other tile widths fill the GPU; the split stays, it fixes the rounding
      n->head = f;
      if (!f.small) {
        n->head.bn = tile_width(BM, out, f.splits, n->sms);
        if (!make_map(&n->head.tb, y.W16, out, in, in, n->head.bn)) return false;
      }
    }
    // weight gradient: dW = D^T [out x Mb] * (A^T [in x Mb])^T
    Gemm& w = n->bwd_w[l];
    w.M = out; w.N = in; w.K = Mb;
    if (!plan_gemm(w, n->DT[l + 1], Mb, n->AT[l], Mb, n->sms)) return false;
    memset(&w.e, 0, sizeof(Epi));
    w.e.op = EPI_F32; w.e.M = out; w.e.N = in; w.e.rows_valid = out;
    w.e.f32 = y.gW; w.e.ld_f32 = in;
    ws = ws > ws_need(w) ? ws : ws_need(w);
    if (l >= 1) {
      // input gradient: D_l = (D_{l+1} [Mb x out] * (W16T [in x out])^T) * GELU'(Z_l)
      Gemm& x = n->bwd_x[l];
      x.M = Mb; x.N = in; x.K = out;
      if (!plan_gemm(x, n->D[l + 1], out, y.W16T, out, n->sms)) return false;
      memset(&x.e, 0, sizeof(Epi));
      x.e.op = EPI_GELU_BWD; x.e.M = Mb; x.e.N = in; x.e.rows_valid = Mb;
      x.e.z = n->Z[l]; x.e.ld_z = in;
      x.e.bf = n->D[l]; x.e.ld_bf = in;
      x.e.bt = n->DT[l]; x.e.ld_bt = Mb;
      ws = ws > ws_need(x) ? ws : ws_need(x);
    }
  }
  n->ws_elems = ws;
  return ws == 0 || dalloc(n, &n->ws, ws);
}

static acopf_status check_err(Net* n) {
  int e = 0;
  if (cudaMemcpyAsync(&e, n->err, sizeof(int), cudaMemcpyDeviceToHost, n->stream) != cudaSuccess ||
      cudaStreamSynchronize(n->stream) != cudaSuccess)
    return nfail(n, ACOPF_ECUDA, std::string("cuda: ") + cudaGetErrorString(cudaGetLastError()));
  if (e) {
    cudaMemsetAsync(n->err, 0, sizeof(int), n->stream);
    return nfail(n, ACOPF_ETIMEOUT, "tensor-core GEMM: a pipeline wait ran out");
  }
  return ACOPF_OK;
}

#define NCK(x)                                                                          \
  do {                                                                                  \
    cudaError_t _e = (x);                                                               \
    if (_e != cudaSuccess) return nfail(n, ACOPF_ECUDA, std::string("cuda: ") + cudaGetErrorString(_e)); \
  } while (0)

// the network on the rows of A[0].  Training (out null): pre-activations,
// transposes and Y, all Mb rows.  Inference: the row blocks that hold rows,
// only what the next layer reads, and the de-standardised outputs of the valid
// rows straight into out.
static acopf_status forward(Net* n, int rows, float* out = nullptr) {
  for (int l = 0; l < n->nl; ++l) {
    Gemm g = out && l == n->nl - 1 && rows <= BM ? n->head : n->fwd[l];
    g.e.rows_valid = rows;
    if (out) {
      if (l < n->nl - 1) {
        g.e.M = (rows + BM - 1) / BM * BM;
        g.e.f32 = nullptr;
        g.e.bt = nullptr;
      } else {
        g.e.M = rows;
        g.e.f32 = out;
        g.e.mu = n->mu_y;
        g.e.sd = n->sd_y;
      }
    }
    NCK(run_gemm(g, n->ws, n->err, n->stream, n->spin, n->sms));
  }
  return ACOPF_OK;
}

}  // namespace nn
}  // namespace acopf

using namespace acopf::nn;

extern "C" {

acopf_status acopf_mlp_create(const int32_t* dims, int32_t nlayers, int32_t max_batch, int32_t device,
                              acopf_mlp_handle* out) {
  if (!dims || !out || nlayers < 1 || nlayers > 16 || max_batch < 1) return ACOPF_EINVAL;
  *out = nullptr;
  for (int l = 0; l <= nlayers; ++l)
    if (dims[l] < 8 || dims[l] % 8) return ACOPF_EINVAL;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
    cudaGetLastError();
    return ACOPF_ECUDA;
  }
  if (cudaSetDevice(device) != cudaSuccess) return ACOPF_ECUDA;
  int major = 0;
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device);
  if (major < 10) return ACOPF_ECUDA;
  Net* n = new Net();
  n->device = device;
  n->nl = nlayers;
  n->dims.assign(dims, dims + nlayers + 1);
  n->Mb = ((max_batch + BM - 1) / BM) * BM;
  cudaDeviceGetAttribute(&n->sms, cudaDevAttrMultiProcessorCount, device);
  const int Mb = n->Mb;
  bool ok = true;
  n->L.resize(nlayers);
  for (int l = 0; l < nlayers; ++l) n->nparams += (size_t)dims[l] * dims[l + 1] + dims[l + 1];
  ok = dalloc(n, &n->params, n->nparams) && dalloc(n, &n->grads, n->nparams);
  for (size_t l = 0, off = 0; l < n->L.size() && ok; ++l) {
    Layer& y = n->L[l];
    y.in = dims[l];
    y.out = dims[l + 1];
    const size_t w = (size_t)y.in * y.out;
    y.W = n->params + off;  // widths are multiples of 8: every part is 32-byte aligned
    y.b = y.W + w;
    y.gW = n->grads + off;
    y.gb = y.gW + w;
    off += w + y.out;
    ok = dalloc(n, &y.mW, w) && dalloc(n, &y.vW, w) && dalloc(n, &y.mb, y.out) && dalloc(n, &y.vb, y.out) &&
         dalloc(n, &y.W16, w) && dalloc(n, &y.W16T, w);
  }
  n->A.assign(nlayers, nullptr);
  n->AT.assign(nlayers, nullptr);
  n->Z.assign(nlayers, nullptr);
  n->D.assign(nlayers + 1, nullptr);
  n->DT.assign(nlayers + 1, nullptr);
  for (int l = 0; l < nlayers && ok; ++l) {
    ok = dalloc(n, &n->A[l], (size_t)Mb * dims[l]) && dalloc(n, &n->AT[l], (size_t)Mb * dims[l]);
    if (ok && l >= 1) ok = dalloc(n, &n->Z[l], (size_t)Mb * dims[l]);
  }
  for (int l = 1; l <= nlayers && ok; ++l)
    ok = dalloc(n, &n->D[l], (size_t)Mb * dims[l]) && dalloc(n, &n->DT[l], (size_t)Mb * dims[l]);
  ok = ok && dalloc(n, &n->Y, (size_t)Mb * dims[nlayers]) && dalloc(n, &n->mu_x, dims[0]) &&
       dalloc(n, &n->sd_x, dims[0]) && dalloc(n, &n->mu_y, dims[nlayers]) && dalloc(n, &n->sd_y, dims[nlayers]) &&
       dalloc(n, &n->err, 1) && dalloc(n, &n->loss, 1);
  if (ok) {
    n->nparts = (dims[nlayers] + kMseCols - 1) / kMseCols;
    n->mse_run = mse_run(dims[nlayers], Mb, n->sms);
    ok = dalloc(n, &n->part, (size_t)n->nparts * ((Mb + n->mse_run - 1) / n->mse_run)) && dalloc(n, &n->done, 1);
  }
  if (ok) {
    // identity standardisation until fitted
    std::vector<float> one((size_t)(dims[0] > dims[nlayers] ? dims[0] : dims[nlayers]), 1.0f);
    ok = cudaMemcpy(n->sd_x, one.data(), sizeof(float) * dims[0], cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(n->sd_y, one.data(), sizeof(float) * dims[nlayers], cudaMemcpyHostToDevice) == cudaSuccess;
  }
  // zeros and ones were written on the default stream, which the network's need not wait for
  if (!ok || !plan(n) || cudaStreamSynchronize(nullptr) != cudaSuccess) {
    free_net(n);
    delete n;
    cudaGetLastError();
    return ACOPF_ENOMEM;
  }
  *out = (acopf_mlp_handle)n;
  return ACOPF_OK;
}

acopf_status acopf_mlp_destroy(acopf_mlp_handle h) {
  Net* n = (Net*)h;
  if (!n) return ACOPF_EINVAL;
  cudaSetDevice(n->device);
  if (n->stream) cudaStreamSynchronize(n->stream);
  free_net(n);
  delete n;
  return ACOPF_OK;
}

acopf_status acopf_mlp_set_stream(acopf_mlp_handle h, void* stream) {
  Net* n = (Net*)h;
  if (!n) return ACOPF_EINVAL;
  n->stream = (cudaStream_t)stream;
  return ACOPF_OK;
}

acopf_status acopf_mlp_last_error(acopf_mlp_handle h, char* buf, size_t len) {
  Net* n = (Net*)h;
  if (!n || !buf || len == 0) return ACOPF_EINVAL;
  snprintf(buf, len, "%s", n->last_error.c_str());
  return ACOPF_OK;
}

acopf_status acopf_mlp_num_params(acopf_mlp_handle h, int64_t* count) {
  Net* n = (Net*)h;
  if (!n || !count) return ACOPF_EINVAL;
  *count = (int64_t)n->nparams;
  return ACOPF_OK;
}

static acopf_status copy_params(Net* n, float* host, int64_t count, bool to_device, bool grads) {
  if (!host || count != (int64_t)n->nparams) return nfail(n, ACOPF_EINVAL, "parameter count mismatch");
  cudaSetDevice(n->device);
  NCK(cudaStreamSynchronize(n->stream));
  float* dev = grads ? n->grads : n->params;
  const size_t bytes = sizeof(float) * n->nparams;
  // on the network's stream, before the kernels that read it; set_params waits
  if (to_device) NCK(cudaMemcpyAsync(dev, host, bytes, cudaMemcpyHostToDevice, n->stream));
  else NCK(cudaMemcpy(host, dev, bytes, cudaMemcpyDeviceToHost));
  return ACOPF_OK;
}

acopf_status acopf_mlp_set_params(acopf_mlp_handle h, const float* params, int64_t count) {
  Net* n = (Net*)h;
  if (!n) return ACOPF_EINVAL;
  acopf_status s = copy_params(n, (float*)params, count, true, false);
  if (s) return s;
  for (auto& y : n->L) {
    size_t w = (size_t)y.in * y.out;
    k_w16<<<(unsigned)((w + 255) / 256), 256, 0, n->stream>>>(y.W, y.out, y.in, y.W16, y.W16T);
    NCK(cudaMemsetAsync(y.mW, 0, sizeof(float) * w, n->stream));
    NCK(cudaMemsetAsync(y.vW, 0, sizeof(float) * w, n->stream));
    NCK(cudaMemsetAsync(y.mb, 0, sizeof(float) * y.out, n->stream));
    NCK(cudaMemsetAsync(y.vb, 0, sizeof(float) * y.out, n->stream));
  }
  n->step = 0;
  NCK(cudaGetLastError());
  NCK(cudaStreamSynchronize(n->stream));
  return ACOPF_OK;
}

acopf_status acopf_mlp_get_params(acopf_mlp_handle h, float* params, int64_t count) {
  Net* n = (Net*)h;
  if (!n) return ACOPF_EINVAL;
  return copy_params(n, params, count, false, false);
}

acopf_status acopf_mlp_get_grads(acopf_mlp_handle h, float* grads, int64_t count) {
  Net* n = (Net*)h;
  if (!n) return ACOPF_EINVAL;
  return copy_params(n, grads, count, false, true);
}

acopf_status acopf_mlp_fit_standardiser(acopf_mlp_handle h, const float* X, const float* Y, int32_t rows) {
  Net* n = (Net*)h;
  if (!n || !X || !Y || rows < 1) return nfail(n, ACOPF_EINVAL, "fit_standardiser: bad arguments");
  cudaSetDevice(n->device);
  const int d0 = n->dims[0], dn = n->dims[n->nl];
  k_standardiser<<<(d0 + 127) / 128, 128, 0, n->stream>>>(X, rows, d0, n->mu_x, n->sd_x);
  k_standardiser<<<(dn + 127) / 128, 128, 0, n->stream>>>(Y, rows, dn, n->mu_y, n->sd_y);
  NCK(cudaGetLastError());
  NCK(cudaStreamSynchronize(n->stream));
  return ACOPF_OK;
}

acopf_status acopf_mlp_get_standardiser(acopf_mlp_handle h, float* mu_x, float* sd_x, float* mu_y, float* sd_y) {
  Net* n = (Net*)h;
  if (!n) return ACOPF_EINVAL;
  cudaSetDevice(n->device);
  NCK(cudaStreamSynchronize(n->stream));
  const int d0 = n->dims[0], dn = n->dims[n->nl];
  if (mu_x) NCK(cudaMemcpy(mu_x, n->mu_x, sizeof(float) * d0, cudaMemcpyDeviceToHost));
  if (sd_x) NCK(cudaMemcpy(sd_x, n->sd_x, sizeof(float) * d0, cudaMemcpyDeviceToHost));
  if (mu_y) NCK(cudaMemcpy(mu_y, n->mu_y, sizeof(float) * dn, cudaMemcpyDeviceToHost));
  if (sd_y) NCK(cudaMemcpy(sd_y, n->sd_y, sizeof(float) * dn, cudaMemcpyDeviceToHost));
  return ACOPF_OK;
}

acopf_status acopf_mlp_forward(acopf_mlp_handle h, const float* X, int32_t rows, float* Y) {
  Net* n = (Net*)h;
  if (!n || !X || !Y || rows < 1) return nfail(n, ACOPF_EINVAL, "mlp_forward: bad arguments");
  cudaSetDevice(n->device);
  const int d0 = n->dims[0], dn = n->dims[n->nl];
  for (int r0 = 0; r0 < rows; r0 += n->Mb) {
    int rr = rows - r0 < n->Mb ? rows - r0 : n->Mb;
    NCK(launch(k_input, (d0 + 31) / 32 * ((rr + BM - 1) / BM * (BM / 32)), dim3(32, 8), 0, n->stream,
               X + (size_t)r0 * d0, (const int*)nullptr, rr, n->Mb, d0, n->mu_x, n->sd_x, n->A[0], (bf16*)nullptr));
    acopf_status s = forward(n, rr, Y + (size_t)r0 * dn);
    if (s) return s;
  }
  return check_err(n);
}

acopf_status acopf_mlp_train_step(acopf_mlp_handle h, const float* X, const float* T, const int32_t* idx,
                                  int32_t rows, float lr, float* loss) {
  Net* n = (Net*)h;
  if (!n || !X || !T || rows < 1 || rows > n->Mb || !(lr > 0)) return nfail(n, ACOPF_EINVAL, "mlp_train_step: bad arguments");
  cudaSetDevice(n->device);
  const int nl = n->nl, Mb = n->Mb, d0 = n->dims[0], dn = n->dims[nl];
  NCK(launch(k_input, (d0 + 31) / 32 * (Mb / 32), dim3(32, 8), 0, n->stream, X, idx, rows, Mb, d0, n->mu_x,
             n->sd_x, n->A[0], n->AT[0]));
  acopf_status s = forward(n, rows);
  if (s) return s;
  // k_mse stores the loss where it is asked for if that is aligned memory of this
  // device; anything else is left to a copy, which takes or refuses it
  bool direct = loss && ((uintptr_t)loss & 3) == 0;
  if (direct) {
    cudaPointerAttributes at{};
    direct = cudaPointerGetAttributes(&at, loss) == cudaSuccess &&
             (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged) && at.device == n->device;
    if (!direct) cudaGetLastError();
  }
  const bool whole = n->mse_run >= Mb;  // one run: k_mse forms the output layer's bias gradient
  NCK(launch(k_mse, dim3(n->nparts, (Mb + n->mse_run - 1) / n->mse_run), 256, 0, n->stream, n->Y, T, idx, rows, Mb, dn,
             n->mu_y, n->sd_y, n->mse_run, n->D[nl], n->DT[nl], whole ? n->L[nl - 1].gb : (float*)nullptr, n->part,
             n->done, n->loss, direct ? loss : (float*)nullptr));
  for (int l = nl - 1; l >= 0; --l) {
    const Gemm &w = n->bwd_w[l], &x = n->bwd_x[l];
    if (l >= 1 && w.small && x.small) {
      NCK(run_small(w, &x, n->err, n->stream, n->spin));
      continue;
    }
    NCK(run_gemm(w, n->ws, n->err, n->stream, n->spin, n->sms));
    if (l >= 1) NCK(run_gemm(x, n->ws, n->err, n->stream, n->spin, n->sms));
  }
  n->step += 1;
  AdamP p;
  p.nl = nl;
  p.rows = Mb;
  p.lr = lr; p.b1 = 0.9f; p.b2 = 0.999f; p.eps = 1e-8f;
  p.c1 = (float)(1.0 - pow(0.9, n->step));
  p.c2 = (float)(1.0 - pow(0.999, n->step));
  int blocks = 0;
  auto tiles = [](int w) { return (w + kAdamTile - 1) / kAdamTile; };
  for (int l = 0; l < nl; ++l) {
    const Layer& y = n->L[l];
    p.l[l] = AdamLayer{y.W, y.gW, y.mW, y.vW, y.b, y.gb, y.mb, y.vb, y.W16, y.W16T,
                       l < nl - 1 || !whole ? n->DT[l + 1] : nullptr, y.in, y.out, blocks, 0};
    blocks += tiles(y.in) * tiles(y.out);
  }
  for (int l = 0; l < nl; ++l) {
    p.l[l].bias0 = blocks;
    blocks += (n->L[l].out + kAdamBias - 1) / kAdamBias;
  }
  NCK(launch(k_adam, blocks, 256, 0, n->stream, p));
  if (loss && !direct) NCK(cudaMemcpyAsync(loss, n->loss, sizeof(float), cudaMemcpyDeviceToDevice, n->stream));
  return ACOPF_OK;
}

acopf_status acopf_mlp_sync(acopf_mlp_handle h) {
  Net* n = (Net*)h;
  if (!n) return ACOPF_EINVAL;
  cudaSetDevice(n->device);
  return check_err(n);
}

// C[M x N] = A[M x K] B[N x K]^T: bfloat16 operands (row stride K), FP32 output
// (row stride N), all device pointers; on the given stream, synchronised.
acopf_status acopf_gemm_bf16(const void* A, const void* B, float* C, int32_t M, int32_t N, int32_t K, int32_t splits,
                             void* stream, float* ms) {
  if (!A || !B || !C || M < 1 || N < 1 || K < 8 || K % 8) return ACOPF_EINVAL;
  Gemm g{};
  g.M = M; g.N = N; g.K = K;
  int kt = (K + BK - 1) / BK;
  int s = splits < 1 ? 1 : (splits > kt ? kt : splits);
  g.kts = (kt + s - 1) / s;
  g.splits = (kt + g.kts - 1) / g.kts;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  g.bn = tile_width(M, N, g.splits, sms);
  if (!make_map(&g.ta, A, M, K, K, BM) || !make_map(&g.tb, B, N, K, K, g.bn)) return ACOPF_EINVAL;
  g.e.op = EPI_F32; g.e.M = M; g.e.N = N; g.e.rows_valid = M; g.e.f32 = C; g.e.ld_f32 = N;
  cudaStream_t st = (cudaStream_t)stream;
  float* ws = nullptr;
  int* err = nullptr;
  if (cudaMalloc(&err, sizeof(int)) != cudaSuccess) return ACOPF_ENOMEM;
  cudaMemsetAsync(err, 0, sizeof(int), st);
  if (g.splits > 1 && cudaMalloc(&ws, sizeof(float) * (size_t)g.splits * M * N) != cudaSuccess) {
    cudaFree(err);
    return ACOPF_ENOMEM;
  }
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (ms) {
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, st);
  }
  cudaError_t e = run_gemm(g, ws, err, st, 1ll << 32, sms);
  if (ms) cudaEventRecord(e1, st);
  int hv = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hv, err, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (ms) {
    *ms = 0.0f;
    if (e == cudaSuccess) cudaEventElapsedTime(ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
  }
  if (ws) cudaFree(ws);
  cudaFree(err);
  if (e != cudaSuccess) return ACOPF_ECUDA;
  return hv ? ACOPF_ETIMEOUT : ACOPF_OK;
}

}  // extern "C"


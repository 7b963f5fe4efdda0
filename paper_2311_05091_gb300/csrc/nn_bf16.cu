// Kernels of the learned warm start: a small convolutional encoder-decoder
// that maps (solid indicator, initial phase field, cos theta) to a phase field
// close to equilibrium, followed by plain lattice Boltzmann relaxation.  The
// network is not part of the paper; it is a throughput device for the
// method (the paper's steps still decide the final state).
//
// Tensors are NHWC float32 in memory (pixel p = (n h + y) w + x, channel
// innermost).  3x3 convolutions run on the tensor cores with BF16 operands
// and FP32 accumulation: the forward (and data-gradient) convolution with
// tcgen05.mma and a TMEM accumulator, the weight gradient likewise with
// both operands MN-major; activations are rounded to BF16 as they enter a convolution,
// weights are kept as a BF16 copy of FP32 master weights.  Weight layout: wt[tap][cout][cin], tap = 3 ky + kx, so a
// pair of input channels is one 32-bit word.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>

#include "../../include/lbm_nn.h"
#include "nn_plan.cuh"
#include "nn_wait.cuh"

namespace {

using namespace lbm_nn;

constexpr int kThreads = 128;
constexpr int kProjectPasses = 3;   // mass-correction passes of lbm_nn_project

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// ---------------------------------------------------------------------------
// forward: y[p][co] = act(b[co] + sum_{tap, ci} x[p + shift(tap)][ci] wt[tap][co][ci])
//
// Implicit GEMM on the 5th-generation tensor cores: D (128 positions x N output channels, FP32 in TMEM) +=
// A_tap (128 x 16 input channels, BF16) * B_tap^T (N x 16) for every chunk of 16 input channels and, inside it, the
// nine taps (this order fixes the rounding of the sums).
//
// Positions, not pixels.  A work item is a block of R image rows x Wt columns, staged with one halo row above and
// below and one halo column on each side as a flat sequence of positions of pitch Wt + 2, zero outside the image.
// Output position m = row * pitch + column reads position m + ky * pitch + kx for tap (ky, kx), so one staged copy
// serves all nine taps of any image width: the A operand of a tap is the window of 128 consecutive positions that
// starts ky * pitch + kx positions further, in the canonical K-major layout without swizzle (16 bytes per position
// and 8-channel group; core matrices 128 bytes apart along M, channel groups LBO apart).  The two outputs per row
// that fall on the halo columns are dropped (3 % of the products at Wt = 64).  The images of the batch are one tall
// image with a zero row between them, so blocks of rows run across image borders.
//
// One persistent CTA per SM, three roles that run concurrently:
//   producers:  load FP32 activations, 32 bytes per thread, round to BF16 into the stage (16-byte stores, free of bank conflicts); one thread starts
//               the TMA copy of the stage's weights, [tap][co][KC channels] in the matching 64- or 32-byte swizzle;
//   products:   one thread issues the tcgen05.mma of a stage and commits them to the barrier that frees it;
//   epilogue:   reads a finished accumulator (tcgen05.ld), adds the bias, applies the ReLU, transposes through
//               shared memory and stores whole 128-byte lines.
// Stages of KC channels form a ring over items; the accumulators have two sets, so an item's products overlap the
// previous item's epilogue.  Every barrier wait is bounded (nn_wait.cuh); a give-up sets g_nn_fault and ends the CTA.
//
// What bounds it: the wide levels HBM (403 MB for 64 -> 32 on 16 x 256^2: 60 us at copy speed), the deep ones shared
// memory (an M = 128, K = 16 product reads 4 KB of A, 32 cycles, whatever N) and the pipeline's latency per stage.
// Measured (GB300, 16 images; the kernel before staged every tile between two CTA barriers, without overlap):
// 64 -> 32 on 256^2 331 -> 105 us, 128 -> 128 on 64^2 137 -> 33 us, 256 -> 256 on 32^2 101 -> 31 us, one image of the
// last 54 -> 15 us.  12 producer warps with four 32-byte loads each in flight: 816 us over the network's seventeen
// forward and data-gradient shapes, against 837 with 8 warps and 827 with 16; loads issued one batch ahead gave
// nothing, and neither did stores of a lane's own 128-byte line without the transposition (860: slower from 64
// output channels on).
// ---------------------------------------------------------------------------
__device__ unsigned int g_nn_fault = 0;    // set when a bounded wait on the tensor cores gave up

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptors as two words.  Low: start address and leading offset, both in 16 bytes; a later
// start is an addition (shared memory has fewer than 2^14 units).  High: stride offset, version 1, swizzle.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo) { return (addr >> 4) | ((lbo >> 4) << 16); }
__device__ __forceinline__ uint32_t desc_hi(uint32_t sbo) { return (sbo >> 4) | (1u << 14); }
// K-major rows of `row` bytes (32 or 64) in TMA's swizzle of that width, rows contiguous: 8-row groups 8 row bytes
// apart; a later K = 16 slice of the row starts 32 bytes further
template <int row>
__device__ __forceinline__ uint32_t desc_hi_sw() {
  static_assert(row == 32 || row == 64, "swizzle widths used here");
  return desc_hi(8 * row) | ((row == 64 ? 4u : 6u) << 29);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major, M x N
__host__ __device__ constexpr uint32_t umma_idesc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// D (TMEM) = or += A B^T, one K = 16 product of kind::f16, issued by the lane with `leader` set.  The whole warp runs
// the code around it, so that descriptors stay in uniform registers: with a branch on the lane, the chain of integer
// instructions of the one thread, not the tensor cores, set the pace of the products.
__device__ __forceinline__ void umma_f16(uint32_t d, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi, uint32_t idesc,
                                         uint32_t accumulate, uint32_t leader) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b64 a, b;\n setp.ne.b32 p, %6, 0;\n setp.ne.b32 q, %7, 0;\n mov.b64 a, {%1, %2};\n"
      " mov.b64 b, {%3, %4};\n @q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n" ::"r"(d),
      "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(accumulate), "r"(leader));
}

// the products issued so far by the leader arrive on an mbarrier when they are done
__device__ __forceinline__ void umma_commit(uint32_t bar, uint32_t leader) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar),
      "r"(leader));
}

// eight floats from a 32-byte boundary, through the read-only path
__device__ __forceinline__ void ldg8(const float* p, float* r) {
  asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
               : "l"(p));
}

struct FwdArgs {
  const float* x;
  const float* bias;
  float* y;
  int n, h, w, cin, cout, relu;
  FwdPlan p;
};

template <int N, int KC>
__global__ void __launch_bounds__(kCvThreads, 1)
    conv3x3_fwd(const FwdArgs a, const __grid_constant__ CUtensorMap wmap) {
  extern __shared__ __align__(1024) unsigned char smem[];
  constexpr int KG = KC / 8;                        // channel groups per stage
  constexpr int kW = 9 * N * KC * 2;                // bytes of a stage's weights
  const FwdPlan& p = a.p;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int S = p.stages;
  // barriers: activations staged[S], weights landed[S], stage free[S], accumulator ready[2], accumulator free[2]
  const uint32_t b_full = smem_addr(smem), b_w = b_full + 8 * kCvMaxStages, b_empty = b_w + 8 * kCvMaxStages,
                 b_acc = b_empty + 8 * kCvMaxStages, b_free = b_acc + 16;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + 24 * kCvMaxStages + 32);
  float* tbuf = reinterpret_cast<float*>(smem + 512);
  unsigned char* stage0 = smem + kCvHead;

  if (warp == kCvMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tslot)),
                 "r"(p.tmem));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int k = 0; k < S; ++k) {
      mbar_init(b_full + 8 * k, 32 * kCvProd);
      mbar_init(b_w + 8 * k, 1);
      mbar_init(b_empty + 8 * k, 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(b_acc + 8 * k, 1);
      mbar_init(b_free + 8 * k, 32 * kCvEpi);
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(tslot);

  const int ntile = a.cout / N;
  const int nst = a.cin / KC;
  const int rows_all = a.n * (a.h + 1) - 1;         // rows of the tall image
  bool ok = true;

  if (warp > kCvMma) {
    // ---- producers ----
    PosMap pm{p.mp, p.mh, p.pitch, a.h, a.w};
    const int tp = tid - 32 * (kCvMma + 1);
    constexpr int TP = 32 * kCvProd;
    constexpr int PP = TP / KG;                     // positions per pass of the producer threads
    const int kg = tp % KG, q0 = tp / KG;
    int it = 0;                                     // stage count over all items
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x) {
      const int ct = item % ntile, rest = item / ntile;
      const int row0 = rest / p.strips * p.R;
      const int NP = (min(p.R, rows_all - row0) + 2) * p.pitch;
      // the halo row above the first image is the zero row of an image before it
      pm.block(row0 + a.h, rest % p.strips * p.Wt - 1);
      pm.img0 -= 1;
      for (int s = 0; s < nst; ++s, ++it) {
        const int st = it % S;
        unsigned char* sw = stage0 + st * p.stage_bytes;
        if (it >= S && !mbar_wait(b_empty + 8 * st, (uint32_t)((it / S - 1) & 1))) {
          ok = false;
          break;
        }
        if (tp == 0) {                              // the weights of the nine taps: one TMA tile
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(b_w + 8 * st), "r"(kW)
                       : "memory");
          asm volatile(
              "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
              "%4}], [%5];\n" ::"r"(smem_addr(sw)),
              "l"(reinterpret_cast<unsigned long long>(&wmap)), "r"(s * KC), "r"(ct * N), "r"(0), "r"(b_w + 8 * st)
              : "memory");
        }
        const float* src = a.x + s * KC + 8 * kg;
        unsigned char* dst = sw + kW + kg * p.Pn * 16;
        for (int q = q0; q < NP; q += PP * kCvBatch) {
          float4 v[kCvBatch][2];
#pragma unroll
          for (int u = 0; u < kCvBatch; ++u) {
            const int qq = q + u * PP;
            int r, c;
            pm.split(qq, r, c);
            const int pix = qq < NP ? pm.pixel(r, c) : -1;
            v[u][0] = v[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (pix >= 0) {
              const float4* at = reinterpret_cast<const float4*>(src + (long long)pix * a.cin);
              v[u][0] = __ldg(at);
              v[u][1] = __ldg(at + 1);
            }
          }
#pragma unroll
          for (int u = 0; u < kCvBatch; ++u)
            if (q + u * PP < NP)
              *reinterpret_cast<uint4*>(dst + (q + u * PP) * 16) =
                  make_uint4(pack_bf16(v[u][0].x, v[u][0].y), pack_bf16(v[u][0].z, v[u][0].w),
                             pack_bf16(v[u][1].x, v[u][1].y), pack_bf16(v[u][1].z, v[u][1].w));
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // stores visible to the tensor cores
        mbar_arrive(b_full + 8 * st);
      }
    }
    // leave no copy in flight: the last weight tiles issued (landed already unless a wait gave up)
    if (tp == 0)
      for (int k = 0; k < S && k < it; ++k)
        if (!mbar_wait(b_w + 8 * ((it - 1 - k) % S), (uint32_t)(((it - 1 - k) / S) & 1))) break;
  } else if (warp == kCvMma) {
    // ---- products: issued by one lane ----
    constexpr uint32_t idesc = umma_idesc(128, N);
    const uint32_t leader = lane == 0;
    const uint32_t ahi = desc_hi(128), bhi = desc_hi_sw<2 * KC>();
    const uint32_t r1 = (uint32_t)p.pitch, r2 = 2 * r1;
    int it = 0, na = 0;
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x, ++na) {
      const int acc = na & 1;
      if (na >= 2 && !mbar_wait(b_free + 8 * acc, (uint32_t)((na / 2 - 1) & 1))) {
        ok = false;
        break;
      }
      const int rows = min(p.R, rows_all - item / (ntile * p.strips) * p.R);
      const int T = ((rows - 1) * p.pitch + p.Wt + 127) / 128;
      const uint32_t d0 = tmem + (uint32_t)(acc * p.T * N);
      for (int s = 0; s < nst; ++s, ++it) {
        const int st = it % S;
        if (!mbar_wait(b_w + 8 * st, (uint32_t)((it / S) & 1)) || !mbar_wait(b_full + 8 * st, (uint32_t)((it / S) & 1))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t sw = smem_addr(stage0 + st * p.stage_bytes), sx = sw + kW;
        const uint32_t blo = desc_lo(sw, 16), alo = desc_lo(sx, (uint32_t)p.Pn * 16);
        for (int t = 0; t < T; ++t) {
#pragma unroll
          for (int sub = 0; sub < KC / 16; ++sub) {
            const uint32_t at = alo + (uint32_t)(2 * sub * p.Pn + t * 128);
#pragma unroll
            for (int tap = 0; tap < 9; ++tap)
              umma_f16(d0 + t * N, at + (tap < 3 ? 0u : (tap < 6 ? r1 : r2)) + tap % 3, ahi,
                       blo + (uint32_t)(tap * N * KC * 2 / 16 + 2 * sub), bhi, idesc,
                       (s > 0 || sub > 0 || tap > 0) ? 1u : 0u, leader);
          }
        }
        umma_commit(b_empty + 8 * st, leader);
      }
      if (ok) umma_commit(b_acc + 8 * acc, leader);
    }
    // leave no product in flight: the last commits of the stages
    for (int k = 0; k < S && k < it; ++k) {
      const int last = it - 1 - k;
      if (!mbar_wait(b_empty + 8 * (last % S), (uint32_t)((last / S) & 1))) break;
    }
  } else {
    // ---- epilogue ----
    PosMap pm{p.mp, p.mh, p.pitch, a.h, a.w};
    const int quarter = warp & 3;
    float* buf = tbuf + warp * 1024;                // 32 pixels x 32 channels, 16-byte chunks swizzled by pixel
    const int j = lane & 7;                         // lane j + 8 k stores channels 4 j .. of pixels k, k + 4, ...
    int na = 0;
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x, ++na) {
      const int acc = na & 1;
      const int ct = item % ntile, rest = item / ntile;
      const int row0 = rest / p.strips * p.R;
      const int rows = min(p.R, rows_all - row0);
      const int T = ((rows - 1) * p.pitch + p.Wt + 127) / 128;
      pm.block(row0, rest % p.strips * p.Wt);
      if (!mbar_wait(b_acc + 8 * acc, (uint32_t)((na / 2) & 1))) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
      // (tile, 32 channels) units alternate between the two warps of a lane quarter
      for (int unit = warp >> 2; unit < T * (N / 32); unit += 2) {
        const int t = unit / (N / 32), c0 = unit % (N / 32) * 32;
        // output pixel of this lane's TMEM row, -1: a halo column or row
        const int m = t * 128 + quarter * 32 + lane;
        int r, c;
        pm.split(m, r, c);
        const int pix = (r < rows && c < p.Wt) ? pm.pixel(r, c) : -1;
        const int ch = ct * N + c0 + 4 * j;
        float4 bv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (a.bias) bv = make_float4(a.bias[ch], a.bias[ch + 1], a.bias[ch + 2], a.bias[ch + 3]);
        {
          uint32_t v[32];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
              "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
              : "r"(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((acc * p.T + t) * N + c0)));
          asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
          for (int i = 0; i < 8; ++i)
            *reinterpret_cast<uint4*>(buf + lane * 32 + ((i ^ (lane & 7)) * 4)) =
                make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int px = 4 * i + (lane >> 3);
            const int at = __shfl_sync(0xffffffffu, pix, px);   // whole 128-byte lines
            float4 o = *reinterpret_cast<const float4*>(buf + px * 32 + ((j ^ (px & 7)) * 4));
            o = make_float4(o.x + bv.x, o.y + bv.y, o.z + bv.z, o.w + bv.w);
            if (a.relu) o = make_float4(fmaxf(o.x, 0.f), fmaxf(o.y, 0.f), fmaxf(o.z, 0.f), fmaxf(o.w, 0.f));
            if (at >= 0) *reinterpret_cast<float4*>(a.y + (long long)at * a.cout + ch) = o;
          }
          __syncwarp();
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      mbar_arrive(b_free + 8 * acc);
    }
  }
  if (!ok) atomicExch(&g_nn_fault, 1u);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == kCvMma) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem));
}

// Tensor map of the weights: boxes of KC input channels x N output channels x nine taps.
bool weight_map(CUtensorMap* map, const void* wt, int cin, int cout, int N, int KC) {
  static std::atomic<void*> entry{nullptr};
  void* fn = entry.load(std::memory_order_acquire);
  if (!fn) {
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &qr) != cudaSuccess ||
        qr != cudaDriverEntryPointSuccess || !fn)
      return false;
    entry.store(fn, std::memory_order_release);
  }
  const cuuint64_t dims[3] = {(cuuint64_t)cin, (cuuint64_t)cout, 9};
  const cuuint64_t strides[2] = {(cuuint64_t)cin * 2, (cuuint64_t)cin * cout * 2};
  const cuuint32_t box[3] = {(cuuint32_t)KC, (cuuint32_t)N, 9};
  const cuuint32_t estr[3] = {1, 1, 1};
  return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn)(
             map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(wt), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, KC == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ---------------------------------------------------------------------------
// weight gradient: dw[ky, kx][co][ci] = sum_p dy[p][co] x[p + shift(ky, kx)][ci]
//
// A contraction over the pixels on the tensor cores.  As in the forward kernel, a column strip of Wt columns of the
// tall image (the batch's images below one another, a zero row between them) is a flat sequence of positions of pitch
// Wt + 2, and a tap is an offset in it.  With one of the two tensors as U (M side) and the other as V (N side),
//   D[a, u; b, v] = sum_q U[q + a - 1][u] V[q + (b - 1) pitch][v],   a, b = 0 .. 2,
// holds all nine taps: U = x: kx = a, ky = 2 - b; U = dy: kx = 2 - a, ky = b.  dy is zero on the halo columns and
// between the images, so no product counts twice.  Both operands are staged as BF16 in the canonical MN-major layout
// without swizzle: one plane per 8 channels, 16 bytes per position, so a window of 16 positions (K of one product)
// may start anywhere.
//   V: a ring of positions, staged once (halo rows included): tap row b is the window (b - 1) pitch further.  The 16
//      positions at the start of the ring are stored behind its end too, so that no window wraps.
//   U: a slot of KP positions per step.  128 channels fill M, one product per a (the window a positions further, the
//      slot holds one position more on each side).  With at most 64 (32) channels, two (three) of the a share one
//      product: the slot holds three copies of the channels, shifted by a - 1, and M = 128 covers two (three) of them.
// The accumulators (one column block of V channels per product and b) stay in TMEM for a segment of positions.
//
// A CTA (one per SM) owns a tile of U x V channels and a chunk z of the positions, cut into segments no longer than
// the float32 chains of the sums should get (and at strip ends); the first segment's sums are written to part[z], the
// others added.  Producer warps load and round, and sum dy for the bias gradient (unrounded, in a fixed order), in
// three groups that stage every third step each; one lane issues the products; then four warps move the sums out.
// Where x is not finite next to a halo column or a zero row, the products with dy = 0 there make NaN of taps that do not
// reach that value otherwise.
//
// What bounds it: the producers' instructions and load latency on the wide levels (HBM: 40 us for 32 -> 32 on
// 16 x 256^2), the products elsewhere.  Measured (GB300, 16 images, with the sums and the bias gradient): 32 -> 32 on
// 256^2 258 -> 116 us, 128 -> 64 on 128^2 393 -> 100 us, 256 -> 128 on 64^2 331 -> 111 us, 256 -> 256 on 32^2 181 -> 80
// us; the kernels before staged x or dy three times per kernel row between CTA barriers, and dy once more for the bias.
// ---------------------------------------------------------------------------
// instruction descriptor of kind::f16 with both operands MN-major (transpose bits 15 and 16)
__host__ __device__ constexpr uint32_t umma_idesc_mn(int m, int n) { return umma_idesc(m, n) | (1u << 15) | (1u << 16); }

// barrier `id` of `count` threads with the conjunction of their predicates
template <int id, int count>
__device__ __forceinline__ bool meet(bool ok) {
  int all;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n bar.red.and.pred q, %2, %3, p;\n selp.s32 %0, 1, 0, q;\n}\n"
      : "=r"(all)
      : "r"((int)ok), "n"(id), "n"(count)
      : "memory");
  return all != 0;
}

struct WgradArgs {
  const float *u, *v;
  float *part, *bias_part;     // bias_part: [chunks][cout] or NULL
  int n, h, w, cu, cv, cin, cout;
  int wide;                    // both tensors on 32 bytes: 32-byte loads
  WgradPlan p;
};

// MB: products per b (1: three copies of U in one, 2: two and one, 3: no copies)
template <int MB>
__global__ void __launch_bounds__(kWgThreads, 1) conv3x3_wgrad(const WgradArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const WgradPlan& p = a.p;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int S = p.slots;
  // barriers: step staged[S], step free[S], accumulator ready
  const uint32_t b_full = smem_addr(smem), b_empty = b_full + 8 * kWgMaxSlots, b_acc = b_empty + 8 * kWgMaxSlots;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + 16 * kWgMaxSlots + 8);
  unsigned char* const su = smem + kWgHead;                  // U slots, then the V ring
  unsigned char* const sv = su + (size_t)S * p.u_bytes;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tslot)),
                 "r"(p.tmem));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int k = 0; k < S; ++k) {
      mbar_init(b_full + 8 * k, kWgGroup);
      mbar_init(b_empty + 8 * k, 1);
    }
    mbar_init(b_acc, 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(tslot);

  const int ntile = p.utiles * p.vtiles;
  const int tile = blockIdx.x % ntile;
  const long long z = blockIdx.x / ntile;
  const int u0 = tile % p.utiles * p.mt, v0 = tile / p.utiles * p.vt;
  const int nu = min(p.mt, a.cu - u0), nv = min(p.vt, a.cv - v0);   // channels present (multiples of 16)
  const long long total = p.steps * p.strips;
  const long long t0 = total * z / p.chunks, t1 = total * (z + 1) / p.chunks;   // steps of this chunk
  // end of the segment that starts at step t
  auto seg_end = [&](long long t) {
    return min(min(t1, t + p.seg_steps), (t / p.steps + 1) * p.steps);
  };
  bool ok = true;

  if (warp >= kWgEpi) {
    // ---- producers ----
    const int tp = tid - 32 * kWgEpi, tg = tp % kWgGroup, group = tp / kWgGroup;
    WgradSegment seg(p, a.h, a.w);
    auto pow2 = [](int g) { return g <= 1 ? 1 : (g <= 2 ? 2 : (g <= 4 ? 4 : 8)); };
    // thread -> (position, 16-channel group), groups fastest; a thread keeps its group for the whole chunk
    const int gu = pow2(nu / 16), gv = pow2(nv / 16);
    const int ku = tg % gu, qu = tg / gu, kv = tg % gv, qv = tg / gv;
    const int pu = kWgGroup / gu, pv = kWgGroup / gv;        // positions per pass of a group
    const bool u_on = ku < nu / 16, v_on = kv < nv / 16;
    const bool bias = a.bias_part != nullptr && (p.u_dy ? v0 == 0 : u0 == 0);
    float bs[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) bs[k] = 0.f;
    const float *usrc = nullptr, *vsrc = nullptr;            // this thread's channels of the segment map's origin
    // sixteen channels of the segment's position q, zero outside the images; dy only on the strip's own columns
    auto fetch = [&](float (&r)[16], const float* src, int c, bool dy, int q, bool on) {
#pragma unroll
      for (int k = 0; k < 16; ++k) r[k] = 0.f;
      if (on && q >= seg.lo && q < seg.hi) {
        int row, col;
        seg.map.split(q + seg.off, row, col);
        const unsigned pix = seg.map.offset(row, col);
        if (pix != ~0u && (!dy || (unsigned)(col - 1) < (unsigned)p.Wt)) {
          const float* at = src + (unsigned long long)pix * (unsigned)c;
          if (a.wide) {
            ldg8(at, r);
            ldg8(at + 8, r + 8);
          } else {
#pragma unroll
            for (int k = 0; k < 16; k += 4) {
              const float4 t = __ldg(reinterpret_cast<const float4*>(at + k));
              r[k] = t.x, r[k + 1] = t.y, r[k + 2] = t.z, r[k + 3] = t.w;
            }
          }
        }
      }
    };
    auto round8 = [](const float* r) {
      return make_uint4(pack_bf16(r[0], r[1]), pack_bf16(r[2], r[3]), pack_bf16(r[4], r[5]), pack_bf16(r[6], r[7]));
    };
    auto tally = [&](const float (&r)[16]) {
#pragma unroll
      for (int k = 0; k < 16; ++k) bs[k] += r[k];
    };
    int qb = 0;                                              // end of the segment
    auto put_v = [&](const float (&r)[16], int q, int at) {
      if (at >= p.rv) at -= p.rv;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const uint4 val = round8(r + 8 * e);
        unsigned char* dst = sv + ((2 * kv + e) * p.vlen + at) * 16;
        *reinterpret_cast<uint4*>(dst) = val;
        if (at < 16) *reinterpret_cast<uint4*>(dst + p.rv * 16) = val;
      }
      if (bias && !p.u_dy && q >= 0 && q < qb) tally(r);
    };
    auto put_u = [&](const float (&r)[16], unsigned char* slot, int at) {   // at: position - (first - 1)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const uint4 val = round8(r + 8 * e);
        unsigned char* dst = slot + ((2 * ku + e) * p.ulen + at) * 16;
        if (MB == 3) {
          *reinterpret_cast<uint4*>(dst) = val;
        } else {
          // copy c holds position first + i + c - 1 at i
#pragma unroll
          for (int c = 0; c < 3; ++c)
            if ((unsigned)(at - c) < (unsigned)p.KP)
              *reinterpret_cast<uint4*>(dst + (c * ((MB == 1 ? 4 : 8) * p.ulen) - c) * 16) = val;
        }
      }
      if (bias && p.u_dy && at >= 1 && at <= p.KP) tally(r);
    };
    int it = 0;                                              // steps over all segments
    for (long long t = t0; t < t1;) {
      const long long te = seg_end(t);
      qb = (int)(te - t) * p.KP;
      seg.start(p, t % p.steps * p.KP, (int)(t / p.steps));
      usrc = a.u + u0 + 16 * ku + seg.map.origin() * a.cu;
      vsrc = a.v + v0 + 16 * kv + seg.map.origin() * a.cv;
      // the ring restarts at position -pitch: every step of the previous segment is staged (the groups meet first: a
      // phase may only be waited for once the one before it is known to be complete) and its products are done; then
      // the ring's first 2 pitch positions, by all producers
      if (!(ok = meet<1, kWgProd>(ok))) break;
      for (int k = 1; k <= S && k <= it && ok; ++k)
        ok = mbar_wait(b_empty + 8 * ((it - k) % S), (uint32_t)(((it - k) / S) & 1));
      if (ok)
        for (int q = group * pv + qv; q < 2 * p.pitch; q += kWgGroups * pv * kWgBatch) {
          float r[kWgBatch][16];
#pragma unroll
          for (int k = 0; k < kWgBatch; ++k) {
            const int at = q + k * kWgGroups * pv;
            fetch(r[k], vsrc, a.cv, !p.u_dy, at - p.pitch, v_on && at < 2 * p.pitch);
          }
#pragma unroll
          for (int k = 0; k < kWgBatch; ++k) {
            const int at = q + k * kWgGroups * pv;
            if (v_on && at < 2 * p.pitch) put_v(r[k], at - p.pitch, at);
          }
        }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      if (!(ok = meet<1, kWgProd>(ok))) break;
      const int nstep = (int)(te - t);
      const int base = it;
      for (int sn = (group + kWgGroups - base % kWgGroups) % kWgGroups; sn < nstep; sn += kWgGroups) {
        const int step = base + sn, st = step % S, qs = sn * p.KP;
        if (step >= S && !mbar_wait(b_empty + 8 * st, (uint32_t)((step / S - 1) & 1))) {
          ok = false;
          break;
        }
        const int ring = (2 * p.pitch + qs) % p.rv;          // ring index of position qs + pitch
        unsigned char* slot = su + (size_t)st * p.u_bytes;
        for (int iv = qv, iu = qu; iv < p.KP || iu < p.KP + 2; iv += kWgBatch * pv, iu += kWgBatch * pu) {
          float rv[kWgBatch][16], ru[kWgBatch][16];
#pragma unroll
          for (int k = 0; k < kWgBatch; ++k)
            fetch(rv[k], vsrc, a.cv, !p.u_dy, qs + p.pitch + iv + k * pv, v_on && iv + k * pv < p.KP);
#pragma unroll
          for (int k = 0; k < kWgBatch; ++k)
            fetch(ru[k], usrc, a.cu, p.u_dy, qs - 1 + iu + k * pu, u_on && iu + k * pu < p.KP + 2);
#pragma unroll
          for (int k = 0; k < kWgBatch; ++k)
            if (v_on && iv + k * pv < p.KP) put_v(rv[k], qs + p.pitch + iv + k * pv, ring + iv + k * pv);
#pragma unroll
          for (int k = 0; k < kWgBatch; ++k)
            if (u_on && iu + k * pu < p.KP + 2) put_u(ru[k], slot, iu + k * pu);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(b_full + 8 * st);
      }
      it = base + nstep;
      t = te;
    }
    ok = meet<1, kWgProd>(ok);
    // bias partials: the threads of a channel group in their order.  The stages are free once the products are done.
    for (int k = 1; k <= S && k <= it && ok; ++k)
      ok = mbar_wait(b_empty + 8 * ((it - k) % S), (uint32_t)(((it - k) / S) & 1));
    if (bias) {
      const int g = p.u_dy ? gu : gv, nc = p.u_dy ? nu : nv, c0 = p.u_dy ? u0 : v0;
      float* red = reinterpret_cast<float*>(sv);             // [16][kWgProd]: fits the ring (at least 24.6 KB)
      if (ok) {
#pragma unroll
        for (int k = 0; k < 16; ++k) red[k * kWgProd + tp] = bs[k];
      }
      (void)meet<1, kWgProd>(ok);
      if (tp < nc) {
        float s = 0.f;
        for (int k = tp / 16; k < kWgProd; k += g) s += red[(tp & 15) * kWgProd + k];
        a.bias_part[z * a.cout + c0 + tp] = s;
      }
    }
  } else {
    // ---- products: one thread; then the epilogue of the segment: four warps ----
    const uint32_t idesc = umma_idesc_mn(128, nv);
    const uint32_t usbo = (uint32_t)p.ulen * 16, vsbo = (uint32_t)p.vlen * 16;
    const uint32_t ahi = desc_hi(usbo), bhi = desc_hi(vsbo);
    const uint32_t vlo = desc_lo(smem_addr(sv), 128), ulo = desc_lo(smem_addr(su), 128);
    const uint32_t leader = lane == 0;
    const int quarter = warp;
    const int fold = MB == 3 ? 1 : (MB == 2 ? 2 : 4);    // copies of U's channels in one product's 128 rows
    const int row = quarter * 32 + lane;
    const int per = 128 / fold;                              // rows per copy
    const int c = row % per;                                 // U channel of this lane's TMEM row
    int it = 0, ns = 0;
    for (long long t = t0; t < t1 && ok; ++ns) {
      const long long te = seg_end(t);
      if (warp == 0) {
        // ring indices of the windows of tap rows 0 .. 2 at the segment's first position
        int r0 = 0, r1 = p.pitch, r2 = 2 * p.pitch;
        for (long long s = t; s < te; ++s, ++it) {
          const int st = it % S;
          if (!mbar_wait(b_full + 8 * st, (uint32_t)((it / S) & 1))) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t slot = ulo + (uint32_t)(st * (p.u_bytes / 16));
          for (int k = 0; k < p.KP; k += 16) {
            const uint32_t acc = (s > t || k > 0) ? 1u : 0u;
            const uint32_t w0 = vlo + (uint32_t)r0, w1 = vlo + (uint32_t)r1, w2 = vlo + (uint32_t)r2;
            for (int m = 0; m < MB; ++m) {
              // mb 3: the window m positions further; else block m of the copies' planes
              const uint32_t ua = slot + (uint32_t)k + (uint32_t)(MB == 3 ? m : m * 16 * p.ulen);
              const uint32_t d = tmem + (uint32_t)(m * 3 * p.vt);
              umma_f16(d, ua, ahi, w0, bhi, idesc, acc, leader);
              umma_f16(d + p.vt, ua, ahi, w1, bhi, idesc, acc, leader);
              umma_f16(d + 2 * p.vt, ua, ahi, w2, bhi, idesc, acc, leader);
            }
            r0 = r0 + 16 >= p.rv ? r0 + 16 - p.rv : r0 + 16;
            r1 = r1 + 16 >= p.rv ? r1 + 16 - p.rv : r1 + 16;
            r2 = r2 + 16 >= p.rv ? r2 + 16 - p.rv : r2 + 16;
          }
          umma_commit(b_empty + 8 * st, leader);
        }
        if (ok) umma_commit(b_acc, leader);
        __syncwarp();
      }
      ok = mbar_wait(b_acc, (uint32_t)(ns & 1)) && ok;
      if (!(ok = meet<2, 32 * kWgEpi>(ok))) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
      const int nblk = nv / 16;
      for (int unit = 0; unit < MB * 3 * nblk; ++unit) {
        const int blk = unit % nblk, b = unit / nblk % 3, m = unit / (3 * nblk);
        const int cp = m * fold + row / per;                 // a of this row
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
            "%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
              "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((m * 3 + b) * p.vt + blk * 16)));
        asm volatile("tcgen05.wait::ld.sync.aligned;");
        if (cp < 3 && c < nu) {
          const int tap = p.u_dy ? 3 * b + 2 - cp : 3 * (2 - b) + cp;
          float* base = a.part + (z * 9 + tap) * a.cout * a.cin;
          if (p.u_dy) {                                      // row = co, columns = ci
            float4* dst = reinterpret_cast<float4*>(base + (long long)(u0 + c) * a.cin + v0 + blk * 16);
            float4 e[4];                                     // the earlier segments' sums, all loads before the stores
#pragma unroll
            for (int j = 0; j < 4; ++j) e[j] = ns > 0 ? dst[j] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              dst[j] = make_float4(e[j].x + __uint_as_float(r[4 * j]), e[j].y + __uint_as_float(r[4 * j + 1]),
                                   e[j].z + __uint_as_float(r[4 * j + 2]), e[j].w + __uint_as_float(r[4 * j + 3]));
          } else {                                           // row = ci, columns = co
            float* dst = base + (long long)(v0 + blk * 16) * a.cin + u0 + c;
            float e[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) e[j] = ns > 0 ? dst[(long long)j * a.cin] : 0.f;
#pragma unroll
            for (int j = 0; j < 16; ++j) dst[(long long)j * a.cin] = e[j] + __uint_as_float(r[j]);
          }
        }
      }
      // the sums are read before the next segment overwrites them
      asm volatile("tcgen05.fence::before_thread_sync;");
      (void)meet<2, 32 * kWgEpi>(true);
      asm volatile("tcgen05.fence::after_thread_sync;");
      t = te;
    }
    if (warp == 0)
      for (int k = 1; k <= S && k <= it; ++k)                // leave no product in flight
        if (!mbar_wait(b_empty + 8 * ((it - k) % S), (uint32_t)(((it - k) / S) & 1))) break;
  }
  if (!ok) atomicExch(&g_nn_fault, 1u);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem));
}

// out[i] = sum_z part[z][i] for the n weight gradients and, in the blocks behind theirs, for the n2 bias gradients: L
// lanes per output take the chunks z = lane, lane + L, ... in order, then the lane sums are added in a fixed tree
// (deterministic).  Block = 32 outputs x L lanes.  A few MB out of L2, bound by latency: about ten loads per lane (152
// chunks of 32 x 32 channels: 7.5 + 6.6 us as two launches of eight lanes, 5 us as this one of sixteen).
constexpr int kSumLanes = 16;   // most lanes
__global__ void __launch_bounds__(32 * kSumLanes) sum_parts(const float* __restrict__ part, float* __restrict__ out,
                                                            long long n, const float* __restrict__ part2,
                                                            float* __restrict__ out2, int n2, int chunks) {
  __shared__ float red[kSumLanes][32];
  const long long nb = (n + 31) / 32;
  long long blk = blockIdx.x;
  if (blk >= nb) part = part2, out = out2, n = n2, blk -= nb;
  const int o = threadIdx.x & 31, lane = threadIdx.x >> 5, L = blockDim.x >> 5;
  const long long i = blk * 32 + o;
  float s = 0.f;
  if (i < n) {
#pragma unroll 10
    for (int z = lane; z < chunks; z += L) s += part[(long long)z * n + i];
  }
  red[lane][o] = s;
  __syncthreads();
  for (int k = L / 2; k > 0; k >>= 1) {
    if (lane < k) red[lane][o] += red[lane + k][o];
    __syncthreads();
  }
  if (lane == 0 && i < n) out[i] = red[0][o];
}

// wt'[tap][ci][co] = wt[8 - tap][co][ci]: the kernel of the data gradient
__global__ void flip_transpose(const __nv_bfloat16* __restrict__ wt, __nv_bfloat16* __restrict__ wf, int cin,
                               int cout) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long total = 9LL * cin * cout;
  if (i >= total) return;
  const int co = (int)(i % cout), ci = (int)((i / cout) % cin), tap = (int)(i / ((long long)cout * cin));
  wf[i] = wt[((long long)(8 - tap) * cout + co) * cin + ci];
}

// dx = dy where y > 0, else 0 (dx may be dy)
__global__ void relu_bwd(const float* dy, const float* __restrict__ y, float* dx, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dx[i] = y[i] > 0.f ? dy[i] : 0.f;
}

// 2x2 average pooling and its adjoint
__global__ void pool2_fwd(const float* __restrict__ x, float* __restrict__ y, int n, int h, int w, int c) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int h2 = h / 2, w2 = w / 2;
  if (i >= (long long)n * h2 * w2 * c) return;
  const int ch = (int)(i % c);
  const long long q = i / c;
  const int xx = (int)(q % w2), yy = (int)((q / w2) % h2), nn = (int)(q / ((long long)w2 * h2));
  const long long b = (((long long)nn * h + 2 * yy) * w + 2 * xx) * c + ch;
  y[i] = 0.25f * ((x[b] + x[b + c]) + (x[b + (long long)w * c] + x[b + (long long)w * c + c]));
}
__global__ void pool2_bwd(const float* __restrict__ dy, float* __restrict__ dx, int n, int h, int w, int c) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)n * h * w * c) return;
  const int ch = (int)(i % c);
  const long long q = i / c;
  const int xx = (int)(q % w), yy = (int)((q / w) % h), nn = (int)(q / ((long long)w * h));
  dx[i] = 0.25f * dy[(((long long)nn * (h / 2) + yy / 2) * (w / 2) + xx / 2) * c + ch];
}

// nearest 2x upsampling and its adjoint (h, w: the coarse size)
__global__ void up2_fwd(const float* __restrict__ x, float* __restrict__ y, int n, int h, int w, int c) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)n * 4 * h * w * c) return;
  const int ch = (int)(i % c);
  const long long q = i / c;
  const int xx = (int)(q % (2 * w)), yy = (int)((q / (2 * w)) % (2 * h)), nn = (int)(q / (4LL * w * h));
  y[i] = x[(((long long)nn * h + yy / 2) * w + xx / 2) * c + ch];
}
__global__ void up2_bwd(const float* __restrict__ dy, float* __restrict__ dx, int n, int h, int w, int c) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)n * h * w * c) return;
  const int ch = (int)(i % c);
  const long long q = i / c;
  const int xx = (int)(q % w), yy = (int)((q / w) % h), nn = (int)(q / ((long long)w * h));
  const long long b = (((long long)nn * 2 * h + 2 * yy) * 2 * w + 2 * xx) * c + ch;
  const long long row = 2LL * w * c;
  dx[i] = (dy[b] + dy[b + c]) + (dy[b + row] + dy[b + row + c]);
}

// The same four maps on float4 groups of channels with 32-bit index arithmetic (c4 = c / 4 groups; the callers
// use them when c % 4 == 0 and the element count fits 32 bits)
__global__ void pool2_fwd4(const float4* __restrict__ x, float4* __restrict__ y, int n, int h, int w, int c4) {
  const unsigned h2 = h / 2, w2 = w / 2;
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (unsigned)n * h2 * w2 * c4) return;
  const unsigned ch = i % c4, q = i / c4;
  const unsigned xx = q % w2, r = q / w2, yy = r % h2, nn = r / h2;
  const unsigned b = ((nn * h + 2 * yy) * w + 2 * xx) * c4 + ch, row = (unsigned)w * c4;
  const float4 a = x[b], bb = x[b + c4], cc = x[b + row], d = x[b + row + c4];
  y[i] = make_float4(0.25f * ((a.x + bb.x) + (cc.x + d.x)), 0.25f * ((a.y + bb.y) + (cc.y + d.y)),
                     0.25f * ((a.z + bb.z) + (cc.z + d.z)), 0.25f * ((a.w + bb.w) + (cc.w + d.w)));
}
__global__ void pool2_bwd4(const float4* __restrict__ dy, float4* __restrict__ dx, int n, int h, int w, int c4) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (unsigned)n * h * w * c4) return;
  const unsigned ch = i % c4, q = i / c4;
  const unsigned xx = q % w, r = q / w, yy = r % h, nn = r / h;
  const float4 v = dy[((nn * (h / 2) + yy / 2) * (w / 2) + xx / 2) * c4 + ch];
  dx[i] = make_float4(0.25f * v.x, 0.25f * v.y, 0.25f * v.z, 0.25f * v.w);
}
__global__ void up2_fwd4(const float4* __restrict__ x, float4* __restrict__ y, int n, int h, int w, int c4) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (unsigned)n * 4 * h * w * c4) return;
  const unsigned ch = i % c4, q = i / c4;
  const unsigned xx = q % (2 * w), r = q / (2 * w), yy = r % (2 * h), nn = r / (2 * h);
  y[i] = x[((nn * h + yy / 2) * w + xx / 2) * c4 + ch];
}
__global__ void up2_bwd4(const float4* __restrict__ dy, float4* __restrict__ dx, int n, int h, int w, int c4) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (unsigned)n * h * w * c4) return;
  const unsigned ch = i % c4, q = i / c4;
  const unsigned xx = q % w, r = q / w, yy = r % h, nn = r / h;
  const unsigned b = ((nn * 2 * h + 2 * yy) * 2 * w + 2 * xx) * c4 + ch, row = 2u * w * c4;
  const float4 a = dy[b], bb = dy[b + c4], cc = dy[b + row], d = dy[b + row + c4];
  dx[i] = make_float4((a.x + bb.x) + (cc.x + d.x), (a.y + bb.y) + (cc.y + d.y), (a.z + bb.z) + (cc.z + d.z),
                      (a.w + bb.w) + (cc.w + d.w));
}

// float4 forms of relu_bwd and add (n % 4 == 0, 16-byte aligned pointers)
__global__ void relu_bwd4(const float4* dy, const float4* __restrict__ y, float4* dx, long long n4) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  const float4 g = dy[i], v = y[i];
  dx[i] = make_float4(v.x > 0.f ? g.x : 0.f, v.y > 0.f ? g.y : 0.f, v.z > 0.f ? g.z : 0.f, v.w > 0.f ? g.w : 0.f);
}
__global__ void add4(float4* z, const float4* x, const float4* y, float a, long long n4) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  const float4 u = x[i], v = y[i];
  z[i] = make_float4(u.x + a * v.x, u.y + a * v.y, u.z + a * v.z, u.w + a * v.w);
}

// z = x + a y (z may be x or y)
__global__ void add(float* z, const float* x, const float* y, float a, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) z[i] = x[i] + a * y[i];
}

// input tensor [p][16]: phi0, phi1, cos theta of the image, zeros.  Bound by its writes (64 bytes a node), so they must
// be whole lines: a warp's 32 nodes are one run of 2 KB, which it writes as consecutive float4 with the values taken from
// the lanes that loaded them (16 images of 256^2: 12 us, where a thread that wrote its own node took 70).  V4 needs x on
// 16 bytes; without it a thread writes its own node's 16 words.
template <bool V4>
__global__ void pack_input(const float* __restrict__ phi0, const float* __restrict__ phi1,
                           const float* __restrict__ costh, float* __restrict__ x, long long P, long long hw) {
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  float a = 0.f, b = 0.f, t = 0.f;
  if (p < P) {
    a = phi0[p];
    b = phi1[p];
    t = costh[P < (1LL << 31) ? (int)((unsigned)p / (unsigned)hw) : p / hw];
  }
  if constexpr (V4) {
    const int lane = threadIdx.x & 31;
    const long long w0 = p - lane;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = j * 32 + lane, from = i >> 2;
      const float va = __shfl_sync(~0u, a, from), vb = __shfl_sync(~0u, b, from), vt = __shfl_sync(~0u, t, from);
      if (w0 + from < P)
        reinterpret_cast<float4*>(x)[w0 * 4 + i] = i & 3 ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(va, vb, vt, 0.f);
    }
  } else if (p < P) {
    float* o = x + p * 16;
    o[0] = a;
    o[1] = b;
    o[2] = t;
#pragma unroll
    for (int c = 3; c < 16; ++c) o[c] = 0.f;
  }
}

// prediction = base + out[p][0]; loss partials (FP64) and d loss / d out = 2 (pred - target) / P in channel 0.  Bound by
// the writes of dout (cpad words a node): V4 (cpad % 4 == 0, dout on 16 bytes) writes a warp's nodes as one run of
// consecutive float4, as pack_input does (16 images of 256^2, 32 words: 54 us with the sum of the partials, before 180).
template <bool V4>
__global__ void mse_residual(const float* __restrict__ out, int cpad, const float* __restrict__ base,
                             const float* __restrict__ target, float* __restrict__ dout, double* __restrict__ part,
                             long long P) {
  __shared__ double s[kThreads];
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double e2 = 0.0;
  float g = 0.f;
  if (p < P) {
    const float d = (base[p] + out[p * cpad]) - target[p];
    e2 = (double)d * d;
    g = 2.f * d / (float)P;
  }
  if constexpr (V4) {
    const int lane = threadIdx.x & 31, q4 = cpad / 4;
    const long long w0 = p - lane;
    for (int j = 0; j < q4; ++j) {
      const int i = j * 32 + lane, from = i / q4;
      const float v = __shfl_sync(~0u, g, from);
      if (w0 + from < P)
        reinterpret_cast<float4*>(dout)[w0 * q4 + i] = make_float4(i == from * q4 ? v : 0.f, 0.f, 0.f, 0.f);
    }
  } else if (p < P) {
    dout[p * cpad] = g;
    for (int c = 1; c < cpad; ++c) dout[p * cpad + c] = 0.f;
  }
  s[threadIdx.x] = e2;
  __syncthreads();
  for (int k = kThreads / 2; k > 0; k >>= 1) {
    if ((int)threadIdx.x < k) s[threadIdx.x] += s[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}

// out = sum of n partials: one CTA, strided per-thread sums, then a fixed-order tree (deterministic)
__global__ void __launch_bounds__(256) sum_double(const double* __restrict__ part, int n, double* __restrict__ out) {
  __shared__ double s[256];
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) v += part[i];
  s[threadIdx.x] = v;
  __syncthreads();
  for (int k = 128; k > 0; k >>= 1) {
    if ((int)threadIdx.x < k) s[threadIdx.x] += s[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = s[0];
}

// Adam with bias correction; writes the BF16 copy of the updated weights
__global__ void adam_step(float* __restrict__ wm, float* __restrict__ m, float* __restrict__ v,
                          const float* __restrict__ grad, __nv_bfloat16* __restrict__ wb, long long n, float lr,
                          float b1, float b2, float eps, float c1, float c2) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = grad[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float wi = wm[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  wm[i] = wi;
  if (wb) wb[i] = __float2bfloat16_rn(wi);
}

__global__ void to_bf16(const float* __restrict__ a, __nv_bfloat16* __restrict__ b, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = __float2bfloat16_rn(a[i]);
}

// warm-start projection.  hi = max(1 - phi0, 0); the bump b(q) = q (hi - q) / hi (0 where hi = 0) vanishes at
// both bounds, and for |lambda| <= 1 the map q -> q + lambda b(q) is monotone on [0, hi] with fixed points 0 and
// hi, so a correction step never leaves the bounds.
__device__ __forceinline__ float proj_bump(float q, float hi) { return hi > 0.f ? q * (hi - q) / hi : 0.f; }

// One stage of the projection over an image's nodes (grid: parts, images):
//   INIT   field = clamp(phi1 + out[p][0], 0, hi)
//   APPLY  field += lambda b(field), lambda = clamp((sum phi1 - sum field) / sum b, -1, 1) from the sums of stage `in`
//   SUM    per image and part: sums of phi1 (target mass), of the field and of its bump, into `sums`
// A thread meets the same nodes in every stage, so the update of one pass and the sums of the next are one launch; `in`
// and `sums` are then two buffers, since other CTAs may still read `in`.  Short launches: what counts is their number
// and the chain of 64 partials, which three threads add (by every thread it is 192 FP64 additions each, at an FP64 rate
// that is a small part of FP32's).  Three passes on one image of 256^2: 47 us in four launches, 78 before in seven; on 16
// images 93 against 257.
template <bool INIT, bool APPLY, bool SUM>
__global__ void project_stage(const float* __restrict__ out, int cpad, const float* __restrict__ phi0, const float* phi1,
                              const double* in, double* sums, float* field, long long hw) {
  __shared__ double s[3][kThreads];
  const int img = blockIdx.y, parts = gridDim.x;
  float lam = 0.f;
  if constexpr (APPLY) {
    __shared__ double tot[3];
    const double* part = in + (long long)img * parts * 3;
    if (threadIdx.x < 3) {
      double v = 0.0;
#pragma unroll 16
      for (int k = 0; k < parts; ++k) v += part[k * 3 + threadIdx.x];
      tot[threadIdx.x] = v;
    }
    __syncthreads();
    lam = tot[2] > 0.0 ? (float)fmin(1.0, fmax(-1.0, (tot[0] - tot[1]) / tot[2])) : 0.f;
  }
  double a = 0.0, b = 0.0, c = 0.0;
  for (long long k = (long long)blockIdx.x * kThreads + threadIdx.x; k < hw; k += (long long)parts * kThreads) {
    const long long p = img * hw + k;
    const float hi = fmaxf(1.f - phi0[p], 0.f);
    float q;
    if constexpr (INIT) q = fminf(fmaxf(phi1[p] + out[p * cpad], 0.f), hi);
    else q = field[p];
    if constexpr (APPLY) q = q + lam * proj_bump(q, hi);
    if constexpr (INIT || APPLY) field[p] = q;
    if constexpr (SUM) {
      a += phi1[p];
      b += q;
      c += proj_bump(q, hi);
    }
  }
  if constexpr (SUM) {
    s[0][threadIdx.x] = a;
    s[1][threadIdx.x] = b;
    s[2][threadIdx.x] = c;
    __syncthreads();
    for (int k = kThreads / 2; k > 0; k >>= 1) {
      if ((int)threadIdx.x < k)
        for (int j = 0; j < 3; ++j) s[j][threadIdx.x] += s[j][threadIdx.x + k];
      __syncthreads();
    }
    if (threadIdx.x == 0)
      for (int j = 0; j < 3; ++j) sums[((long long)img * parts + blockIdx.x) * 3 + j] = s[j][0];
  }
}

unsigned blocks(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

int status(cudaError_t e) { return e == cudaSuccess ? 0 : -3; }

}  // namespace

extern "C" {

int lbm_nn_conv3x3(const float* x, const void* wt_bf16, const float* bias, float* y, int n, int h, int w, int cin,
                   int cout, int relu, void* stream) {
  if (!x || !wt_bf16 || !y || n < 1 || h < 1 || w < 1 || cin < 16 || cin % 16 || cout < 32 || cout % 32) return -1;
  // the opt-in above 48 KB of shared memory is a per-device attribute: set it once for each device used
  static std::atomic<unsigned long long> attr_set{0};
  static std::atomic<int> sm_count[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -3;
  if (!(attr_set.load(std::memory_order_acquire) & (1ull << dev))) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return -3;
    for (const void* fn : {(const void*)conv3x3_fwd<32, 16>, (const void*)conv3x3_fwd<32, 32>,
                           (const void*)conv3x3_fwd<64, 16>, (const void*)conv3x3_fwd<64, 32>,
                           (const void*)conv3x3_fwd<128, 16>, (const void*)conv3x3_fwd<128, 32>})
      if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kCvSmem) != cudaSuccess) return -3;
    sm_count[dev].store(sms);
    attr_set.fetch_or(1ull << dev, std::memory_order_acq_rel);
  }
  const int sms = sm_count[dev].load();
  // rows and pixels of one launch are 32-bit numbers; a larger batch runs in parts
  const int most = (int)std::max(1LL, std::min<long long>((1LL << 30) / (h + 1), ((1LL << 31) - 1) / ((long long)h * w)));
  cudaStream_t s = (cudaStream_t)stream;
  for (int i0 = 0; i0 < n; i0 += most) {
    const int ni = std::min(most, n - i0);
    const long long pix = (long long)i0 * h * w;
    FwdArgs a{x + pix * cin, bias, y + pix * cout, ni, h, w, cin, cout, relu, fwd_plan(ni, h, w, cin, cout, sms)};
    // tensor map of the weights [tap][cout][cin]: a box holds the nine taps of N output and KC input channels
    CUtensorMap wmap;
    if (!weight_map(&wmap, wt_bf16, cin, cout, a.p.N, a.p.KC)) return -3;
    const unsigned grid = (unsigned)std::min(a.p.items, sms);
    const int kc16 = a.p.KC == 16;
#define LBM_NN_FWD(NN)                                                              \
  do {                                                                              \
    if (kc16) conv3x3_fwd<NN, 16><<<grid, kCvThreads, a.p.smem, s>>>(a, wmap);      \
    else conv3x3_fwd<NN, 32><<<grid, kCvThreads, a.p.smem, s>>>(a, wmap);           \
  } while (0)
    if (a.p.N == 128) LBM_NN_FWD(128);
    else if (a.p.N == 64) LBM_NN_FWD(64);
    else LBM_NN_FWD(32);
#undef LBM_NN_FWD
    if (cudaGetLastError() != cudaSuccess) return -3;
  }
  return 0;
}

int lbm_nn_check(void) {
  unsigned int f = 0;
  if (cudaMemcpyFromSymbol(&f, g_nn_fault, sizeof f) != cudaSuccess) return -3;
  if (f) {
    const unsigned int zero = 0;
    cudaMemcpyToSymbol(g_nn_fault, &zero, sizeof zero);
    return -5;
  }
  return 0;
}

long long lbm_nn_wgrad_workspace(int n, int h, int w, int cin, int cout) {
  if (n < 1 || h < 1 || w < 1 || cin < 1 || cout < 1) return 0;
  const WgradPlan p = wgrad_plan(n, h, w, cin, cout);
  return p.ws_chunks * 9LL * cin * cout + p.bias_chunks * cout;
}

int lbm_nn_conv3x3_wgrad(const float* x, const float* dy, float* dw, float* db, float* work, long long work_len,
                         int n, int h, int w, int cin, int cout, void* stream) {
  if (!x || !dy || !dw || !work || n < 1 || h < 1 || w < 1 || cin < 16 || cin % 16 || cout < 16 || cout % 16)
    return -1;
  if (work_len < lbm_nn_wgrad_workspace(n, h, w, cin, cout)) return -1;
  cudaStream_t s = (cudaStream_t)stream;
  const WgradPlan p = wgrad_plan(n, h, w, cin, cout);
  const long long nw = 9LL * cin * cout;
  static std::atomic<unsigned long long> attr_set{0};   // shared-memory opt-in, per device
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -3;
  if (!(attr_set.load(std::memory_order_acquire) & (1ull << dev))) {
    for (const void* fn : {(const void*)conv3x3_wgrad<1>, (const void*)conv3x3_wgrad<2>, (const void*)conv3x3_wgrad<3>})
      if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kCvSmem) != cudaSuccess) return -3;
    attr_set.fetch_or(1ull << dev, std::memory_order_acq_rel);
  }
  float* bpart = work + p.chunks * nw;
  const WgradArgs a{p.u_dy ? dy : x, p.u_dy ? x : dy, work, db ? bpart : nullptr, n, h, w,
                    p.u_dy ? cout : cin, p.u_dy ? cin : cout, cin, cout,
                    ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(dy)) & 31) == 0, p};
  const unsigned grid = (unsigned)(p.chunks * p.utiles * p.vtiles);
  if (p.mb == 1) conv3x3_wgrad<1><<<grid, kWgThreads, p.smem, s>>>(a);
  else if (p.mb == 2) conv3x3_wgrad<2><<<grid, kWgThreads, p.smem, s>>>(a);
  else conv3x3_wgrad<3><<<grid, kWgThreads, p.smem, s>>>(a);
  const int nb = db ? cout : 0;
  const int lanes = p.chunks > 64 ? kSumLanes : (p.chunks > 32 ? 8 : (p.chunks > 12 ? 4 : 2));
  sum_parts<<<(unsigned)((nw + 31) / 32 + (nb + 31) / 32), 32 * lanes, 0, s>>>(work, dw, nw, bpart, db, nb, (int)p.chunks);
  return status(cudaGetLastError());
}

int lbm_nn_flip_transpose(const void* wt_bf16, void* wf_bf16, int cin, int cout, void* stream) {
  if (!wt_bf16 || !wf_bf16 || cin < 1 || cout < 1) return -1;
  flip_transpose<<<blocks(9LL * cin * cout), 256, 0, (cudaStream_t)stream>>>(
      static_cast<const __nv_bfloat16*>(wt_bf16), static_cast<__nv_bfloat16*>(wf_bf16), cin, cout);
  return status(cudaGetLastError());
}

int lbm_nn_relu_bwd(const float* dy, const float* y, float* dx, long long n, void* stream) {
  if (!dy || !y || !dx || n < 0) return -1;
  if (n % 4 == 0 && ((uintptr_t)dy | (uintptr_t)y | (uintptr_t)dx) % 16 == 0) {
    if (n)
      relu_bwd4<<<blocks(n / 4), 256, 0, (cudaStream_t)stream>>>(reinterpret_cast<const float4*>(dy),
                                                                  reinterpret_cast<const float4*>(y),
                                                                  reinterpret_cast<float4*>(dx), n / 4);
  } else if (n) {
    relu_bwd<<<blocks(n), 256, 0, (cudaStream_t)stream>>>(dy, y, dx, n);
  }
  return status(cudaGetLastError());
}

int lbm_nn_pool2(const float* x, float* y, int n, int h, int w, int c, int backward, void* stream) {
  if (!x || !y || n < 1 || h < 2 || w < 2 || h % 2 || w % 2 || c < 1) return -1;
  cudaStream_t s = (cudaStream_t)stream;
  const long long total = (long long)n * h * w * c;
  if (c % 4 == 0 && total < (1LL << 31) && ((uintptr_t)x | (uintptr_t)y) % 16 == 0) {
    const int c4 = c / 4;
    if (!backward)
      pool2_fwd4<<<blocks(total / 16), 256, 0, s>>>(reinterpret_cast<const float4*>(x), reinterpret_cast<float4*>(y),
                                                     n, h, w, c4);
    else
      pool2_bwd4<<<blocks(total / 4), 256, 0, s>>>(reinterpret_cast<const float4*>(x), reinterpret_cast<float4*>(y),
                                                    n, h, w, c4);
  } else if (!backward) {
    pool2_fwd<<<blocks(total / 4), 256, 0, s>>>(x, y, n, h, w, c);
  } else {
    pool2_bwd<<<blocks(total), 256, 0, s>>>(x, y, n, h, w, c);
  }
  return status(cudaGetLastError());
}

int lbm_nn_up2(const float* x, float* y, int n, int h, int w, int c, int backward, void* stream) {
  if (!x || !y || n < 1 || h < 1 || w < 1 || c < 1) return -1;
  cudaStream_t s = (cudaStream_t)stream;
  const long long fine = 4LL * n * h * w * c;
  if (c % 4 == 0 && fine < (1LL << 31) && ((uintptr_t)x | (uintptr_t)y) % 16 == 0) {
    const int c4 = c / 4;
    if (!backward)
      up2_fwd4<<<blocks(fine / 4), 256, 0, s>>>(reinterpret_cast<const float4*>(x), reinterpret_cast<float4*>(y), n,
                                                 h, w, c4);
    else
      up2_bwd4<<<blocks(fine / 16), 256, 0, s>>>(reinterpret_cast<const float4*>(x), reinterpret_cast<float4*>(y), n,
                                                  h, w, c4);
  } else if (!backward) {
    up2_fwd<<<blocks(fine), 256, 0, s>>>(x, y, n, h, w, c);
  } else {
    up2_bwd<<<blocks(fine / 4), 256, 0, s>>>(x, y, n, h, w, c);
  }
  return status(cudaGetLastError());
}

int lbm_nn_add(float* z, const float* x, const float* y, float a, long long n, void* stream) {
  if (!z || !x || !y || n < 0) return -1;
  if (n % 4 == 0 && ((uintptr_t)z | (uintptr_t)x | (uintptr_t)y) % 16 == 0) {
    if (n)
      add4<<<blocks(n / 4), 256, 0, (cudaStream_t)stream>>>(reinterpret_cast<float4*>(z),
                                                             reinterpret_cast<const float4*>(x),
                                                             reinterpret_cast<const float4*>(y), a, n / 4);
  } else if (n) {
    add<<<blocks(n), 256, 0, (cudaStream_t)stream>>>(z, x, y, a, n);
  }
  return status(cudaGetLastError());
}

int lbm_nn_pack_input(const float* phi0, const float* phi1, const float* costh, float* x, int n, int h, int w,
                      void* stream) {
  if (!phi0 || !phi1 || !costh || !x || n < 1 || h < 1 || w < 1) return -1;
  const long long hw = (long long)h * w;
  const auto pack = reinterpret_cast<uintptr_t>(x) % 16 == 0 ? pack_input<true> : pack_input<false>;
  pack<<<blocks(n * hw), 256, 0, (cudaStream_t)stream>>>(phi0, phi1, costh, x, n * hw, hw);
  return status(cudaGetLastError());
}

int lbm_nn_mse_residual(const float* out, int cpad, const float* base, const float* target, float* dout,
                        double* work, long long work_len, double* loss, long long P, void* stream) {
  if (!out || !base || !target || !dout || !work || !loss || P < 1 || cpad < 1) return -1;
  const int nb = (int)((P + kThreads - 1) / kThreads);
  if (work_len < nb) return -1;
  cudaStream_t s = (cudaStream_t)stream;
  const bool v4 = cpad % 4 == 0 && reinterpret_cast<uintptr_t>(dout) % 16 == 0;
  const auto mse = v4 ? mse_residual<true> : mse_residual<false>;
  mse<<<nb, kThreads, 0, s>>>(out, cpad, base, target, dout, work, P);
  sum_double<<<1, 256, 0, s>>>(work, nb, loss);
  return status(cudaGetLastError());
}

int lbm_nn_adam(float* w, float* m, float* v, const float* grad, void* w_bf16, long long n, float lr, float b1,
                float b2, float eps, int t, void* stream) {
  if (!w || !m || !v || !grad || n < 0 || t < 1) return -1;
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  if (n)
    adam_step<<<blocks(n), 256, 0, (cudaStream_t)stream>>>(w, m, v, grad, static_cast<__nv_bfloat16*>(w_bf16), n, lr,
                                                           b1, b2, eps, c1, c2);
  return status(cudaGetLastError());
}

int lbm_nn_to_bf16(const float* a, void* b, long long n, void* stream) {
  if (!a || !b || n < 0) return -1;
  if (n) to_bf16<<<blocks(n), 256, 0, (cudaStream_t)stream>>>(a, static_cast<__nv_bfloat16*>(b), n);
  return status(cudaGetLastError());
}

int lbm_nn_project(const float* out, int cpad, const float* phi0, const float* phi1, float* field, double* work,
                   long long work_len, int n, int h, int w, void* stream) {
  if (!out || cpad < 1 || !phi0 || !phi1 || !field || !work || n < 1 || h < 1 || w < 1) return -1;
  const int parts = 64;
  if (work_len < 3LL * parts * n) return -1;
  const long long hw = (long long)h * w;
  cudaStream_t s = (cudaStream_t)stream;
  const dim3 grid(parts, n);
  // one launch a pass needs the sums twice, and a field apart from phi1, whose sums are the target: else three
  const uintptr_t f0 = reinterpret_cast<uintptr_t>(field), q0 = reinterpret_cast<uintptr_t>(phi1), len = n * hw * 4;
  if (work_len >= 6LL * parts * n && (f0 + len <= q0 || q0 + len <= f0)) {
    double* const buf[2] = {work, work + 3LL * parts * n};
    project_stage<true, false, true><<<grid, kThreads, 0, s>>>(out, cpad, phi0, phi1, nullptr, buf[0], field, hw);
    for (int pass = 1; pass < kProjectPasses; ++pass)
      project_stage<false, true, true><<<grid, kThreads, 0, s>>>(out, cpad, phi0, phi1, buf[(pass - 1) & 1],
                                                                 buf[pass & 1], field, hw);
    project_stage<false, true, false><<<grid, kThreads, 0, s>>>(out, cpad, phi0, phi1, buf[(kProjectPasses - 1) & 1],
                                                                nullptr, field, hw);
    return status(cudaGetLastError());
  }
  project_stage<true, false, false><<<grid, kThreads, 0, s>>>(out, cpad, phi0, phi1, nullptr, nullptr, field, hw);
  for (int pass = 0; pass < kProjectPasses; ++pass) {
    project_stage<false, false, true><<<grid, kThreads, 0, s>>>(out, cpad, phi0, phi1, nullptr, work, field, hw);
    project_stage<false, true, false><<<grid, kThreads, 0, s>>>(out, cpad, phi0, phi1, work, nullptr, field, hw);
  }
  return status(cudaGetLastError());
}

}  // extern "C"

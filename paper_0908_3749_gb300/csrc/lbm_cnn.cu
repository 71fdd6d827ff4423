// lbm_cnn.cu -- training and inference kernels of the coarse-grid corrector
// (include/lbm_cnn.h).
//
// Activations and output gradients are BF16 in groups of 8 channels, row by
// row: element (y, x, c) of a C-channel image at
//   ((y * C/8 + c/8) * W + x) * 8 + c % 8,
// so that a tile of pixels with its halo is one TMA box whose shared-memory
// image holds, for every row and channel group, consecutive pixels 16 bytes
// apart: 8 pixels x 8 channels are 128 contiguous bytes, the unit of ldmatrix
// and of the tcgen05 operand layout, and a tap of the 3 x 3 stencil is an
// address offset (pixels outside the image are the box's zero fill).
// The input features stay FP32 and the first layer (4 -> 32) runs in FP32 on
// the CUDA cores. The other 3 x 3 convolutions are implicit GEMMs on the
// 5th-generation tensor cores (tcgen05, BF16 inputs, FP32 accumulation in tensor
// memory; mma.sync for 4 -> 32 channels): rows are pixels, the reduction index
// k = tap * CIN + ci runs over the 9 taps and the input channels, columns are output
// channels. The weights of a layer are packed once per update into [COUT][K] BF16 (K contiguous, the "col" operand) for
// the forward pass and into the tap-flipped, channel-transposed [CIN][K'] for
// the input-gradient pass, which is the same GEMM run on the output
// gradients. Weight gradients are contractions over the pixels, by tcgen05 too
// (the first layer's FP32 features as three BF16 parts), as
// per-CTA partials, then a fixed-order sum (reproducible). Adam keeps FP32
// master weights.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>  // header-only; ranges cost nothing without a profiler attached

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "../../include/lbm_cnn.h"
#include "dw.cuh"
#include "tc05.cuh"

namespace {

constexpr int NL = LBM_CNN_LAYERS;
constexpr int CH[NL + 1] = {4, 32, 32, 32, 32, 4};
__host__ __device__ constexpr int ru(int a, int m) { return (a + m - 1) / m * m; }

__host__ __device__ constexpr int wsize(int l) { return 9 * (l == 0 ? 4 : 32) * (l == NL - 1 ? 4 : 32); }
__host__ __device__ constexpr int cin_of(int l) { return l == 0 ? 4 : 32; }
__host__ __device__ constexpr int cout_of(int l) { return l == NL - 1 ? 4 : 32; }

__host__ __device__ constexpr int nout_of(int l) { return wsize(l) + cout_of(l); }
// Start of layer l in the packed parameter vector.
__host__ __device__ constexpr int param_offset(int l) { return l == 0 ? 0 : param_offset(l - 1) + nout_of(l - 1); }
static_assert(param_offset(NL) == LBM_CNN_NPARAMS, "packed parameters");
__host__ __device__ constexpr int kp_of(int l) { return ru(9 * cin_of(l), 16); }   // K of the forward operand
__host__ __device__ constexpr int kb_of(int l) { return ru(9 * cout_of(l), 16); }  // of the input-gradient one

// Results that a call hands to the host, in one copy.
struct Results {
  double loss;
  double mass[2];  // sums of the corrected and of the coarse density
  int timeout;     // a bounded wait expired in some kernel since the last report
  int skipped;     // updates left out since then
  unsigned done;   // blocks of k_apply finished
};

// Waits of the convolution and weight-gradient kernels: bounded; when one expires,
// the block sets Results::timeout, waits once more for the copies and products that
// it has in flight, frees its tensor memory and leaves. k_update then leaves
// the parameters alone. give_up (test hook): the waits that expire at once, in instances
// of the kernels of their own (HOOK): a look at it beside every wait takes 2 %.
enum GiveUp { GIVE_UP_COPIES = 1, GIVE_UP_PRODUCTS = 2 };
__device__ __forceinline__ bool wait_for(unsigned long long* bar, unsigned parity, bool give_up) {
  return !give_up && gbtma::mbar_wait_bounded(bar, parity, gbtma::TMA_WAIT_CYCLES);
}

// ---------------------------------------------------------------------------
// Tensor-core implicit-GEMM 3 x 3 convolution
// ---------------------------------------------------------------------------
enum Epi { EPI_RELU_BF16 = 0, EPI_LINEAR_F32 = 1, EPI_MASK_BF16 = 2 };

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4],
                                         unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, "
      "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Which values of a BF16 pair without negative numbers are positive, at bits 15
// (low value) and 31 (high value): 0x7fff + x sets the top bit of its half for
// every non-zero x, and no carry leaves the half.
__device__ __forceinline__ unsigned positive_bits(__nv_bfloat162 v) {
  return ((*reinterpret_cast<const unsigned*>(&v) & 0x7fff7fffu) + 0x7fff7fffu) & 0x80008000u;
}
// A pixel's word of 32 such bits: channels 8 j + 2 t, + 1 (j, t = 0..3) at bits
// 15 - s and 31 - s, s = j + 4 t.

constexpr unsigned PX_BYTES = 16;  // 8 BF16 channels of a pixel

// A box of `map` (3D: x in 32-bit words, channel group, row) whose first pixel
// is (x, y), all channel groups.
__device__ __forceinline__ void tma_load_box(void* dst, const CUtensorMap* map, int x, int y,
                                             unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4}], [%5];" ::"r"(gbtma::smem_addr(dst)),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(4 * x), "r"(0), "r"(y),
      "r"(gbtma::smem_addr(bar))
      : "memory");
}

// 32 -> COUT channels: out[p][c] = epilogue(sum_k patch(p, k) * Wt[c][k]) on the
// 5th-generation tensor cores. A tile is 16 x 16 output pixels, its input with
// a halo of one pixel one TMA box of 18 rows x 4 channel groups x 18 pixels. In
// shared memory 8 pixels of a row x 8 channels are a core matrix (128
// contiguous bytes), tile rows are CV_ROW apart: M = 128 rows of A are 8 pixels of 16
// rows, a tap is an offset of the start address, K = 16 two channel groups; nothing
// is gathered by threads. The packed weights stay in shared memory as core
// matrices of 8 output channels x 8 k. Persistent CTAs, two per SM, of six warps:
// one thread issues the copies, one the products (36 per tile: two M = 128 halves;
// K in order, tap by tap), four warps the epilogue, in which a thread holds all
// channels of a pixel; CV_SLOTS slots of a tile in shared memory and its
// accumulators in tensor memory go round between them.
// The results are those of mma.sync m16n8k16 over the same K steps, bit for bit.
// Bound by the tensor cores' reads of shared memory (5 KB per product, 5 us) and
// by the launch. Measured, 512 x 512, 32 -> 32 channels: 12.4 us with and without
// the mask; with one tile at a time per CTA (copy, products, epilogue in turn) 14 us; as
// mma.sync with ldmatrix fragments (8 us at its 1024 multiply-adds per clock and
// SM) 18 us; with patches gathered from global memory (L1 91 % busy) 67 us, and 72 us
// with the mask read from the activations.
constexpr int CV_X = 16, CV_Y = 16, CV_HX = CV_X + 2, CV_HY = CV_Y + 2;
constexpr int CV_EPI_T = 128, CV_T = CV_EPI_T + 64;  // epilogue threads; and two warps
constexpr int CV_CTAS_PER_SM = 2, CV_SLOTS = 4;
constexpr int CV_KG = 9 * 32 / 8;                          // groups of 8 k
constexpr unsigned CV_GROUP = CV_HX * PX_BYTES, CV_ROW = 4 * CV_GROUP;
constexpr unsigned CV_TILE = CV_HY * CV_ROW, CV_STAGE = (CV_TILE + 127) / 128 * 128;
__host__ __device__ constexpr int cv_n(int cout) { return cout == 32 ? 32 : 16; }  // N of the products (zero rows)
__host__ __device__ constexpr unsigned cv_smem(int cout) {
  return CV_SLOTS * CV_STAGE + CV_KG * cv_n(cout) * 16 + 128;
}

template <int COUT, int EPI, bool HOOK>
__global__ void __launch_bounds__(CV_T, CV_CTAS_PER_SM)
    k_conv(const __grid_constant__ CUtensorMap map, int H, int W, int tiles_x, int ntiles,
           const __nv_bfloat16* Wt, const float* bias,
           const unsigned* bits_in, __nv_bfloat16* out_bf,
           float* out_f, unsigned* bits_out, int* timeout,
           int give_up) {
  constexpr int NP = cv_n(COUT), TM = CV_SLOTS * 2 * NP;  // TMEM columns
  constexpr unsigned IDESC = tc05::idesc_f32acc(tc05::FMT_BF16, 128, NP);
  extern __shared__ __align__(128) unsigned char conv_raw[];
  unsigned char* const base = conv_raw + ((128u - (gbtma::smem_addr(conv_raw) & 127u)) & 127u);
  // per slot: copy landed; products complete; accumulators read
  __shared__ unsigned long long full[CV_SLOTS], done[CV_SLOTS], drained[CV_SLOTS];
  __shared__ unsigned s_tmem;
  __shared__ __align__(16) float s_bias[32];
  const int t = threadIdx.x, warp = t >> 5;
  const int G = (int)gridDim.x, mine = (ntiles - (int)blockIdx.x + G - 1) / G;  // tiles of this CTA
  gbtma::dependents_may_start();
  if (t == 0)
    for (int k = 0; k < CV_SLOTS; ++k) {
      gbtma::mbar_init(&full[k], 1);
      gbtma::mbar_init(&done[k], 1);
      gbtma::mbar_init(&drained[k], CV_EPI_T);
    }
  __syncthreads();
  gbtma::wait_for_previous();
  auto load = [&](int k) {  // the CTA's k-th tile into slot k % CV_SLOTS
    const int tile = (int)blockIdx.x + k * G, s = k % CV_SLOTS;
    gbtma::mbar_expect_tx(&full[s], CV_TILE);
    tma_load_box(base + s * CV_STAGE, &map, (tile % tiles_x) * CV_X - 1, (tile / tiles_x) * CV_Y - 1, &full[s]);
  };
  auto phase = [](int k) { return (unsigned)(k / CV_SLOTS) & 1u; };
  if (t == CV_EPI_T)  // the first tiles' copies run while the CTA sets up
    for (int k = 0; k < min(mine, CV_SLOTS); ++k) load(k);
  if (warp == 0) tc05::alloc(&s_tmem, TM);
  // Wt [ru(COUT, 8)][288] -> [k / 8][row][8]; rows beyond it zero
  unsigned char* const sw = base + CV_SLOTS * CV_STAGE;
  for (int i = t; i < NP * CV_KG; i += CV_T) {
    const int n = i / CV_KG, kg = i % CV_KG;
    *reinterpret_cast<uint4*>(sw + (kg * NP + n) * 16) =
        n < ru(COUT, 8) ? reinterpret_cast<const uint4*>(Wt)[i] : make_uint4(0, 0, 0, 0);
  }
  if (EPI != EPI_MASK_BF16 && t < COUT) s_bias[t] = bias[t];
  tc05::fence_async_smem();
  tc05::fence_before();
  __syncthreads();
  tc05::fence_after();
  const unsigned tmem = s_tmem, a0 = gbtma::smem_addr(base), b0 = gbtma::smem_addr(sw);

  // (no products without copies)
  const bool no_copy = HOOK && (give_up & GIVE_UP_COPIES), no_product = HOOK && give_up != 0;
  bool ok = true;  // every wait of this thread has ended in time
  int issued = 0;  // by this thread: tiles copied, tiles multiplied
  if (t == CV_EPI_T) {  // copies beyond the first CV_SLOTS: once the slot's products have read it
    for (issued = min(mine, CV_SLOTS); issued < mine; ++issued) {
      ok = wait_for(&done[issued % CV_SLOTS], phase(issued - CV_SLOTS), no_product);
      if (!ok) break;
      load(issued);
    }
  } else if (t == CV_EPI_T + 32) {  // products
    for (int k = 0; k < mine; ++k) {
      const int s = k % CV_SLOTS;
      if (k >= CV_SLOTS) ok = wait_for(&drained[s], phase(k - CV_SLOTS), no_product);
      ok = ok && wait_for(&full[s], phase(k), no_copy);
      if (!ok) break;
      tc05::fence_after();
      const unsigned as = a0 + s * CV_STAGE, ts = tmem + s * 2 * NP;
#pragma unroll 1
      for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int q = 0; q < 6; ++q)  // dx = q / 2, channels 16 (q % 2) ..
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const int ks = dy * 6 + q;
            tc05::mma_f16(ts + m * NP,
                          tc05::smem_desc(as + dy * CV_ROW + (8 * m + q / 2) * PX_BYTES + (q & 1) * 2 * CV_GROUP,
                                          CV_GROUP, CV_ROW),
                          tc05::smem_desc(b0 + ks * 2 * NP * 16, NP * 16, 128), IDESC, ks > 0 ? 1u : 0u);
          }
      tc05::commit(&done[s]);
      issued = k + 1;
    }
  } else if (t < CV_EPI_T) {  // epilogue: row t / 8 of the tile, pixels t % 8 and 8 + t % 8
    for (int k = 0; k < mine; ++k) {
      const int tile = (int)blockIdx.x + k * G, s = k % CV_SLOTS;
      const int x0 = (tile % tiles_x) * CV_X + (t & 7), y = (tile / tiles_x) * CV_Y + (t >> 3);
      // The ReLU masks (which channels of a pixel are positive), read while the
      // products run.
      unsigned keep[2] = {0u, 0u};
      if constexpr (EPI == EPI_MASK_BF16)
#pragma unroll
        for (int m = 0; m < 2; ++m)
          if (y < H && x0 + 8 * m < W) keep[m] = bits_in[(long long)y * W + x0 + 8 * m];
      ok = __all_sync(0xffffffffu, wait_for(&done[s], phase(k), no_product));
      if (!ok) break;
      tc05::fence_after();
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const int x = x0 + 8 * m;
        const unsigned lanes = tmem + ((unsigned)(warp * 32) << 16) + (s * 2 + m) * NP;
        float v[NP];
        if constexpr (NP == 16) tc05::ld16(lanes, v);
        else tc05::ld32(lanes, v);
        if (m == 1) {  // both halves are in registers
          tc05::fence_before();
          gbtma::mbar_arrive(&drained[s]);
        }
        if (y < H && x < W) {
          if constexpr (EPI == EPI_LINEAR_F32) {
            *reinterpret_cast<float4*>(out_f + ((long long)y * W + x) * 4) =
                make_float4(v[0] + s_bias[0], v[1] + s_bias[1], v[2] + s_bias[2], v[3] + s_bias[3]);
          } else {
            unsigned pos = 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              __nv_bfloat162 r[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const int c = 8 * j + 2 * i;
                if constexpr (EPI == EPI_RELU_BF16) {
                  r[i] = __floats2bfloat162_rn(fmaxf(v[c] + s_bias[c], 0.f), fmaxf(v[c + 1] + s_bias[c + 1], 0.f));
                  pos |= positive_bits(r[i]) >> (j + 4 * i);
                } else {
                  r[i] = __floats2bfloat162_rn(v[c] * (keep[m] & (0x8000u >> (j + 4 * i)) ? 1.f : 0.f),
                                               v[c + 1] * (keep[m] & (0x80000000u >> (j + 4 * i)) ? 1.f : 0.f));
                }
              }
              *reinterpret_cast<uint4*>(out_bf + (((long long)y * 4 + j) * W + x) * 8) =
                  *reinterpret_cast<const uint4*>(r);
            }
            if (EPI == EPI_RELU_BF16 && bits_out) bits_out[(long long)y * W + x] = pos;
          }
        }
        __syncwarp();
      }
    }
  }
  __syncwarp();
  if (__syncthreads_or(!ok)) {
    // A copy or products did not complete in time: record it; the threads that issued
    // them give the last of each slot (the others have been waited for) a second
    // bounded wait, so that nothing reads or writes this CTA's memory after it.
    if (t == 0) atomicExch(timeout, 1);
    for (int k = max(0, issued - CV_SLOTS); k < issued; ++k)
      gbtma::mbar_wait_bounded(t == CV_EPI_T ? &full[k % CV_SLOTS] : &done[k % CV_SLOTS], phase(k),
                               gbtma::TMA_WAIT_CYCLES);
    __syncwarp();
  }
  tc05::fence_before();
  __syncthreads();
  if (warp == 0) tc05::dealloc(tmem, TM);
}

// Tiles of the 4 -> 32 convolution and of the weight gradients: CT_Y x CT_X
// output pixels; their inputs with a halo of one pixel are one TMA box of CT_HY
// rows x channel groups x CT_HX pixels.
constexpr int CT_X = 32, CT_Y = 8, CT_HX = CT_X + 2, CT_HY = CT_Y + 2;
constexpr int CT_WARPS = 4, CT_T = 32 * CT_WARPS;  // a warp computes two rows

__device__ __forceinline__ void ldmatrix4(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ unsigned lds32(unsigned addr) {
  unsigned v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}

// The input gradient of the last layer, 4 -> 32 channels with the ReLU mask: its
// K = tap * 4 + ci (36, padded to 48) has no core matrices in the tile (8 k are
// two taps), so the fragments of mma.sync m16n8k16 are read from the tile word by
// word. Persistent CTAs of four warps, three per SM; a warp computes two rows of
// 32 pixels (four 16-pixel M tiles), the B fragments serve all four. 8 us at 512 x
// 512; 21 us with the patches and the activations' mask read from global memory.
constexpr int C4_KS = 3, C4_KP = 16 * C4_KS, C4_CTAS_PER_SM = 3;
// Weight rows in shared memory, 16 bytes longer than K: the 8 rows that an 8 x 8
// ldmatrix reads then start in different 16-byte bank groups.
constexpr int C4_PITCH = C4_KP + 8;
constexpr unsigned C4_ROW = CT_HX * PX_BYTES, C4_TILE = CT_HY * C4_ROW, C4_STAGE = (C4_TILE + 127) / 128 * 128;
constexpr unsigned C4_SMEM = C4_STAGE + 32 * C4_PITCH * 2 + 128;

template <bool HOOK>
__global__ void __launch_bounds__(CT_T, C4_CTAS_PER_SM)
    k_conv4(const __grid_constant__ CUtensorMap map, int H, int W, int tiles_x, int ntiles,
            const __nv_bfloat16* Wt, const unsigned* bits_in,
            __nv_bfloat16* out, int* timeout, int give_up) {
  extern __shared__ __align__(128) unsigned char conv_raw[];
  unsigned char* const base = conv_raw + ((128u - (gbtma::smem_addr(conv_raw) & 127u)) & 127u);
  __shared__ unsigned long long bar;
  const unsigned in = gbtma::smem_addr(base), sw = in + C4_STAGE;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, tig = lane & 3;
  const int G = (int)gridDim.x;
  auto load = [&](int tile) {
    gbtma::mbar_expect_tx(&bar, C4_TILE);
    tma_load_box(base, &map, (tile % tiles_x) * CT_X - 1, (tile / tiles_x) * CT_Y - 1, &bar);
  };
  gbtma::dependents_may_start();
  if (threadIdx.x == 0) gbtma::mbar_init(&bar, 1);
  gbtma::wait_for_previous();
  if (threadIdx.x == 0) load(blockIdx.x);  // the grid has at most ntiles CTAs
  constexpr int CHUNKS = C4_KP / 8;  // 16-byte pieces of a weight row
  for (int i = threadIdx.x; i < 32 * CHUNKS; i += CT_T)
    *reinterpret_cast<uint4*>(base + C4_STAGE + (i / CHUNKS) * (C4_PITCH * 2) + (i % CHUNKS) * 16) =
        reinterpret_cast<const uint4*>(Wt)[i];
  __syncthreads();

  for (int k = 0, tile = blockIdx.x; tile < ntiles; tile += G, ++k) {
    const bool more = tile + G < ntiles;
    const int x0 = (tile % tiles_x) * CT_X, y0 = (tile / tiles_x) * CT_Y + 2 * warp;
    // The ReLU masks (which channels of a pixel are positive) of this thread's
    // outputs, read while the tile's copy is in flight.
    unsigned keep[4][2];
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int y = y0 + (m >> 1), x = x0 + (m & 1) * 16 + h * 8 + g;
        keep[m][h] = y < H && x < W ? bits_in[(long long)y * W + x] << (4 * tig) : 0u;
      }
    if (!__syncthreads_and(wait_for(&bar, k & 1, HOOK && (give_up & GIVE_UP_COPIES)))) {
      // The copy did not land in time: record it, wait once more (bounded), leave.
      if (threadIdx.x == 0) {
        atomicExch(timeout, 1);
        gbtma::mbar_wait_bounded(&bar, k & 1, gbtma::TMA_WAIT_CYCLES);
      }
      return;
    }
    float acc[4][4][4];
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[m][j][0] = acc[m][j][1] = acc[m][j][2] = acc[m][j][3] = 0.f;
    // M tile m: row 2 warp + m / 2, pixels 16 (m % 2) .. + 15.
    const unsigned arow = in + 2 * warp * C4_ROW;
    const unsigned b_lane = (((lane & 7) + (lane >> 4) * 8) * C4_PITCH + ((lane >> 3) & 1) * 8) * 2;
#pragma unroll
    for (int ks = 0; ks < C4_KS; ++ks) {
      unsigned b[4][2];
#pragma unroll
      for (int j = 0; j < 4; j += 2) {
        unsigned r[4];
        ldmatrix4(r, sw + b_lane + j * 8 * C4_PITCH * 2 + ks * 32);
        b[j][0] = r[0]; b[j][1] = r[1]; b[j + 1][0] = r[2]; b[j + 1][1] = r[3];
      }
      // The thread's channel pairs belong to taps 4 ks + tig / 2 and 4 ks + 2 +
      // tig / 2 (zero beyond tap 8).
      const int t0 = ks * 4 + (tig >> 1), t1 = t0 + 2;
      const unsigned o0 = (t0 / 3) * C4_ROW + (t0 % 3) * PX_BYTES;
      const unsigned o1 = (t1 / 3) * C4_ROW + (t1 % 3) * PX_BYTES;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const unsigned px = arow + (m >> 1) * C4_ROW + ((m & 1) * 16 + g) * PX_BYTES + (tig & 1) * 4;
        unsigned a[4];
        a[0] = t0 < 9 ? lds32(px + o0) : 0u;
        a[1] = t0 < 9 ? lds32(px + 8 * PX_BYTES + o0) : 0u;
        a[2] = t1 < 9 ? lds32(px + o1) : 0u;
        a[3] = t1 < 9 ? lds32(px + 8 * PX_BYTES + o1) : 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_bf16(acc[m][j], a, b[j][0], b[j][1]);
      }
    }
    __syncthreads();  // the tile is free again
    if (threadIdx.x == 0 && more) load(tile + G);
    // Thread (g, tig) holds channels j * 8 + 2 tig, + 1 of pixels g and g + 8
    // of each M tile.
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int y = y0 + (m >> 1);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int x = x0 + (m & 1) * 16 + h * 8 + g;
        if (y >= H || x >= W) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<__nv_bfloat162*>(out + (((long long)y * 4 + j) * W + x) * 8 + tig * 2) =
              __floats2bfloat162_rn(acc[m][j][2 * h] * (keep[m][h] & (0x8000u >> j) ? 1.f : 0.f),
                                    acc[m][j][2 * h + 1] * (keep[m][h] & (0x80000000u >> j) ? 1.f : 0.f));
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Weight and bias gradients on the tensor cores (tcgen05)
// ---------------------------------------------------------------------------
// dW[tap][ci][co] = sum_p act[p + off(tap)][ci] dz[p][co] is a contraction
// over the pixels: D (M x N) = A (M x K) B (K x N), K = the pixels, N = the
// output channels (32, or 4 padded to 16). Both operands are MN-major: a core
// matrix is 8 pixels (K) x 8 channels, 128 contiguous bytes of the row-planar
// tiles that TMA copies, so nothing is gathered or transposed by threads.
//   A  the activations' tile with a halo of one pixel (10 x 34): its channel
//      groups lie CT_HX pixels apart, and the tile's rows follow each other
//      with the same stride, so the 16 core matrices of M = 128 run over
//      (row offset dy, channel group) and a start address picks the column
//      offset dx: three products (dx = -1, 0, 1) give the nine taps.
//      32-channel layers: 4 row offsets x 4 groups, the fourth offset unused;
//      first layer (FP32 features, 4 channels): each feature as three BF16
//      parts x = x0 + x1 + x2 (x0 = bf16(x), x1 = bf16(x - x0), x2 = bf16(x -
//      x0 - x1), the differences exact in FP32; 24 significant bits
//      together), 12 channels padded to 16: 8 row offsets x 2 groups, three
//      used; the epilogue adds the three parts' sums (x2 first), which gives
//      the contraction of the FP32 features.
//   B  the output gradients' tile (8 x 32, no halo). The last layer's 4
//      channels are one group with 4 zeros; the second group of N = 16 is
//      the box's zero fill.
// Pixels outside the image are zero fill in both. Persistent CTAs, two per SM,
// two stages: one thread issues a tile's 48 products (M = 128, K = 16) and
// commits them to the stage's mbarrier, which it waits for before the stage is
// copied into again; meanwhile the four warps add the tile's bias gradient
// (sum_p dz[p][co], FP32, a fixed order). At the end each thread reads its rows
// of the accumulators (tcgen05.ld) into the CTA's partial sums; k_update adds
// the partials of all CTAs in a fixed order.
// Bound by the tensor cores' reads of A and B from shared memory (5 KB per
// product; about 10 us at 512 x 512, 32 -> 32). Measured: 15 us (32 -> 32),
// 13 us (32 -> 4), 14 us (first layer); one CTA per SM with five stages 19 us; gathering and transposing the
// operands with threads took 83, 55 and 34 us, bound by L1 (83 %).
constexpr int WG_T = 128;
constexpr int WG_CTAS_PER_SM = 2;
constexpr unsigned WG_TMEM_COLS = 128;

template <int CG, int NP>
struct WgShape {
  static constexpr unsigned GROUP = CT_HX * PX_BYTES;   // bytes of one (row, group) of A
  static constexpr unsigned ROW = CG * GROUP;           // bytes of one tile row of A
  static constexpr int DY = 16 / CG;                    // row offsets that M = 128 spans
  static constexpr unsigned A_TX = CT_HY * ROW;         // copied
  static constexpr unsigned A_BYTES = ((CT_Y - 1 + DY) * ROW + 2 * PX_BYTES + 127) / 128 * 128;  // read
  static constexpr int BG = NP / 8;                     // channel groups of B
  static constexpr unsigned BGROUP = CT_X * PX_BYTES, BROW = BG * BGROUP;
  static constexpr unsigned B_BYTES = CT_Y * BROW;
  static constexpr unsigned STAGE = A_BYTES + B_BYTES;
  static_assert(STAGE % 128 == 0 && A_BYTES >= A_TX, "stages");
  static constexpr unsigned SMEM = 2 * STAGE + 128;
};

__device__ __forceinline__ float bf_lo(unsigned w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(unsigned w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ unsigned bf_bits(__nv_bfloat16 h) {
  return (unsigned)__bfloat16_as_ushort(h);
}

// The three BF16 parts of x (bit patterns).
__device__ __forceinline__ void split3(float x, unsigned (&p)[3]) {
  const __nv_bfloat16 h0 = __float2bfloat16_rn(x);
  const float r1 = x - __bfloat162float(h0);
  const __nv_bfloat16 h1 = __float2bfloat16_rn(r1);
  const __nv_bfloat16 h2 = __float2bfloat16_rn(r1 - __bfloat162float(h1));
  p[0] = bf_bits(h0);
  p[1] = bf_bits(h1);
  p[2] = bf_bits(h2);
}

// CG: channel groups of A (4: a 32-channel layer, 2: the split features); COUT
// output channels.
template <int CG, int COUT, bool HOOK>
__global__ void __launch_bounds__(WG_T, WG_CTAS_PER_SM)
    k_wgrad(const __grid_constant__ CUtensorMap act, const __grid_constant__ CUtensorMap dz,
            int tiles_x, int ntiles, float* partial, int* timeout, int give_up) {
  constexpr int NP = COUT == 32 ? 32 : 16;  // N of the MMA
  constexpr int CIN = CG == 4 ? 32 : 4;
  constexpr int NOUT = 9 * CIN * COUT + COUT;
  using S = WgShape<CG, NP>;
  constexpr unsigned IDESC = tc05::idesc_f32acc(tc05::FMT_BF16, 128, NP) | tc05::IDESC_A_MN | tc05::IDESC_B_MN;
  extern __shared__ __align__(128) unsigned char wg_raw[];
  unsigned char* const base = wg_raw + ((128u - (gbtma::smem_addr(wg_raw) & 127u)) & 127u);
  __shared__ unsigned long long full[2], used[2];  // copies landed; products done
  __shared__ unsigned s_tmem;
  __shared__ float s_db[32];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int G = (int)gridDim.x;
  auto load = [&](int tile, int st) {
    const int x = (tile % tiles_x) * CT_X, y = (tile / tiles_x) * CT_Y;
    unsigned char* const a = base + st * S::STAGE;
    gbtma::mbar_expect_tx(&full[st], S::A_TX + S::B_BYTES);
    tma_load_box(a, &act, x - 1, y - 1, &full[st]);
    tma_load_box(a + S::A_BYTES, &dz, x, y, &full[st]);
  };
  gbtma::dependents_may_start();
  if (t == 0)
    for (int k = 0; k < 2; ++k) {
      gbtma::mbar_init(&full[k], 1);
      gbtma::mbar_init(&used[k], 1);
    }
  gbtma::wait_for_previous();
  if (warp == 0) tc05::alloc(&s_tmem, WG_TMEM_COLS);
  if (t == 0) {
    load(blockIdx.x, 0);  // the grid has at most ntiles CTAs
  }
  tc05::fence_before();
  __syncthreads();
  tc05::fence_after();
  const unsigned tmem = s_tmem;

  float db[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // bias sums: pixel column `lane`, group `warp`
  const bool no_copy = HOOK && (give_up & GIVE_UP_COPIES), no_product = HOOK && (give_up & GIVE_UP_PRODUCTS);
  bool ok = true;
  int k = 0, loaded = 1, multiplied = 0;  // tiles copied and multiplied (thread 0)
  for (int tile = blockIdx.x; tile < ntiles; tile += G, ++k) {
    const int st = k & 1;
    if (t == 0) {
      // Stage 1 - st: tile k - 1's products must have read it (the bias sums
      // have, by the barrier at the end of the loop body).
      if (k > 0) ok = wait_for(&used[1 - st], ((k - 1) >> 1) & 1, no_product);
      if (ok && tile + G < ntiles) {
        load(tile + G, 1 - st);
        ++loaded;
      }
    }
    ok = __syncthreads_and(ok && wait_for(&full[st], (k >> 1) & 1, no_copy));
    if (!ok) break;
    const unsigned a = gbtma::smem_addr(base) + st * S::STAGE, b = a + S::A_BYTES;
    if (t == 0) {
      tc05::fence_after();
#pragma unroll 1
      for (int r = 0; r < CT_Y; ++r)
#pragma unroll
        for (int kg = 0; kg < CT_X / 16; ++kg)
#pragma unroll
          for (int dx = 0; dx < 3; ++dx)
            tc05::mma_f16(tmem + dx * NP,
                          tc05::smem_desc(a + r * S::ROW + (kg * 16 + dx) * PX_BYTES, 128, S::GROUP),
                          tc05::smem_desc(b + r * S::BROW + kg * 16 * PX_BYTES, 128, S::BGROUP), IDESC,
                          (k > 0 || r > 0 || kg > 0) ? 1u : 0u);
      tc05::commit(&used[st]);
      ++multiplied;
    }
    if (warp < COUT / 8 || warp == 0) {
#pragma unroll
      for (int r = 0; r < CT_Y; ++r) {
        const uint4 v = *reinterpret_cast<const uint4*>(base + st * S::STAGE + S::A_BYTES + r * S::BROW +
                                                        warp * S::BGROUP + lane * PX_BYTES);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const unsigned w = (&v.x)[c];
          db[2 * c] += bf_lo(w);
          db[2 * c + 1] += bf_hi(w);
        }
      }
    }
    __syncthreads();
  }
  // The last tile's products (every earlier one was waited for).
  if (ok) ok = wait_for(&used[(k - 1) & 1], ((k - 1) >> 1) & 1, no_product);
  ok = __syncthreads_and(ok);
  float* out = partial + (long long)blockIdx.x * NOUT;
  if (!ok) {
    // A copy or the products did not complete in time: record it, wait once more
    // (bounded) for the last copy and the last products of each stage (the others
    // have been waited for), free tensor memory.
    if (t == 0) {
      atomicExch(timeout, 1);
      for (int j = max(0, loaded - 2); j < loaded; ++j)
        gbtma::mbar_wait_bounded(&full[j & 1], (j >> 1) & 1, gbtma::TMA_WAIT_CYCLES);
      for (int j = max(0, multiplied - 2); j < multiplied; ++j)
        gbtma::mbar_wait_bounded(&used[j & 1], (j >> 1) & 1, gbtma::TMA_WAIT_CYCLES);
    }
    tc05::fence_before();
    __syncthreads();
    if (warp == 0) tc05::dealloc(tmem, WG_TMEM_COLS);
    return;
  }
  tc05::fence_after();
  const unsigned trow = tmem + ((unsigned)(warp * 32) << 16);
  if constexpr (COUT == 4) {  // D row = dy * 32 + ci: warp = dy, lane = ci
    for (int dx = 0; dx < 3; ++dx) {
      float v[16];
      tc05::ld16(trow + dx * NP, v);
      if (warp < 3)
        reinterpret_cast<float4*>(out)[(warp * 3 + dx) * 32 + lane] = make_float4(v[0], v[1], v[2], v[3]);
    }
  } else if constexpr (CG == 4) {
    // The rows of 32 sums through shared memory (every product has completed;
    // 16-byte pieces swizzled by row), so that a warp stores whole lines:
    // storing them from the threads that hold them took 11 of 26 us.
    float4* sD = reinterpret_cast<float4*>(base);
    static_assert(2 * S::STAGE >= 288 * 32 * sizeof(float), "epilogue scratch");
    for (int dx = 0; dx < 3; ++dx) {
      float v[32];
      tc05::ld32(trow + dx * NP, v);
      if (warp < 3)
#pragma unroll
        for (int c = 0; c < 8; ++c)
          sD[((warp * 3 + dx) * 32 + lane) * 8 + (c ^ (lane & 7))] =
              make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
    }
    __syncthreads();
    for (int i = t; i < 288 * 8; i += WG_T)
      reinterpret_cast<float4*>(out)[i] = sD[(i & ~7) + ((i & 7) ^ ((i >> 3) & 7))];
  } else {
    // D row = dy * 16 + part * 4 + ci, 48 rows used; the three parts are added
    // through shared memory (every product has completed).
    float* sD = reinterpret_cast<float*>(base);  // 64 rows x 33
    static_assert(2 * S::STAGE >= 64 * 33 * sizeof(float), "epilogue scratch");
    for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
      for (int cb = 0; cb < 2; ++cb) {
        float v[16];
        tc05::ld16(trow + dx * NP + cb * 16, v);
        if (t < 64)
#pragma unroll
          for (int c = 0; c < 16; ++c) sD[t * 33 + cb * 16 + c] = v[c];
      }
      __syncthreads();
      for (int i = t; i < 3 * 4 * 32; i += WG_T) {
        const int dy = i / 128, ci = (i >> 5) & 3, co = i & 31;
        const float* d = sD + (dy * 16 + ci) * 33 + co;
        out[((dy * 3 + dx) * 4 + ci) * 32 + co] = (d[8 * 33] + d[4 * 33]) + d[0];
      }
      __syncthreads();
    }
  }
  // bias: add the pixel columns (lanes) by a fixed butterfly; warp = group
#pragma unroll
  for (int c = 0; c < 8; ++c)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) db[c] += __shfl_xor_sync(0xffffffffu, db[c], o);
  if (lane == 0)
#pragma unroll
    for (int c = 0; c < 8; ++c) s_db[warp * 8 + c] = db[c];
  tc05::fence_before();
  __syncthreads();
  if (t < COUT) out[9 * CIN * COUT + t] = s_db[t];
  if (warp == 0) tc05::dealloc(tmem, WG_TMEM_COLS);
}

// First layer (4 -> 32 channels) in FP32 on the CUDA cores, straight from the
// FP32 input features [p][4]: 3 x 3 correlation with zero padding, bias,
// ReLU, stored BF16 for the tensor-core layers. Keeping the input in
// FP32 keeps differences between neighbouring nodes that are below one BF16
// step of the fields (smooth regions of fine-grained coarse grids).
// w: the layer's FP32 parameters, (3, 3, 4, 32) then 32 biases.
// A thread computes two neighbouring pixels of a row in paired FP32 (f32x2 over
// channel pairs; taps in order, as fused multiply-adds, zeros outside the
// image): the weights, read from shared memory four at a time by every thread
// alike, then serve two pixels. Bound by the FP32 units (7.8 us at 512 x 512):
// 17 us; one pixel per thread in scalar FP32 was bound by its shared-memory
// reads, 24 us.
constexpr int C0_T = 128;
__global__ void __launch_bounds__(C0_T) k_conv0(const float* xf, int H, int W,
                                                const float* w,
                                                __nv_bfloat16* out,
                                                unsigned* bits) {
  __shared__ __align__(16) float sw[9 * 4 * 32 + 32];
  gbtma::dependents_may_start();
  gbtma::wait_for_previous();
  for (int i = threadIdx.x; i < 9 * 4 * 32 + 32; i += C0_T) sw[i] = w[i];
  __syncthreads();
  const int W2 = (W + 1) / 2, q = blockIdx.x * C0_T + threadIdx.x;
  if (q >= H * W2) return;
  const int y = q / W2, x = 2 * (q - y * W2);
  float2 acc[2][16];
#pragma unroll
  for (int c = 0; c < 16; ++c)
    acc[0][c] = acc[1][c] = *reinterpret_cast<const float2*>(sw + 9 * 4 * 32 + 2 * c);
#pragma unroll
  for (int dy = 0; dy < 3; ++dy) {
    const int yy = y + dy - 1;
    float4 in[4];  // columns x - 1 .. x + 2
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int xx = x + k - 1;
      in[k] = yy >= 0 && yy < H && xx >= 0 && xx < W
                  ? reinterpret_cast<const float4*>(xf)[(long long)yy * W + xx]
                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
      for (int ci = 0; ci < 4; ++ci) {
        const float a = (&in[dx].x)[ci], b = (&in[dx + 1].x)[ci];
        const float2 a2 = make_float2(a, a), b2 = make_float2(b, b);
        const float4* row = reinterpret_cast<const float4*>(sw + ((dy * 3 + dx) * 4 + ci) * 32);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float4 k = row[c];
          const float2 k0 = make_float2(k.x, k.y), k1 = make_float2(k.z, k.w);
          acc[0][2 * c] = __ffma2_rn(a2, k0, acc[0][2 * c]);
          acc[0][2 * c + 1] = __ffma2_rn(a2, k1, acc[0][2 * c + 1]);
          acc[1][2 * c] = __ffma2_rn(b2, k0, acc[1][2 * c]);
          acc[1][2 * c + 1] = __ffma2_rn(b2, k1, acc[1][2 * c + 1]);
        }
      }
  }
#pragma unroll
  for (int n = 0; n < 2; ++n) {
    if (x + n >= W) break;
    unsigned pos = 0u;
#pragma unroll
    for (int cg = 0; cg < 4; ++cg) {
      __nv_bfloat162 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float2 s = acc[n][cg * 4 + k];
        v[k] = __floats2bfloat162_rn(fmaxf(s.x, 0.f), fmaxf(s.y, 0.f));
        pos |= positive_bits(v[k]) >> (cg + 4 * k);
      }
      *reinterpret_cast<uint4*>(out + (((long long)y * 4 + cg) * W + x + n) * 8) =
          *reinterpret_cast<const uint4*>(v);
    }
    if (bits) bits[(long long)y * W + x + n] = pos;
  }
}

// ---------------------------------------------------------------------------
// Features, loss, Adam, packing, correction, restriction
// ---------------------------------------------------------------------------
// log32(x) = (float)log(x), bit for bit, mostly on the FP32 units. GB300 retires
// one FP64 instruction per warp and 19 clocks, and log() takes about 31.
//
// x = 2^e m, m in [sqrt(1/2), sqrt(2)); with c the reciprocal of m rounded to a
// 1/128 grid (10 significant bits, from a table with -log c as two FP32 words)
//   log x = e log 2 - log c + log(1 + r),   r = m c - 1, |r| < 2^-7,
// r as an FP32 pair (m as 24 + 29 bits, the product's rounding error by an FMA,
// p - 1 exact), e log 2 as an exact product with a 13-bit word plus the rest,
// log(1 + r) = r + t by its Taylor series, t = r^2 (-1/2 + r/3 - r^2/4 + r^3/5 -
// r^4/6) in FP32 (|t| < 2^-15, truncation below 2^-51), the large terms added
// by TwoSum. What remains is the rounding of the small terms, below
//   delta = 2^-36 (1 + |e|),  and near x = 1 (e = 0, c = 1)  2^-20 |t| + 2^-21 |r_l|,
// with a factor of 2 to spare (5.1 roundings of t: 2^-37.3, 3 x 2^-40 per |e|). If the sum rounds to the same FP32 number with
// delta added and subtracted, so does log(x), which is within its last FP64
// bit of the true value; else (one value in 700 for x in [0.1, 10], and values that
// are not positive normal numbers) log() decides.
struct LogEntry {
  float c, lh, ll, pad;  // 1 / m, -log c = lh + ll
};
constexpr int LOG_J0 = 90, LOG_N = 93;  // grid points (LOG_J0 + k) / 128
__device__ __forceinline__ float log32(double x, const LogEntry* __restrict__ table) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  if ((unsigned)(hi - 0x00100000) >= 0x7fe00000u) return (float)log(x);
  const int e = (hi - 0x3fe6a09e) >> 20;  // 0x3fe6a09e: the high word of sqrt(1/2)
  const int mhi = hi - e * (1 << 20);
  const float mh = __int_as_float((int)(((unsigned)(mhi - 0x38000000) << 3) | (lo >> 29)));
  const float ml = (float)(lo & 0x1fffffffu) * (mhi >= 0x3ff00000 ? 0x1p-52f : 0x1p-53f);
  const int j = __float2int_rn(__fmul_rn(mh, 128.f));
  const float4 q = __ldg(reinterpret_cast<const float4*>(table) + (j - LOG_J0));
  const float c = q.x;
  const float p = __fmul_rn(mh, c);
  const float rh = __fsub_rn(p, 1.f), rl = __fmaf_rn(ml, c, __fmaf_rn(mh, c, -p));
  const float r = __fadd_rn(rh, rl);
  const float t = r * r * (-0.5f + r * (1.f / 3.f + r * (-0.25f + r * (0.2f - r * (1.f / 6.f)))));
  const float fe = (float)e;
  constexpr float LN2_H = 0x1.62ep-1f;                             // 13 bits
  constexpr float LN2_L = (float)(0.693147180559945309417 - (double)LN2_H);
  float s1, e1, s2, e2;
  d2v16::two_sum(__fmul_rn(fe, LN2_H), q.y, s1, e1);
  d2v16::two_sum(s1, rh, s2, e2);
  const float low = __fadd_rn(__fadd_rn(__fadd_rn(e1, e2), __fadd_rn(q.z, rl)), __fmaf_rn(fe, LN2_L, t));
  const float delta = e == 0 && c == 1.f ? __fmaf_rn(fabsf(t), 0x1p-20f, fabsf(rl) * 0x1p-21f)
                                         : __fmaf_rn(fabsf(fe), 0x1p-36f, 0x1p-36f);
  const float up = __fadd_rn(s2, __fadd_rn(low, delta)), down = __fadd_rn(s2, __fsub_rn(low, delta));
  return up == down ? up : (float)log(x);
}
// The table (host).
std::vector<LogEntry> log_table() {
  std::vector<LogEntry> t(LOG_N);
  for (int k = 0; k < LOG_N; ++k) {
    const double c = std::nearbyint(1024.0 * 128.0 / (LOG_J0 + k)) / 1024.0;
    const double l = -std::log(c);
    t[k].c = (float)c;
    t[k].lh = (float)l;
    t[k].ll = (float)(l - (double)t[k].lh);
    t[k].pad = 0.f;
  }
  return t;
}

// exp of an FP32 number in FP64, within 0.6 units in the last place: q = n log 2 /
// 64 + r with n log 2 / 64 as an exact product and a correction, 2^(j/64) (j = n
// mod 64) from a table as the sum of two doubles, exp(r) - 1 by its Taylor
// series (|r| < 0.0055, the r^7 / 5040 left out is below 2^-65), the power of two
// 2^(n div 64) added to the exponent: 13 FP64 instructions against about 20 for
// exp(), which takes what is not in the normal range.
struct ExpEntry {
  double h, l;
};
constexpr int EXP_N = 64;
__device__ __forceinline__ double exp32(float q, const ExpEntry* __restrict__ table) {
  if (!(fabsf(q) < 700.f)) return exp((double)q);
  const float nf = rintf(q * 92.33248f);  // 64 / log 2
  const int n = (int)nf;
  const double2 t = __ldg(reinterpret_cast<const double2*>(table) + (n & (EXP_N - 1)));
  constexpr double STEP = 0.693147180559945309417 / 64;
  constexpr double STEP_H = 0x1.62e42fefp-7;                 // 33 bits: n STEP_H is exact
  constexpr double STEP_L = 0x1.473de6af278edp-40;           // log 2 / 64 - STEP_H
  static_assert(STEP_H + STEP_L == STEP, "log 2 / 64");
  const double nd = (double)nf;
  const double r = fma(-nd, STEP_L, fma(-nd, STEP_H, (double)q));
  double c = fma(r, 1.0 / 720, 1.0 / 120);
  c = fma(c, r, 1.0 / 24);
  c = fma(c, r, 1.0 / 6);
  c = fma(c, r, 0.5);
  const double p = fma(c * r, r, r);
  const double v = t.x + fma(t.x, p, t.y);
  return __hiloint2double(__double2hiint(v) + ((n >> 6) << 20), __double2loint(v));
}
// The table (host): 2^(k/64) in extended precision as h + l.
std::vector<ExpEntry> exp_table() {
  std::vector<ExpEntry> t(EXP_N);
  for (int k = 0; k < EXP_N; ++k) {
    // l from h's own logarithm: 2^(k/64) = h exp(d), d = k log 2 / 64 - log h small,
    // in long double (64 significant bits or more).
    const long double x = exp2l((long double)k / 64);
    t[k].h = (double)x;
    t[k].l = (double)(x - (long double)t[k].h);
  }
  return t;
}

// Planes [4][H][W] (rho, u, v, T) -> features (log rho, u, v, log T) in FP32
// [p][4]; with `xs`, also their three BF16 parts (channel = part * 4 + feature,
// 12 of 16 channels, row-planar; the other 4 stay zero).
// Bound by memory (80 bytes a pixel with xs): 512 x 512 7 us; 33 us with the FP64
// logarithms (the loss kernel, which takes the target's, 41 -> 16 us).
__global__ void k_features(const double* f, int npix, int W, float* xf,
                           __nv_bfloat16* xs, const LogEntry* __restrict__ logs) {
  gbtma::dependents_may_start();
  gbtma::wait_for_previous();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npix) return;
  const float4 q = make_float4(log32(f[p], logs), (float)f[npix + p], (float)f[2 * npix + p],
                               log32(f[3 * npix + p], logs));
  reinterpret_cast<float4*>(xf)[p] = q;
  if (xs) {
    unsigned s[4][3];
    split3(q.x, s[0]);
    split3(q.y, s[1]);
    split3(q.z, s[2]);
    split3(q.w, s[3]);
    const int y = p / W, x = p - y * W;
    uint4* const o = reinterpret_cast<uint4*>(xs) + (long long)y * 2 * W + x;
    o[0] = make_uint4(s[0][0] | s[1][0] << 16, s[2][0] | s[3][0] << 16,
                      s[0][1] | s[1][1] << 16, s[2][1] | s[3][1] << 16);
    o[W] = make_uint4(s[0][2] | s[1][2] << 16, s[2][2] | s[3][2] << 16, 0u, 0u);
  }
}

// out = x + z; d = out - target; dz = 2 d / N (BF16); block partial of sum d^2.
// Per-channel output scale: the network predicts the correction of feature
// c in units of s[c] (out = x + s z).
struct Scale4 {
  float s[4];
};

// Loss per element of d = out - target: d^2 (LBM_CNN_LOSS_MSE) or |d|
// (LBM_CNN_LOSS_L1, whose gradient is sign(d), 0 at d = 0), and its gradient
// with respect to the network's output (BF16, 4 channels and 4 zeros). A pixel
// per thread, whose target features are taken here; the sums in FP64, per block.
__global__ void __launch_bounds__(256) k_loss(const float4* xf, const float4* z,
                                              const double* target, int npix,
                                              uint4* dz, double* partial,
                                              const Scale4 sc, int l1,
                                              const LogEntry* __restrict__ logs) {
  __shared__ double sm[8];
  gbtma::dependents_may_start();
  gbtma::wait_for_previous();
  const int p = blockIdx.x * 256 + threadIdx.x;
  double s = 0.0;
  if (p < npix) {
    const float4 x4 = xf[p], z4 = z[p];
    const float4 t4 = make_float4(log32(target[p], logs), (float)target[npix + p],
                                  (float)target[2 * npix + p], log32(target[3 * npix + p], logs));
    const float n = (float)(4 * npix);
    unsigned g[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float k = sc.s[c];
      const float d = (&x4.x)[c] + k * (&z4.x)[c] - (&t4.x)[c];
      if (l1) {
        s += fabs((double)d);
        const float sg = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
        g[c] = bf_bits(__float2bfloat16(k * sg / n));
      } else {
        s += (double)d * d;
        g[c] = bf_bits(__float2bfloat16(2.f * k * d / n));
      }
    }
    dz[p] = make_uint4(g[0] | g[1] << 16, g[2] | g[3] << 16, 0u, 0u);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) s += sm[w];
    partial[blockIdx.x] = s;
  }
}

// After the backward pass, one launch: the gradients from the weight-gradient
// partials, the loss from its partials and, with `adam`, the update of the
// FP32 parameters and of their packed BF16 copies (k_pack's positions; their
// padding stays zero). A block takes UP_N parameters, the threads of a
// parameter every UP_S-th partial, added in a fixed order; the last block takes
// the loss. Bound by the read of the partials (36 MB at 304 CTAs, from the L2):
// 14 us. One thread per parameter in a launch per layer, one thread for the
// loss, and launches of their own for Adam and each layer's packing took 117 +
// 195 + 13 us.
constexpr int UP_N = 32, UP_S = 8;
struct UpdateArgs {
  const float* part[NL];  // [blocks][nout_of(l)]
  int nblocks;
  float *w, *m, *v, *grad;
  __nv_bfloat16 *wt[NL], *wb[NL];
  const double* lpart;    // loss partials
  int nl;
  double lscale;
  Results* res;           // loss, timeout, skipped
  int adam;
  float lr, b1, b2, eps, c1, c2;
};
__global__ void __launch_bounds__(UP_N * UP_S) k_update(const UpdateArgs A) {
  gbtma::dependents_may_start();
  gbtma::wait_for_previous();
  const int t = threadIdx.x;
  // A wait of a kernel before expired: its partials are not this step's. Nothing
  // is updated; the host learns of it from the flag (which arrives beside the partials).
  const int expired = *(volatile int*)&A.res->timeout;
  if (blockIdx.x == gridDim.x - 1) {
    __shared__ double sl[UP_N * UP_S];
    double s = 0.0;
    for (int i = t; i < A.nl; i += UP_N * UP_S) s += A.lpart[i];
    sl[t] = s;
    __syncthreads();
    for (int st = UP_N * UP_S / 2; st > 0; st >>= 1) {
      if (t < st) sl[t] += sl[t + st];
      __syncthreads();
    }
    if (t == 0 && !expired) A.res->loss = sl[0] * A.lscale;
    if (t == 0 && expired && A.adam) ++A.res->skipped;
    return;
  }
  __shared__ float sm[UP_S][UP_N];
  const int i = blockIdx.x * UP_N + (t % UP_N), slice = t / UP_N;
  int l = 0;
#pragma unroll
  for (int k = 1; k < NL; ++k) l += i >= param_offset(k);
  const int j = i - param_offset(l);
  float s = 0.f;
  if (i < LBM_CNN_NPARAMS) {
    const int n = nout_of(l);
    const float* q = A.part[l] + j;
#pragma unroll 8
    for (int b = slice; b < A.nblocks; b += UP_S) s += q[(long long)b * n];
  }
  sm[slice][t % UP_N] = s;
  __syncthreads();
  if (slice > 0 || i >= LBM_CNN_NPARAMS || expired) return;
#pragma unroll
  for (int k = 1; k < UP_S; ++k) s += sm[k][t];
  A.grad[i] = s;
  if (!A.adam) return;
  const float mi = A.b1 * A.m[i] + (1.f - A.b1) * s;
  const float vi = A.b2 * A.v[i] + (1.f - A.b2) * s * s;
  A.m[i] = mi;
  A.v[i] = vi;
  const float wi = A.w[i] - A.lr * (mi / A.c1) / (sqrtf(vi / A.c2) + A.eps);
  A.w[i] = wi;
  if (l == 0 || j >= wsize(l)) return;  // the first layer and the biases are used in FP32
  const int cin = cin_of(l), cout = cout_of(l);
  const int co = j % cout, ci = j / cout % cin, tap = j / (cout * cin);
  const __nv_bfloat16 h = __float2bfloat16(wi);
  A.wt[l][co * kp_of(l) + tap * cin + ci] = h;
  A.wb[l][ci * kb_of(l) + (8 - tap) * cout + co] = h;
}

// Packs layer l's FP32 w[3][3][cin][cout] into the forward operand
// Wt[cout_p][kp] (k = tap cin + ci) and the input-gradient operand
// Wb[cin_p][kb] (k' = tap' cout + co with tap' = 8 - tap), BF16, zero padded.
__global__ void k_pack(const float* __restrict__ w, int cin, int cout, int kp, int coutp,
                       int kb, int cinp, __nv_bfloat16* __restrict__ wt,
                       __nv_bfloat16* __restrict__ wb) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < coutp * kp) {
    const int c = i / kp, k = i % kp;
    float val = 0.f;
    if (c < cout && k < 9 * cin) {
      const int tap = k / cin, ci = k % cin;
      val = w[(tap * cin + ci) * cout + c];
    }
    wt[i] = __float2bfloat16(val);
  }
  if (i < cinp * kb) {
    const int ci = i / kb, k = i % kb;
    float val = 0.f;
    if (ci < cin && k < 9 * cout) {
      const int tp = k / cout, co = k % cout, tap = 8 - tp;
      val = w[(tap * cin + ci) * cout + co];
    }
    wb[i] = __float2bfloat16(val);
  }
}

// corrected planes from output features x + z and the two masses (NaN for a
// non-finite output): block partial sums, added by the block that finishes
// last in a fixed order. Bound by the FP64 units (two exponentials per pixel):
// 512 x 512 about 20 us; 32 us with exp(), FP64 finiteness checks and the partials
// added by the host.
__global__ void __launch_bounds__(256) k_apply(const float4* xf, const float4* z,
                                               int npix, double* out,
                                               const double* coarse,
                                               double* partial, const Scale4 sc,
                                               const ExpEntry* __restrict__ exps, Results* res) {
  __shared__ double sm[2][256];
  __shared__ bool s_last;
  gbtma::dependents_may_start();
  gbtma::wait_for_previous();
  const int p = blockIdx.x * 256 + threadIdx.x, t = threadIdx.x;
  double r = 0.0, r0 = 0.0;
  if (p < npix) {
    const float4 x4 = xf[p], z4 = z[p];
    const float q0 = x4.x + sc.s[0] * z4.x, q1 = x4.y + sc.s[1] * z4.y;
    const float q2 = x4.z + sc.s[2] * z4.z, q3 = x4.w + sc.s[3] * z4.w;
    r = exp32(q0, exps);
    out[p] = r;
    out[npix + p] = q1;
    out[2 * npix + p] = q2;
    out[3 * npix + p] = exp32(q3, exps);
    r0 = coarse[p];
    if ((__double2hiint(r) & 0x7fffffff) >= 0x7ff00000 || !isfinite(q1) || !isfinite(q2) || !isfinite(q3))
      r = nan("");
  }
  auto block_sum = [&](double a, double b) {  // into sm[.][0]
    sm[0][t] = a;
    sm[1][t] = b;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
      if (t < st) {
        sm[0][t] += sm[0][t + st];
        sm[1][t] += sm[1][t + st];
      }
      __syncthreads();
    }
  };
  block_sum(r, r0);
  if (t == 0) {
    partial[2 * blockIdx.x] = sm[0][0];
    partial[2 * blockIdx.x + 1] = sm[1][0];
    __threadfence();
    s_last = atomicAdd(&res->done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double a = 0.0, b = 0.0;
  for (int i = t; i < (int)gridDim.x; i += 256) {
    a += __ldcg(partial + 2 * i);
    b += __ldcg(partial + 2 * i + 1);
  }
  block_sum(a, b);
  if (t == 0) {
    res->mass[0] = sm[0][0];
    res->mass[1] = sm[1][0];
    res->done = 0;
  }
}

// Block partial sums of (t - x)^2 per feature channel, [block][4].
__global__ void k_residual_sq(const float* __restrict__ xf, const float* __restrict__ tf, int npix,
                              double* __restrict__ partial) {
  __shared__ double sm[4][256];
  const int p = blockIdx.x * 256 + threadIdx.x;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const double d = p < npix ? (double)tf[4 * p + c] - (double)xf[4 * p + c] : 0.0;
    sm[c][threadIdx.x] = d * d;
  }
  __syncthreads();
  for (int st = 128; st > 0; st >>= 1) {
    if ((int)threadIdx.x < st)
#pragma unroll
      for (int c = 0; c < 4; ++c) sm[c][threadIdx.x] += sm[c][threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x < 4) partial[4 * blockIdx.x + threadIdx.x] = sm[threadIdx.x][0];
}

__global__ void k_restrict(const double* __restrict__ f, int Hf, int Wf, int r,
                           double* __restrict__ c) {
  const int Hc = Hf / r, Wc = Wf / r;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= Hc * Wc) return;
  const int Y = p / Wc, X = p % Wc;
  const long long nf = (long long)Hf * Wf;
  double R = 0, JX = 0, JY = 0, E = 0;
  for (int a = 0; a < r; ++a)
    for (int b = 0; b < r; ++b) {
      const long long q = (long long)(Y * r + a) * Wf + (X * r + b);
      const double rho = f[q], u = f[nf + q], v = f[2 * nf + q], T = f[3 * nf + q];
      R += rho;
      JX += rho * u;
      JY += rho * v;
      E += rho * T + 0.5 * rho * (u * u + v * v);
    }
  const double inv = 1.0 / (r * r);
  R *= inv; JX *= inv; JY *= inv; E *= inv;
  const double U = JX / R, V = JY / R;
  const long long nc = (long long)Hc * Wc;
  c[p] = R;
  c[nc + p] = U;
  c[2 * nc + p] = V;
  c[3 * nc + p] = E / R - 0.5 * (U * U + V * V);
}

thread_local std::string g_cnn_error = "no error";

// Pinned host copies of Results, 4 KB of them at a time: pinning memory costs 0.4 ms, as
// much as the rest of creating a small network, and a copy to memory that is not
// pinned 4 us of every call. Networks give their slot back when they are destroyed;
// the pages stay for the next ones.
class PinnedResults {
 public:
  cudaError_t get(Results** out) {
    std::lock_guard<std::mutex> lock(m_);
    cudaPointerAttributes at;
    // (a reset of the device frees them)
    if (!free_.empty() && (cudaPointerGetAttributes(&at, free_.back()) != cudaSuccess || at.type != cudaMemoryTypeHost))
      free_.clear();
    if (free_.empty()) {
      Results* page = nullptr;
      const cudaError_t e = cudaHostAlloc((void**)&page, SLOTS * sizeof(Results), cudaHostAllocPortable);
      if (e != cudaSuccess) return e;
      for (int k = 0; k < SLOTS; ++k) free_.push_back(page + k);
    }
    *out = free_.back();
    free_.pop_back();
    return cudaSuccess;
  }
  void put(Results* r) {
    std::lock_guard<std::mutex> lock(m_);
    free_.push_back(r);
  }

 private:
  static constexpr int SLOTS = 4096 / sizeof(Results);
  std::mutex m_;
  std::vector<Results*> free_;
};
PinnedResults& pinned_results() {
  static PinnedResults* const p = new PinnedResults;  // outlives every network, also at exit
  return *p;
}

}  // namespace

struct lbm_cnn {
  int H = 0, W = 0, npix = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  unsigned char* slab = nullptr;  // the one allocation, of which all buffers are parts
  float* w = nullptr;        // FP32 master parameters (packed)
  float* m = nullptr;
  float* v = nullptr;
  float* grad = nullptr;
  __nv_bfloat16* wt[NL] = {};
  __nv_bfloat16* wb[NL] = {};
  __nv_bfloat16* act[NL] = {};  // act[l] = relu output of layer l-1; [0] of these four is unused
  unsigned* pos[NL] = {};       // pos[l]: which channels of act[l] are positive, a word per pixel
  __nv_bfloat16* dz[2] = {};    // ping-pong output gradients (32 channels)
  __nv_bfloat16* dz5 = nullptr; // output gradients of the last layer: 4 channels and 4 zeros
  __nv_bfloat16* xs = nullptr;  // input features as three BF16 parts (16 channels)
  CUtensorMap c_act[NL], c_dz[2];        // convolution tiles with halo of act[1..], dz[]
  CUtensorMap m_act[NL], m_dz5, m_xs;    // weight-gradient tiles with halo of act[1..], dz5, xs
  CUtensorMap g_dz[2], g_dz5;            // the same without halo of dz[], dz5
  int tiles_x = 0, ntiles = 0;    // weight-gradient tiles
  int ctiles_x = 0, cntiles = 0;  // convolution tiles
  int sms = 0;
  LogEntry* logs = nullptr;     // table of log32
  ExpEntry* exps = nullptr;     // table of exp32
  Results* res = nullptr;       // device
  Results* h_res = nullptr;     // pinned host copy
  float* xf = nullptr;          // input features FP32 [p][4]
  float* tf = nullptr;          // target features FP32 [p][4]
  float* z = nullptr;           // last layer output FP32 [p][4]
  float* wpartial = nullptr;    // weight-gradient partials, layer by layer
  double* dpart = nullptr;      // loss / mass / residual partials
  int wblocks = 0;              // persistent CTAs of the weight gradients
  long long step = 0;
  float lr = 1e-3f, b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  Scale4 scale = {{1.f, 1.f, 1.f, 1.f}};
  int loss_kind = LBM_CNN_LOSS_MSE;
  int give_up = 0;  // test hook: GiveUp
  std::string err = "no error";
};

namespace {

int cfail(lbm_cnn* n, int code, const std::string& msg) {
  if (n) n->err = msg; else g_cnn_error = msg;
  return code;
}
#define CCK(n, call)                                                              \
  do {                                                                            \
    cudaError_t e_ = (call);                                                      \
    if (e_ != cudaSuccess)                                                        \
      return cfail(n, e_ == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA, \
                   std::string(#call) + ": " + cudaGetErrorString(e_));          \
  } while (0)

int pack_all(lbm_cnn* n) {
  for (int l = 1; l < NL; ++l) {  // the first layer uses its FP32 weights
    const int cin = cin_of(l), cout = cout_of(l);
    const int kp = kp_of(l), coutp = ru(cout, 8), kb = kb_of(l), cinp = ru(cin, 8);
    const int total = std::max(coutp * kp, cinp * kb);
    k_pack<<<(total + 255) / 256, 256, 0, n->stream>>>(n->w + param_offset(l), cin, cout, kp,
                                                        coutp, kb, cinp, n->wt[l], n->wb[l]);
    CCK(n, cudaGetLastError());
  }
  return LBM_OK;
}

// Forgets an expired wait.
int clear_timeout(lbm_cnn* n) {
  static_assert(offsetof(Results, skipped) == offsetof(Results, timeout) + sizeof(int), "one memset");
  CCK(n, cudaMemsetAsync(&n->res->timeout, 0, 2 * sizeof(int), n->stream));
  return LBM_OK;
}

// Copies the results to the host (n->h_res), synchronises and reports an
// expired wait, once: the updates since it were left out, and their numbers are
// taken back.
int fetch_results(lbm_cnn* n) {
  CCK(n, cudaMemcpyAsync(n->h_res, n->res, sizeof(Results), cudaMemcpyDeviceToHost, n->stream));
  CCK(n, cudaStreamSynchronize(n->stream));
  if (!n->h_res->timeout) return LBM_OK;
  n->step -= n->h_res->skipped;
  const int rc = clear_timeout(n);
  return rc != LBM_OK ? rc
                      : cfail(n, LBM_ERR_TIMEOUT, "a tile load (TMA) or product did not complete within its time limit");
}

// Tensor map of a row-planar BF16 image of `ncg` channel groups: dims (x in
// 32-bit words, channel group, row); box = `px` pixels of `rows` rows and
// `box_cg` groups (those beyond ncg are zero fill).
int encode_image(lbm_cnn* n, const void* p, int ncg, int box_cg, int px, int rows, CUtensorMap* out) {
  gbtma::EncodeTiledFn enc = gbtma::tensor_map_encoder();
  if (!enc) return cfail(n, LBM_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
  const cuuint64_t dims[3] = {(cuuint64_t)n->W * 4, (cuuint64_t)ncg, (cuuint64_t)n->H};
  const cuuint64_t strides[2] = {(cuuint64_t)n->W * PX_BYTES, (cuuint64_t)n->W * PX_BYTES * ncg};
  const cuuint32_t box[3] = {4u * (cuuint32_t)px, (cuuint32_t)box_cg, (cuuint32_t)rows};
  const cuuint32_t es[3] = {1, 1, 1};
  const CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<void*>(p), dims, strides, box,
                         es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS)
    return cfail(n, LBM_ERR_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return LBM_OK;
}

template <int COUT, int EPI>
int conv(lbm_cnn* n, const CUtensorMap& in, const __nv_bfloat16* wt, const float* bias,
         const unsigned* bits_in, __nv_bfloat16* ob, float* of, unsigned* bits_out = nullptr) {
  const int grid = std::min(n->cntiles, CV_CTAS_PER_SM * n->sms);
  CCK(n, gbtma::launch_overlapped(n->give_up ? k_conv<COUT, EPI, true> : k_conv<COUT, EPI, false>, grid, CV_T, cv_smem(COUT), n->stream, in, n->H, n->W,
                                  n->ctiles_x, n->cntiles, wt, bias, bits_in, ob, of, bits_out,
                                  &n->res->timeout, n->give_up));
  return LBM_OK;
}

// `train`: also store which activations are positive, for the backward pass.
int forward(lbm_cnn* n, const double* coarse, bool train) {
  int rc;
  auto bits = [&](int l) { return train ? n->pos[l] : nullptr; };
  CCK(n, gbtma::launch_overlapped(k_features, (n->npix + 255) / 256, 256, 0, n->stream, coarse, n->npix, n->W,
                                  n->xf, train ? n->xs : nullptr, n->logs));
  const float* w = n->w;
  CCK(n, gbtma::launch_overlapped(k_conv0, (n->H * ((n->W + 1) / 2) + C0_T - 1) / C0_T, C0_T, 0, n->stream,
                                  n->xf, n->H, n->W, w + param_offset(0), n->act[1], bits(1)));
  if ((rc = conv<32, EPI_RELU_BF16>(n, n->c_act[1], n->wt[1], w + param_offset(1) + wsize(1), nullptr, n->act[2], nullptr, bits(2))) != LBM_OK) return rc;
  if ((rc = conv<32, EPI_RELU_BF16>(n, n->c_act[2], n->wt[2], w + param_offset(2) + wsize(2), nullptr, n->act[3], nullptr, bits(3))) != LBM_OK) return rc;
  if ((rc = conv<32, EPI_RELU_BF16>(n, n->c_act[3], n->wt[3], w + param_offset(3) + wsize(3), nullptr, n->act[4], nullptr, bits(4))) != LBM_OK) return rc;
  if ((rc = conv<4, EPI_LINEAR_F32>(n, n->c_act[4], n->wt[4], w + param_offset(4) + wsize(4), nullptr, nullptr, n->z)) != LBM_OK) return rc;
  return LBM_OK;
}

template <int CG, int COUT>
int wgrad(lbm_cnn* n, const CUtensorMap& act, const CUtensorMap& dz, float* partial) {
  CCK(n, gbtma::launch_overlapped(n->give_up ? k_wgrad<CG, COUT, true> : k_wgrad<CG, COUT, false>, n->wblocks, WG_T, WgShape<CG, COUT == 32 ? 32 : 16>::SMEM,
                                  n->stream, act, dz, n->tiles_x, n->ntiles, partial, &n->res->timeout, n->give_up));
  return LBM_OK;
}

// Loss against the target features and all gradients into n->grad; with
// `adam`, one optimiser step (n->step is its number).
int loss_backward(lbm_cnn* n, const double* target, bool adam) {
  const int nb = (n->npix + 255) / 256;
  int rc;
  CCK(n, gbtma::launch_overlapped(k_loss, nb, 256, 0, n->stream, (const float4*)n->xf, (const float4*)n->z, target,
                                  n->npix, (uint4*)n->dz5, n->dpart, n->scale,
                                  n->loss_kind == LBM_CNN_LOSS_L1, n->logs));
  UpdateArgs U = {};
  for (int l = 0; l < NL; ++l) {
    U.part[l] = n->wpartial + (size_t)n->wblocks * param_offset(l);
    U.wt[l] = n->wt[l];
    U.wb[l] = n->wb[l];
  }
  auto part = [&](int l) { return const_cast<float*>(U.part[l]); };
  // layer 5 (32 -> 4): dz5 holds d loss / d z5
  if ((rc = wgrad<4, 4>(n, n->m_act[4], n->g_dz5, part(4))) != LBM_OK) return rc;
  CCK(n, gbtma::launch_overlapped(n->give_up ? k_conv4<true> : k_conv4<false>, std::min(n->ntiles, C4_CTAS_PER_SM * n->sms), CT_T, C4_SMEM, n->stream,
                                  n->m_dz5, n->H, n->W, n->tiles_x, n->ntiles, n->wb[4], n->pos[4], n->dz[1],
                                  &n->res->timeout, n->give_up));
  if ((rc = wgrad<4, 32>(n, n->m_act[3], n->g_dz[1], part(3))) != LBM_OK) return rc;
  if ((rc = conv<32, EPI_MASK_BF16>(n, n->c_dz[1], n->wb[3], nullptr, n->pos[3], n->dz[0], nullptr)) != LBM_OK) return rc;
  if ((rc = wgrad<4, 32>(n, n->m_act[2], n->g_dz[0], part(2))) != LBM_OK) return rc;
  if ((rc = conv<32, EPI_MASK_BF16>(n, n->c_dz[0], n->wb[2], nullptr, n->pos[2], n->dz[1], nullptr)) != LBM_OK) return rc;
  if ((rc = wgrad<4, 32>(n, n->m_act[1], n->g_dz[1], part(1))) != LBM_OK) return rc;
  if ((rc = conv<32, EPI_MASK_BF16>(n, n->c_dz[1], n->wb[1], nullptr, n->pos[1], n->dz[0], nullptr)) != LBM_OK) return rc;
  if ((rc = wgrad<2, 32>(n, n->m_xs, n->g_dz[0], part(0))) != LBM_OK) return rc;
  U.nblocks = n->wblocks;
  U.w = n->w;
  U.m = n->m;
  U.v = n->v;
  U.grad = n->grad;
  U.lpart = n->dpart;
  U.nl = nb;
  U.lscale = 1.0 / (4.0 * n->npix);
  U.res = n->res;
  U.adam = adam;
  U.lr = n->lr;
  U.b1 = n->b1;
  U.b2 = n->b2;
  U.eps = n->eps;
  if (adam) {
    U.c1 = 1.f - powf(n->b1, (float)n->step);
    U.c2 = 1.f - powf(n->b2, (float)n->step);
  }
  CCK(n, gbtma::launch_overlapped(k_update, (LBM_CNN_NPARAMS + UP_N - 1) / UP_N + 1, UP_N * UP_S, 0, n->stream, U));
  return LBM_OK;
}

}  // namespace

extern "C" {

int lbm_cnn_create(int H, int W, void* cuda_stream, lbm_cnn** out) {
  if (!out) return cfail(nullptr, LBM_ERR_INVALID, "out is NULL");
  *out = nullptr;
  if (H < 1 || W < 1 || (long long)H * W > (1ll << 26))
    return cfail(nullptr, LBM_ERR_INVALID, "bad image size");
  lbm_cnn* n = new lbm_cnn();
  n->H = H;
  n->W = W;
  n->npix = H * W;
  cudaError_t e = cudaSuccess;
  if (cuda_stream) n->stream = (cudaStream_t)cuda_stream;
  else { e = cudaStreamCreate(&n->stream); n->own_stream = true; }
  const size_t P = n->npix;
  int dev = 0, sms = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  auto allow = [&](const void* k, size_t bytes) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  allow((const void*)k_wgrad<4, 32, false>, WgShape<4, 32>::SMEM);
  allow((const void*)k_wgrad<4, 32, true>, WgShape<4, 32>::SMEM);
  allow((const void*)k_wgrad<4, 4, false>, WgShape<4, 16>::SMEM);
  allow((const void*)k_wgrad<4, 4, true>, WgShape<4, 16>::SMEM);
  allow((const void*)k_wgrad<2, 32, false>, WgShape<2, 32>::SMEM);
  allow((const void*)k_wgrad<2, 32, true>, WgShape<2, 32>::SMEM);
  allow((const void*)k_conv<32, EPI_RELU_BF16, false>, cv_smem(32));
  allow((const void*)k_conv<32, EPI_RELU_BF16, true>, cv_smem(32));
  allow((const void*)k_conv<32, EPI_MASK_BF16, false>, cv_smem(32));
  allow((const void*)k_conv<32, EPI_MASK_BF16, true>, cv_smem(32));
  allow((const void*)k_conv<4, EPI_LINEAR_F32, false>, cv_smem(4));
  allow((const void*)k_conv<4, EPI_LINEAR_F32, true>, cv_smem(4));
  allow((const void*)k_conv4<false>, C4_SMEM);
  allow((const void*)k_conv4<true>, C4_SMEM);
  n->sms = std::max(sms, 1);
  n->tiles_x = (W + CT_X - 1) / CT_X;
  n->ntiles = n->tiles_x * ((H + CT_Y - 1) / CT_Y);
  n->ctiles_x = (W + CV_X - 1) / CV_X;
  n->cntiles = n->ctiles_x * ((H + CV_Y - 1) / CV_Y);
  n->wblocks = std::min(n->ntiles, WG_CTAS_PER_SM * n->sms);
  // All buffers are parts of one allocation, zeroed at once: creating and destroying a
  // 512 x 512 network takes 0.33 ms; 1.1 with one allocation each, most of it in the allocator.
  std::vector<std::pair<void**, size_t>> parts;
  auto A = [&](void** p, size_t bytes) { parts.push_back({p, (bytes + 255) / 256 * 256}); };
  A((void**)&n->w, sizeof(float) * LBM_CNN_NPARAMS);
  A((void**)&n->m, sizeof(float) * LBM_CNN_NPARAMS);
  A((void**)&n->v, sizeof(float) * LBM_CNN_NPARAMS);
  A((void**)&n->grad, sizeof(float) * LBM_CNN_NPARAMS);
  for (int l = 0; l < NL; ++l) {
    if (l == 0) continue;  // the first layer takes the FP32 features and weights
    A((void**)&n->wt[l], 2 * (size_t)ru(cout_of(l), 8) * kp_of(l));
    A((void**)&n->wb[l], 2 * (size_t)ru(cin_of(l), 8) * kb_of(l));
    A((void**)&n->act[l], 2 * P * CH[l]);
    A((void**)&n->pos[l], 4 * P);
  }
  A((void**)&n->dz[0], 2 * P * 32);
  A((void**)&n->dz[1], 2 * P * 32);
  A((void**)&n->dz5, 2 * P * 8);
  A((void**)&n->xs, 2 * P * 16);
  A((void**)&n->logs, sizeof(LogEntry) * LOG_N);
  A((void**)&n->xf, 4 * P * 4);
  A((void**)&n->tf, 4 * P * 4);
  A((void**)&n->z, 4 * P * 4);
  A((void**)&n->wpartial, sizeof(float) * (size_t)n->wblocks * LBM_CNN_NPARAMS);
  A((void**)&n->dpart, sizeof(double) * 2 * ((4 * P + 255) / 256 + 1));
  A((void**)&n->res, sizeof(Results));
  A((void**)&n->exps, sizeof(ExpEntry) * EXP_N);
  size_t total = 0;
  for (auto& p : parts) total += p.second;
  if (e == cudaSuccess) e = cudaMalloc((void**)&n->slab, total);
  if (e == cudaSuccess) e = cudaMemsetAsync(n->slab, 0, total, n->stream);
  if (e == cudaSuccess) {
    unsigned char* at = n->slab;
    for (auto& p : parts) {
      *p.first = at;
      at += p.second;
    }
  }
  if (e == cudaSuccess) e = pinned_results().get(&n->h_res);
  const std::vector<LogEntry> logs = log_table();
  const std::vector<ExpEntry> exps = exp_table();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(n->logs, logs.data(), sizeof(LogEntry) * LOG_N, cudaMemcpyHostToDevice, n->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(n->exps, exps.data(), sizeof(ExpEntry) * EXP_N, cudaMemcpyHostToDevice, n->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
  if (e != cudaSuccess) {
    g_cnn_error = std::string("lbm_cnn_create: ") + cudaGetErrorString(e);
    lbm_cnn_destroy(n);
    return e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;
  }
  int rc = LBM_OK;
  auto map = [&](const void* p, int ncg, int box_cg, int px, int rows, CUtensorMap* out) {
    if (rc == LBM_OK) rc = encode_image(n, p, ncg, box_cg, px, rows, out);
  };
  for (int l = 1; l < NL; ++l) {
    map(n->act[l], 4, 4, CV_HX, CV_HY, &n->c_act[l]);
    map(n->act[l], 4, 4, CT_HX, CT_HY, &n->m_act[l]);
  }
  for (int k = 0; k < 2; ++k) {
    map(n->dz[k], 4, 4, CV_HX, CV_HY, &n->c_dz[k]);
    map(n->dz[k], 4, 4, CT_X, CT_Y, &n->g_dz[k]);
  }
  map(n->dz5, 1, 1, CT_HX, CT_HY, &n->m_dz5);
  map(n->dz5, 1, 2, CT_X, CT_Y, &n->g_dz5);
  map(n->xs, 2, 2, CT_HX, CT_HY, &n->m_xs);
  if (rc != LBM_OK || pack_all(n) != LBM_OK) {
    g_cnn_error = n->err;
    lbm_cnn_destroy(n);
    return LBM_ERR_CUDA;
  }
  *out = n;
  return LBM_OK;
}

int lbm_cnn_destroy(lbm_cnn* n) {
  if (!n) return LBM_OK;
  if (n->stream) cudaStreamSynchronize(n->stream);
  if (n->slab) cudaFree(n->slab);
  if (n->h_res) pinned_results().put(n->h_res);
  if (n->own_stream && n->stream) cudaStreamDestroy(n->stream);
  delete n;
  return LBM_OK;
}

int lbm_cnn_set_params(lbm_cnn* n, const float* params, int on_device) {
  if (!n || !params) return cfail(n, LBM_ERR_INVALID, "NULL argument");
  CCK(n, cudaMemcpyAsync(n->w, params, sizeof(float) * LBM_CNN_NPARAMS,
                         on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, n->stream));
  CCK(n, cudaMemsetAsync(n->m, 0, sizeof(float) * LBM_CNN_NPARAMS, n->stream));
  CCK(n, cudaMemsetAsync(n->v, 0, sizeof(float) * LBM_CNN_NPARAMS, n->stream));
  n->step = 0;
  int rc = pack_all(n);
  if (rc == LBM_OK) rc = clear_timeout(n);
  if (rc != LBM_OK) return rc;
  if (!on_device) CCK(n, cudaStreamSynchronize(n->stream));
  return LBM_OK;
}

int lbm_cnn_get_params(lbm_cnn* n, float* params, int on_device) {
  if (!n || !params) return cfail(n, LBM_ERR_INVALID, "NULL argument");
  CCK(n, cudaMemcpyAsync(params, n->w, sizeof(float) * LBM_CNN_NPARAMS,
                         on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, n->stream));
  if (!on_device) CCK(n, cudaStreamSynchronize(n->stream));
  return LBM_OK;
}

int lbm_cnn_set_adam(lbm_cnn* n, double lr, double beta1, double beta2, double eps) {
  if (!n || !(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0))
    return cfail(n, LBM_ERR_INVALID, "bad Adam hyper-parameters");
  n->lr = (float)lr; n->b1 = (float)beta1; n->b2 = (float)beta2; n->eps = (float)eps;
  return LBM_OK;
}

int lbm_cnn_loss_grad(lbm_cnn* n, const double* coarse, const double* target, double* loss,
                      float* grads) {
  if (!n || !coarse || !target) return cfail(n, LBM_ERR_INVALID, "NULL argument");
  nvtxRangePushA("lbm_cnn_train_step");
  struct Pop { ~Pop() { nvtxRangePop(); } } pop;
  int rc = forward(n, coarse, true);
  if (rc == LBM_OK) rc = loss_backward(n, target, false);
  if (rc != LBM_OK) return rc;
  if (grads)
    CCK(n, cudaMemcpyAsync(grads, n->grad, sizeof(float) * LBM_CNN_NPARAMS, cudaMemcpyDeviceToHost,
                           n->stream));
  if ((rc = fetch_results(n)) != LBM_OK) return rc;
  if (loss) *loss = n->h_res->loss;
  return LBM_OK;
}

int lbm_cnn_train_step(lbm_cnn* n, const double* coarse, const double* target, double* loss) {
  if (!n || !coarse || !target) return cfail(n, LBM_ERR_INVALID, "NULL argument");
  int rc = forward(n, coarse, true);
  if (rc != LBM_OK) return rc;
  n->step += 1;
  rc = loss_backward(n, target, true);
  if (rc != LBM_OK) return rc;
  if (loss) {
    if ((rc = fetch_results(n)) != LBM_OK) return rc;
    *loss = n->h_res->loss;
  }
  return LBM_OK;
}

int lbm_cnn_debug_give_up(lbm_cnn* n, int which) {
  if (!n || which < 0 || which > (GIVE_UP_COPIES | GIVE_UP_PRODUCTS))
    return cfail(n, LBM_ERR_INVALID, "lbm_cnn_debug_give_up: which must be 0 .. 3");
  n->give_up = which;
  return LBM_OK;
}

int lbm_cnn_set_output_scale(lbm_cnn* n, const double* scale) {
  if (!n || !scale) return cfail(n, LBM_ERR_INVALID, "NULL argument");
  for (int c = 0; c < 4; ++c)
    if (!(std::isfinite(scale[c]) && scale[c] > 0.0))
      return cfail(n, LBM_ERR_INVALID, "output scales must be finite and > 0");
  for (int c = 0; c < 4; ++c) n->scale.s[c] = (float)scale[c];
  return LBM_OK;
}

int lbm_cnn_set_loss(lbm_cnn* n, int kind) {
  if (!n) return cfail(nullptr, LBM_ERR_INVALID, "NULL argument");
  if (kind != LBM_CNN_LOSS_MSE && kind != LBM_CNN_LOSS_L1)
    return cfail(n, LBM_ERR_INVALID, "unknown loss kind");
  n->loss_kind = kind;
  return LBM_OK;
}

int lbm_cnn_residual_rms(lbm_cnn* n, const double* coarse, const double* target, double* rms) {
  if (!n || !coarse || !target || !rms) return cfail(n, LBM_ERR_INVALID, "NULL argument");
  const int nb = (n->npix + 255) / 256;
  k_features<<<nb, 256, 0, n->stream>>>(coarse, n->npix, n->W, n->xf, nullptr, n->logs);
  k_features<<<nb, 256, 0, n->stream>>>(target, n->npix, n->W, n->tf, nullptr, n->logs);
  std::vector<double> part(4 * (size_t)nb);
  k_residual_sq<<<nb, 256, 0, n->stream>>>(n->xf, n->tf, n->npix, n->dpart);
  CCK(n, cudaGetLastError());
  CCK(n, cudaMemcpyAsync(part.data(), n->dpart, sizeof(double) * part.size(), cudaMemcpyDeviceToHost, n->stream));
  CCK(n, cudaStreamSynchronize(n->stream));
  for (int c = 0; c < 4; ++c) {
    double s = 0.0;
    for (int b = 0; b < nb; ++b) s += part[4 * b + c];
    rms[c] = std::sqrt(s / n->npix);
  }
  return LBM_OK;
}

int lbm_cnn_correct(lbm_cnn* n, const double* coarse, double* corrected, double mass_tol,
                    int* used_fallback) {
  if (!n || !coarse || !corrected) return cfail(n, LBM_ERR_INVALID, "NULL argument");
  int rc = forward(n, coarse, false);
  if (rc != LBM_OK) return rc;
  const int nb = (n->npix + 255) / 256;
  CCK(n, gbtma::launch_overlapped(k_apply, nb, 256, 0, n->stream, (const float4*)n->xf, (const float4*)n->z,
                                  n->npix, corrected, coarse, n->dpart, n->scale, n->exps, n->res));
  if ((rc = fetch_results(n)) != LBM_OK) return rc;
  const double m1 = n->h_res->mass[0], m0 = n->h_res->mass[1];
  const bool fallback = !std::isfinite(m1) || std::fabs(m1 - m0) > mass_tol * std::fabs(m0);
  if (fallback) {
    CCK(n, cudaMemcpyAsync(corrected, coarse, sizeof(double) * 4 * n->npix,
                           cudaMemcpyDeviceToDevice, n->stream));
    CCK(n, cudaStreamSynchronize(n->stream));
  }
  if (used_fallback) *used_fallback = fallback ? 1 : 0;
  return LBM_OK;
}

int lbm_restrict(const double* fine, int Hf, int Wf, int r, double* coarse, void* cuda_stream) {
  if (!fine || !coarse || r < 1 || Hf < r || Wf < r || Hf % r || Wf % r)
    return cfail(nullptr, LBM_ERR_INVALID, "lbm_restrict: bad sizes");
  const int nc = (Hf / r) * (Wf / r);
  k_restrict<<<(nc + 255) / 256, 256, 0, (cudaStream_t)cuda_stream>>>(fine, Hf, Wf, r, coarse);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cfail(nullptr, LBM_ERR_CUDA, cudaGetErrorString(e));
  return LBM_OK;
}

const char* lbm_cnn_last_error(lbm_cnn* n) { return n ? n->err.c_str() : g_cnn_error.c_str(); }

}  // extern "C"

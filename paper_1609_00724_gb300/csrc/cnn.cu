// Learned refinement proposal: a 3-layer CNN over coarse (FLEDGE, log10 Q)
// tiles that marks coarse cells where FLL-jump refinement will be needed.
// conv3x3 2->32 + ReLU, conv3x3 32->32 + ReLU, conv3x3 32->1 (logit); loss:
// binary cross-entropy with a positive-class weight. Weights are BF16 for the
// forward and backward passes (FP32 master copy, Adam in FP32); every
// contraction accumulates in FP32. Activations are NCHW float32.
//
// The convolutions run on the tensor cores (tcgen05) as implicit GEMMs over
// the pixels of a tile. The activations and gradients stay FP32 values: each
// is split into three BF16 pieces that sum to it exactly (8 bits each), the
// pieces' products with the BF16 weights (or with the other operand's pieces)
// are exact, and the sums are FP32. One block's tile goes through all layers
// in shared and tensor memory, so a forward pass reads its input and writes
// its output once.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <cstring>
#include <vector>

#include "qsl_internal.cuh"
#include "umma.cuh"

namespace {

constexpr int C1 = 2, C2 = 32; // input and hidden channels
constexpr int NW1 = 32 * 2 * 9, NB1 = 32, NW2 = 32 * 32 * 9, NB2 = 32, NW3 = 32 * 9, NB3 = 1;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NW1, OFF_W2 = OFF_B1 + NB1, OFF_B2 = OFF_W2 + NW2, OFF_W3 = OFF_B2 + NB2,
              OFF_B3 = OFF_W3 + NW3, NPAR = OFF_B3 + NB3;

// ---------------------------------------------------------------- tiles
// Data-gradient tiles: rows of 32 pixels (one warp each), the MMA's 128 rows
// are four of them. Flattened indices are row * 32 + column; a tap (ky, kx) of
// the pixel m is the pixel m + 32 ky + kx of the layer above, so the last two
// columns of a row see the next row's first ones and are not used.
constexpr int PW = 32;
constexpr int R2 = 12, R1 = R2 + 2;         // rows of the 32-channel layers: outputs, inputs
constexpr int M2 = R2 * PW;                 // output pixels: three MMA tiles
constexpr int NP = R1 * PW + 8;             // input pixels (the last taps read two past the rows)
constexpr int DW = PW - 2, DH = R2;         // valid columns, rows
constexpr int TILE_THREADS = 32 * R2;
constexpr uint32_t CHUNK = NP * 16;         // bytes of one chunk plane
constexpr uint32_t WTAP = 32 * 64;          // one tap's 32 x 32 weights

struct alignas(16) TileSmem {
  unsigned char a[12 * CHUNK];              // [piece][chunk] planes of the layer above's gradient
  unsigned char w2[9 * WTAP];               // [tap][chunk][out channel][8]
  float w3[9 * 32];                         // [tap][channel]
  uint32_t tmem;
  int failed;
  uint64_t bar[3], drained;
};
static_assert(sizeof(TileSmem) <= 113 * 1024, "two blocks per SM");

// Layer 2's weights are kept twice more in the layouts of the MMA's operand
// (K = chunk and element): forward [kx][chunk][ky][output channel][8] over the
// input channels, data gradient [tap][chunk][input channel][8] over the output
// channels with the taps reversed. They are written wherever the BF16 weights
// are.
// Layer 1's are kept as [rotation][MMA][tap of two][output channel][8] (see
// forward_kernel): element 3 c + 0, 1, 2 the weight of input channel c for each
// piece, element 6 a piece of the bias.
constexpr int NOP1 = 3 * 5 * 512;
constexpr int OFF_OP = (NPAR + 7) / 8 * 8, OFF_OP1 = OFF_OP + 2 * NW2, NWB = OFF_OP1 + NOP1;
__device__ __forceinline__ void store_weight(__nv_bfloat16* wb, int i, float v) {
  const __nv_bfloat16 b = __float2bfloat16_rn(v);
  wb[i] = b;
  if (i >= OFF_W2 && i < OFF_W2 + NW2) {
    const int j = i - OFF_W2, co = j / (32 * 9), ci = (j / 9) % 32, k = j % 9;
    wb[OFF_OP + (((k % 3) * 4 + ci / 8) * 96 + (k / 3) * 32 + co) * 8 + ci % 8] = b;
    wb[OFF_OP + NW2 + (((8 - k) * 4 + co / 8) * 32 + ci) * 8 + co % 8] = b;
  } else if (i < NW1) {
    // input slots 0 and 1 at kx: MMA kx; slot 2 at kx = 0, 1: MMA 3; at kx = 2: MMA 4
    const int co = i / 18, c = (i / 9) % 2, ky = (i / 3) % 3, kx = i % 3;
    for (int rot = 0; rot < 3; ++rot) {
      const int slot = (rot + ky) % 3, p = slot < 2 ? kx : 3 + kx / 2, half = slot < 2 ? slot : kx % 2;
      for (int e = 0; e < 3; ++e) wb[OFF_OP1 + rot * 2560 + p * 512 + half * 256 + co * 8 + 3 * c + e] = b;
    }
  } else if (i >= OFF_B1 && i < OFF_B1 + NB1) {
    // the bias, exactly, in three pieces against the ones of slot 0
    uint32_t pc[3];
    umma::split2(v, 0.0f, pc, pc + 1, pc + 2);
    for (int rot = 0; rot < 3; ++rot)
      for (int p = 0; p < 3; ++p)
        wb[OFF_OP1 + rot * 2560 + p * 512 + (i - OFF_B1) * 8 + 6] = __ushort_as_bfloat16((unsigned short)pc[p]);
  }
}

__device__ __forceinline__ void load_w2(unsigned char* w2, const __nv_bfloat16* __restrict__ op, int tid) {
#pragma unroll
  for (int i = tid; i < NW2 / 8; i += TILE_THREADS)
    reinterpret_cast<uint4*>(w2)[i] = __ldg(reinterpret_cast<const uint4*>(op) + i);
}

// The 32 x 32 convolution of the planes in `a` for MMA tile t (128 pixels):
// 9 taps x 3 pieces x 2 K steps into four accumulators of 32 columns. The
// tensor core cuts each sum's low bits, so the leading pieces have one
// accumulator per row of taps (six sums each; the rows are then added in
// FP32) and the middle and last pieces, 2^-8 and 2^-16 of them, the fourth.
// Tile 2 takes tile 0's columns (conv32_read hands them over). One thread.
__device__ __forceinline__ void conv32_issue(TileSmem& S, uint32_t tmem, int t) {
  const uint64_t a0 = umma::desc_k(umma::smem_addr(S.a) + t * 2048, CHUNK), w0 = umma::desc_k(umma::smem_addr(S.w2), 512);
  const uint32_t d0 = tmem + (t & 1) * 128;
  constexpr uint32_t id = umma::idesc(128, 32, false);
#pragma unroll
  for (int piece = 2; piece >= 0; --piece)
#pragma unroll
    for (int tap = 0; tap < 9; ++tap)
#pragma unroll
      for (int k = 0; k < 2; ++k)
        umma::mma(d0 + (piece ? 96 : 32 * (tap / 3)),
                  a0 + ((piece * 4 + 2 * k) * CHUNK / 16 + (tap / 3) * PW + tap % 3), w0 + (tap * WTAP + k * 1024) / 16,
                  id, piece == 0 ? tap % 3 > 0 || k > 0 : piece == 1 || tap > 0 || k > 0);
  umma::commit(&S.bar[t]);
}

// Waits for the MMA tile of the warp's row (warp / 4) and reads its sums; the
// first four warps then let tile 2 be issued into the columns they have read.
__device__ __forceinline__ bool conv32_read(TileSmem& S, uint32_t tmem, int warp, uint32_t phase, uint32_t wait_ns, float* v) {
  const int t = warp >> 2;
  const uint32_t tq = tmem + ((uint32_t)(warp & 3) << 21) + (t & 1) * 128;
  const bool ok = umma::bar_wait(&S.bar[t], phase, wait_ns);
  umma::fence_after();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float u[16];
    umma::tmem_ld16(tq + 96 + 16 * h, v + 16 * h);
#pragma unroll
    for (int row = 0; row < 3; ++row) {
      umma::tmem_ld16(tq + 32 * row + 16 * h, u);
#pragma unroll
      for (int c = 0; c < 16; ++c) v[16 * h + c] += u[c];
    }
  }
  if (t == 0) {
    umma::fence_before();
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (warp == 0 && ok && umma::elect()) {
      umma::fence_after();
      conv32_issue(S, tmem, 2);
    }
    __syncwarp();
  }
  return ok;
}

// Writes a pixel's 16 channels (half h of the 32) as pieces into the planes.
template <uint32_t PLANE>
__device__ __forceinline__ void store_half(unsigned char* a, int m, int h, const float* v) {
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    uint4 p[3];
    umma::split8(v + 8 * c, p);
#pragma unroll
    for (int piece = 0; piece < 3; ++piece)
      *reinterpret_cast<uint4*>(a + (piece * 4 + 2 * h + c) * PLANE + m * 16) = p[piece];
  }
}

__device__ __forceinline__ void zero_tail(unsigned char* a, int tid) {
  if (tid < 12 * (NP - R1 * PW))
    *reinterpret_cast<uint4*>(a + (tid / (NP - R1 * PW)) * CHUNK + (R1 * PW + tid % (NP - R1 * PW)) * 16) =
        make_uint4(0, 0, 0, 0);
}

__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<unsigned long long&>(d))
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)),
        "l"(reinterpret_cast<unsigned long long&>(c)));
  return d;
}

struct TileGrid {
  int n, H, W, tx, ty;  // images, tiles along x and y
  int64_t tiles;
  uint32_t wait_ns;     // limit of a wait
};
__device__ __forceinline__ void tile_of(const TileGrid& G, int64_t t, int w, int h, int* n, int* oy, int* ox) {
  *ox = (int)(t % G.tx) * w;
  t /= G.tx;
  *oy = (int)(t % G.ty) * h;
  *n = (int)(t / G.ty);
}

// ---------------------------------------------------------------- forward pass
// All three layers, row by row: a block marches down the rows of a task, 128
// pixels (the MMA's rows) at a time: one segment of 128 columns, or 2 or 4
// segments of 64 or 32 that march through different tasks of the same height.
// A layer's last two columns of a segment see the next one, so a segment of P
// columns yields P - 6.
//  1. The network input as one 16-byte chunk of pieces per pixel (x0 hi, mid,
//     lo, x1 hi, mid, lo, 1, 0; the one for the bias); the last three rows in
//     three slots. A K = 16
//     step takes two taps; the slot of a row rotates, and the weights with it
//     (three copies); the ninth tap is paired with zeros.
//  2. TMEM -> ReLU (0 outside the image) -> pieces in shared memory. The
//     N = 96 columns of an MMA are the three output rows that this row feeds
//     (tap rows 0, 1, 2): the read of the 128 x 16 operand, 59 cycles for N =
//     32 and 67 for N = 96, sets the pace. 18 MMAs per row against 54.
//  3. A pixel stays in its TMEM lane, so its thread adds the row sums of three
//     successive rows in registers: bias, ReLU, the products with layer 3's
//     nine taps, which are summed over the rows in registers and over the
//     columns through shared memory.
// Warps 0-3 make layer 1's output, warps 4-7 read layer 2's, warp 8 issues the
// MMAs. The tensor core cuts the low bits of its sums: a sum is six K steps of
// leading pieces after the middle and last ones, the rest is FP32 addition.
// Bound: shared memory, about 2,100 of the 2,350 cycles per row and SM (the
// MMAs' operands half of it, layer 3's weights a quarter). 64 slices of 256 x
// 256: 0.42 ms. Tiles of 32 x 12 pixels with N = 32 took 0.69 ms (54 MMAs of 59
// cycles per 128 pixels), FP32 kernels, one per layer, 5.6 ms. Eight warps on
// layer 2's side instead of four: 0.58 against 0.51 ms at that stage (spills).
constexpr int SP = 128, SPAD = SP + 8;      // pixels of a row step; the taps read two past them
constexpr uint32_t ROW = SPAD * 16;         // bytes of a chunk plane
constexpr uint32_t W2KX = 4 * 96 * 16;      // bytes of one kx of layer 2's weights
constexpr int FWD_THREADS = 288;

struct alignas(16) FwdSmem {
  unsigned char a[2][12 * ROW];             // layer 1's row: [piece][chunk] planes, two rows
  unsigned char x[3][ROW];                  // the network input's rows, slot = row mod 3
  unsigned char zero[SP * 16];
  unsigned char w2[3 * W2KX];
  unsigned char w1[3 * 5 * 1024];           // [rotation][MMA][tap of two][output channel][8]
  float w3[9 * 32];                         // [tap][channel]
  alignas(16) float b2[32];
  float b3;
  float z[2][3][SPAD];                      // layer 3's sums over the rows, per tap column
  uint32_t tmem;
  // layer 1's sums ready [2], input row written, planes written [2], layer 2's sums ready [2] and read [2]
  uint64_t l1[2], xw, aw[2], l2[2], rd[2], drained;
};
static_assert(sizeof(FwdSmem) <= 113 * 1024, "two blocks per SM");

struct FwdGrid {
  int H, W, P, nseg, zw, h, tx, ty;  // segment columns, segments per row step, output columns and rows of a task, tasks along x, y
  int64_t tasks, groups;             // groups of nseg tasks
  uint32_t wait_ns;                  // limit of a wait
};

__global__ void __launch_bounds__(FWD_THREADS, 2)
    forward_kernel(const float* __restrict__ x, const __nv_bfloat16* __restrict__ wb, const float* __restrict__ w,
                   float* __restrict__ out, const FwdGrid G) {
  extern __shared__ __align__(16) unsigned char smem[];
  FwdSmem& S = *reinterpret_cast<FwdSmem*>(smem);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const size_t plane = (size_t)G.H * G.W;
  for (int i = tid; i < NW2 / 8; i += FWD_THREADS)
    reinterpret_cast<uint4*>(S.w2)[i] = __ldg(reinterpret_cast<const uint4*>(wb + OFF_OP) + i);
  for (int i = tid; i < NOP1 / 8; i += FWD_THREADS)
    reinterpret_cast<uint4*>(S.w1)[i] = __ldg(reinterpret_cast<const uint4*>(wb + OFF_OP1) + i);
  for (int i = tid; i < 288; i += FWD_THREADS) S.w3[(i % 9) * 32 + i / 9] = __bfloat162float(wb[OFF_W3 + i]);
  if (tid < 32) S.b2[tid] = w[OFF_B2 + tid];
  // what no row writes: the planes' and input rows' tails, the zero rows
  if (tid < 27 * 8)
    *reinterpret_cast<uint4*>((tid < 24 * 8 ? S.a[0] + (tid / 8) * ROW : S.x[0] + (tid / 8 - 24) * ROW) +
                              (SP + tid % 8) * 16) = make_uint4(0, 0, 0, 0);
  if (tid < SP) *reinterpret_cast<uint4*>(S.zero + tid * 16) = make_uint4(0, 0, 0, 0);
  if (tid == 0) {
    S.b3 = w[OFF_B3];
    for (int i = 0; i < 2; ++i) {
      umma::bar_init(&S.l1[i]);
      umma::bar_init(&S.l2[i]);
      umma::bar_init(&S.aw[i], 4);
      umma::bar_init(&S.rd[i], 4);
    }
    umma::bar_init(&S.xw, 4);
    umma::bar_init(&S.drained);
    umma::bar_init_fence();
  }
  if (warp == 0) umma::tmem_alloc(&S.tmem, 256);
  umma::fence_smem();
  umma::fence_before();
  __syncthreads();
  umma::fence_after();
  const uint32_t tmem = S.tmem;  // layer 1: 2 x 32 columns; layer 2: 2 x 96 from column 64
  const uint32_t tq = tmem + ((uint32_t)(warp & 3) << 21);
  const int rows = G.h + 4;      // layer 1 rows of a task; its network input rows: two more
  uint32_t g = 0;                // rows done: buffer g & 1, its use g >> 1
  bool ok = true;                // false once a wait has run out: nothing more is waited for or signalled

  // of the block's 288 x 96 registers: 128 x 72, 128 x 120, 32 x 96
  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    const int p = tid, sg = p / G.P, lc = p - sg * G.P;
    for (int64_t grp = blockIdx.x; grp < G.groups; grp += gridDim.x) {
      int64_t t = grp * G.nseg + sg;
      const bool live = t < G.tasks && sg < G.nseg;
      const int ox = (int)(t % G.tx) * G.zw;
      t /= G.tx;
      const int y0 = (int)(t % G.ty) * G.h;
      const size_t n = (size_t)(t / G.ty);
      const int xc = ox - 3 + lc;
      const bool xin = live && xc >= 0 && xc < G.W;
      const float* xp = x + 2 * n * plane + xc;
      float x0 = 0.0f, x1 = 0.0f;
      auto fetch = [&](int r) {
        const int gy = y0 - 3 + r;
        const bool in = xin && gy >= 0 && gy < G.H;
        x0 = in ? __ldg(xp + (size_t)gy * G.W) : 0.0f;
        x1 = in ? __ldg(xp + plane + (size_t)gy * G.W) : 0.0f;
      };
      // writes the fetched row into its slot and fetches another
      auto put = [&](int r, int next) {
        uint32_t h0, m0, l0;
        umma::split2(x0, x1, &h0, &m0, &l0);  // low halves: channel 0, high halves: channel 1
        *reinterpret_cast<uint4*>(S.x[r % 3] + p * 16) = make_uint4(
            __byte_perm(h0, m0, 0x5410), __byte_perm(l0, h0, 0x7610), __byte_perm(m0, l0, 0x7632), 0x3f80u);
        fetch(next);
      };
      fetch(0);
      put(0, 1);
      put(1, 2);
      put(2, 3);
      umma::fence_smem();
      __syncwarp();
      if (lane == 0 && ok) umma::bar_arrive(&S.xw);
#pragma unroll 1
      for (int r = 0; r < rows; ++r, ++g) {
        const int b = g & 1;
        ok = ok && umma::bar_wait(&S.l1[b], g >> 1 & 1, G.wait_ns);
        umma::fence_after();
        if (r + 1 < rows) {  // the slot of row r is free
          put(r + 3, r + 4);
          umma::fence_smem();
          __syncwarp();
          if (lane == 0 && ok) umma::bar_arrive(&S.xw);
        }
        const int gy = y0 - 2 + r, gx = xc + 1;
        const bool in = live && gy >= 0 && gy < G.H && gx >= 0 && gx < G.W;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float v[16];
          umma::tmem_ld16(tq + b * 32 + 16 * h, v);
#pragma unroll
          for (int c = 0; c < 16; ++c) v[c] = in ? fmaxf(v[c], 0.0f) : 0.0f;
          // the planes are free once the MMAs of two rows ago are done
          if (h == 0 && g >= 2) ok = ok && umma::bar_wait(&S.l2[b], (g >> 1) - 1 & 1, G.wait_ns);
          store_half<ROW>(S.a[b], p, h, v);
        }
        umma::fence_smem();
        umma::fence_before();
        __syncwarp();
        if (lane == 0 && ok) umma::bar_arrive(&S.aw[b]);
      }
    }
  } else if (warp < 8) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 120;");
    const int p = tid - SP, sg = p / G.P, lc = p - sg * G.P;
    for (int64_t grp = blockIdx.x; grp < G.groups; grp += gridDim.x) {
      int64_t t = grp * G.nseg + sg;
      const bool live = t < G.tasks && sg < G.nseg;
      const int ox = (int)(t % G.tx) * G.zw;
      t /= G.tx;
      const int y0 = (int)(t % G.ty) * G.h;
      const size_t n = (size_t)(t / G.ty);
      float A[32], B[32];        // tap rows 0 + 1 of the row before, tap row 0 of this one
      float za[3], zb[3];        // layer 3: rows of taps 0 + 1, 0
#pragma unroll
      for (int c = 0; c < 32; ++c) A[c] = B[c] = 0.0f;
#pragma unroll
      for (int k = 0; k < 3; ++k) za[k] = zb[k] = 0.0f;
#pragma unroll 1
      for (int r = 0; r < rows; ++r, ++g) {
        const int b = g & 1;
        ok = ok && umma::bar_wait(&S.l2[b], g >> 1 & 1, G.wait_ns);
        umma::fence_after();
        // layer 2's row that this row completes
        const int gy = y0 - 3 + r, gx = ox - 1 + lc;
        const bool in = live && r >= 2 && gy >= 0 && gy < G.H && gx >= 0 && gx < G.W;
        float2 dot[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) dot[k] = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int c0 = 8 * q;
          float v[8], u[8];
          umma::tmem_ld8(tq + 64 + b * 96 + 64 + c0, v);
          const float4 e0 = *reinterpret_cast<const float4*>(&S.b2[c0]), e1 = *reinterpret_cast<const float4*>(&S.b2[c0 + 4]);
          const float bias[8] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w};
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            v[c] = in ? fmaxf(A[c0 + c] + v[c] + bias[c], 0.0f) : 0.0f;
          }
          umma::tmem_ld8(tq + 64 + b * 96 + 32 + c0, u);
#pragma unroll
          for (int c = 0; c < 8; ++c) A[c0 + c] = B[c0 + c] + u[c];
          umma::tmem_ld8(tq + 64 + b * 96 + c0, B + c0);
#pragma unroll
          for (int k = 0; k < 9; ++k)
#pragma unroll
            for (int c = 0; c < 8; c += 4) {
              const float4 f = *reinterpret_cast<const float4*>(&S.w3[k * 32 + c0 + c]);
              dot[k] = ffma2(make_float2(v[c], v[c + 1]), make_float2(f.x, f.y), dot[k]);
              dot[k] = ffma2(make_float2(v[c + 2], v[c + 3]), make_float2(f.z, f.w), dot[k]);
            }
        }
        umma::fence_before();
        __syncwarp();
        if (lane == 0 && ok) umma::bar_arrive(&S.rd[b]);
        // layer 3's row that this row completes
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          // a wait that ran out leaves the outputs marked as missing, the neighbours' too
          S.z[b][k][p] = ok ? za[k] + (dot[6 + k].x + dot[6 + k].y) : __int_as_float(0x7fc00000);
          za[k] = zb[k] + (dot[3 + k].x + dot[3 + k].y);
          zb[k] = dot[k].x + dot[k].y;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const int zy = y0 + r - 4, zx = ox + lc;
        if (live && r >= 4 && zy < G.H && lc < G.zw && zx < G.W) {
          const float z = S.b3 + ((S.z[b][0][p] + S.z[b][1][p + 1]) + S.z[b][2][p + 2]);
          out[n * plane + (size_t)zy * G.W + zx] = 1.0f / (1.0f + expf(-z));
        }
      }
    }
  } else {
    const uint64_t w2 = umma::desc_k(umma::smem_addr(S.w2), 96 * 16), w1 = umma::desc_k(umma::smem_addr(S.w1), 512);
    const uint32_t x0 = umma::smem_addr(S.x);
    uint32_t xn = 0;
    // layer 1's row r of the task, row number gl of the block
    auto layer1 = [&](int r, uint32_t gl) {
      ok = ok && umma::bar_wait(&S.xw, xn & 1, G.wait_ns);
      ++xn;
      umma::fence_after();
      if (ok && umma::elect()) {
        const uint64_t wr = w1 + (r % 3) * (5 * 64);
        const uint32_t d = tmem + (gl & 1) * 32;
        constexpr uint32_t id = umma::idesc(128, 32, false);
#pragma unroll
        for (int q = 0; q < 3; ++q) umma::mma(d, umma::desc_k(x0 + q * 16, ROW), wr + q * 64, id, q > 0);
        umma::mma(d, umma::desc_k(x0 + 2 * ROW, 16), wr + 3 * 64, id, true);
        umma::mma(d, umma::desc_k(x0 + 2 * ROW + 32, ROW - 32), wr + 4 * 64, id, true);
        umma::commit(&S.l1[gl & 1]);
      }
      __syncwarp();
    };
    for (int64_t grp = blockIdx.x; grp < G.groups; grp += gridDim.x) {
      layer1(0, g);
#pragma unroll 1
      for (int r = 0; r < rows; ++r, ++g) {
        if (r + 1 < rows) layer1(r + 1, g + 1);
        const int b = g & 1;
        ok = ok && umma::bar_wait(&S.aw[b], g >> 1 & 1, G.wait_ns);
        if (g >= 2) ok = ok && umma::bar_wait(&S.rd[b], (g >> 1) - 1 & 1, G.wait_ns);
        umma::fence_after();
        if (ok && umma::elect()) {
          const uint64_t a = umma::desc_k(umma::smem_addr(S.a[b]), ROW);
          constexpr uint32_t id = umma::idesc(128, 96, false);
#pragma unroll
          for (int piece = 2; piece >= 0; --piece)
#pragma unroll
            for (int kx = 0; kx < 3; ++kx)
#pragma unroll
              for (int k = 0; k < 2; ++k)
                umma::mma(tmem + 64 + b * 96, a + ((piece * 4 + 2 * k) * ROW / 16 + kx),
                          w2 + (kx * W2KX + k * 2 * 1536) / 16, id, piece < 2 || kx > 0 || k > 0);
          umma::commit(&S.l2[b]);
        }
        __syncwarp();
      }
    }
    umma::drain(&S.drained);  // another warp may have given up on the last ones
  }
  umma::fence_before();
  __syncthreads();
  if (warp == 0) umma::tmem_free(tmem, 256);
}

// ---------------------------------------------------------------- training forward pass
// One layer in FP32 on the CUDA cores, sums in the order (input channel, tap)
// from the bias on. A gradient depends on the sign of every pre-activation, and
// one that rounds to the other side of zero moves it by up to 1e-5: the
// training pass keeps this order of sums, so its masks stay those it always
// had. A thread has two pixels (rows 8 apart of a 16 x 16 tile) and all output
// channels, in pairs (fma.rn.f32x2 rounds each like fmaf); four weights per
// shared-memory read. Bound: those reads (16 wavefronts per tap for 64 pixels)
// and the multiply-adds alike. 32 x 64 x 64 pixels: a training step of 259 us (9
// more with the weights staged in their stored order, 32 lanes on one bank).
constexpr int T = 16, TH = T + 2, CONV_THREADS = T * T / 2;
template <int CIN, int COUT, bool RELU>
__global__ void __launch_bounds__(CONV_THREADS) conv3x3_kernel(const float* __restrict__ x,
                                                               const __nv_bfloat16* __restrict__ w,
                                                               const float* __restrict__ b, float* __restrict__ y, int H,
                                                               int W, int tx, int ty) {
  extern __shared__ __align__(16) float sm[];
  float* ws = sm;                   // [input channel][tap][output channel]
  float* xs = sm + COUT * CIN * 9;  // [input channel][18][18]
  constexpr int CO2 = (COUT + 1) / 2;
  const int n = blockIdx.x / (tx * ty), t = blockIdx.x % (tx * ty), ox = t % tx * T, oy = t / tx * T;
  const int tid = threadIdx.x;
  const size_t plane = (size_t)H * W;
  const float* xn = x + (size_t)n * CIN * plane;
  for (int i = tid; i < CIN * TH * TH; i += CONV_THREADS) {
    const int c = i / (TH * TH), r = (i / TH) % TH, q = i % TH, gy = oy + r - 1, gx = ox + q - 1;
    xs[i] = (gy >= 0 && gy < H && gx >= 0 && gx < W) ? __ldg(xn + c * plane + (size_t)gy * W + gx) : 0.0f;
  }
#pragma unroll 8
  for (int i = tid; i < COUT * CIN * 9; i += CONV_THREADS)
    ws[i] = __bfloat162float(w[(i % COUT) * (CIN * 9) + i / COUT]);
  __syncthreads();
  const int lx = tid % T, ly = tid / T;
  float2 acc[2][CO2];
#pragma unroll
  for (int c = 0; c < CO2; ++c) acc[0][c] = acc[1][c] = make_float2(b[2 * c], 2 * c + 1 < COUT ? b[2 * c + 1] : 0.0f);
#pragma unroll 1
  for (int ci = 0; ci < CIN; ++ci) {
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const float v0 = xs[(ci * TH + ly + k / 3) * TH + lx + k % 3], v1 = xs[(ci * TH + ly + 8 + k / 3) * TH + lx + k % 3];
      const float* wk = ws + (ci * 9 + k) * COUT;
      if (COUT == 1) {
        acc[0][0].x = fmaf(v0, wk[0], acc[0][0].x);
        acc[1][0].x = fmaf(v1, wk[0], acc[1][0].x);
      } else {
#pragma unroll
        for (int c = 0; c < CO2; c += 2) {
          const float4 f = *reinterpret_cast<const float4*>(wk + 2 * c);
          acc[0][c] = ffma2(make_float2(v0, v0), make_float2(f.x, f.y), acc[0][c]);
          acc[1][c] = ffma2(make_float2(v1, v1), make_float2(f.x, f.y), acc[1][c]);
          acc[0][c + 1] = ffma2(make_float2(v0, v0), make_float2(f.z, f.w), acc[0][c + 1]);
          acc[1][c + 1] = ffma2(make_float2(v1, v1), make_float2(f.z, f.w), acc[1][c + 1]);
        }
      }
    }
  }
  const int gx = ox + lx;
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const int gy = oy + ly + 8 * p;
    if (gx < W && gy < H) {
      float* yn = y + (size_t)n * COUT * plane + (size_t)gy * W + gx;
#pragma unroll
      for (int c = 0; c < COUT; ++c) {
        const float v = c & 1 ? acc[p][c / 2].y : acc[p][c / 2].x;
        yn[c * plane] = RELU ? fmaxf(v, 0.0f) : v;
      }
    }
  }
}

// Data gradients of a 30 x 12 tile: d2 = layer 3's transposed convolution of
// dz times (a2 > 0), written once and as pieces into the planes; d1 = layer
// 2's transposed convolution of d2 times (a1 > 0) by conv32_issue. Bound: the
// MMAs (59 cycles each, set by the read of A, 162 per tile) and the reads of a1
// and a2; 32 x 64 x 64 pixels: 41 us.
__global__ void __launch_bounds__(TILE_THREADS, 2)
    dgrad_kernel(const float* __restrict__ dz, const __nv_bfloat16* __restrict__ wb, const float* __restrict__ a1,
                 const float* __restrict__ a2, float* __restrict__ d1, float* __restrict__ d2, float* __restrict__ grad,
                 const TileGrid G) {
  extern __shared__ __align__(16) unsigned char smem[];
  TileSmem& S = *reinterpret_cast<TileSmem*>(smem);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const size_t plane = (size_t)G.H * G.W;
  load_w2(S.w2, wb + OFF_OP + NW2, tid);
  for (int i = tid; i < 288; i += TILE_THREADS) S.w3[(i % 9) * 32 + i / 9] = __bfloat162float(wb[OFF_W3 + i]);
  if (tid == 0) {
    S.failed = 0;
    for (int i = 0; i < 3; ++i) umma::bar_init(&S.bar[i]);
    umma::bar_init(&S.drained);
    umma::bar_init_fence();
  }
  if (warp == 0) umma::tmem_alloc(&S.tmem, 256);
  umma::fence_before();
  __syncthreads();
  umma::fence_after();
  const uint32_t tmem = S.tmem;
  uint32_t phase = 0;
  for (int64_t tile = blockIdx.x; tile < G.tiles; tile += gridDim.x, phase ^= 1) {
    int n, oy, ox;
    tile_of(G, tile, DW, DH, &n, &oy, &ox);
#pragma unroll 1
    for (int r = warp; r < R1; r += R2) {
      const int gy = oy - 1 + r, gx = ox - 1 + lane;
      const bool in = gy >= 0 && gy < G.H && gx >= 0 && gx < G.W;
      const bool own = in && r >= 1 && r < 1 + DH && lane >= 1 && lane < 1 + DW;
      float g[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) {  // dz at the outputs this pixel feeds through tap k
        const int yy = gy + 1 - k / 3, xx = gx + 1 - k % 3;
        g[k] = in && yy >= 0 && yy < G.H && xx >= 0 && xx < G.W ? __ldg(dz + (size_t)n * plane + (size_t)yy * G.W + xx)
                                                                : 0.0f;
      }
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        float v[16];
        const size_t o = ((size_t)n * 32 + 16 * h) * plane + (size_t)gy * G.W + gx;
#pragma unroll
        for (int c = 0; c < 16; ++c) v[c] = in ? __ldg(a2 + o + c * plane) : 0.0f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
          for (int k = 0; k < 9; ++k)
            s = ffma2(make_float2(g[k], g[k]), *reinterpret_cast<const float2*>(&S.w3[k * 32 + 16 * h + 2 * c]), s);
          v[2 * c] = v[2 * c] > 0.0f ? s.x : 0.0f;
          v[2 * c + 1] = v[2 * c + 1] > 0.0f ? s.y : 0.0f;
        }
        if (own)
#pragma unroll
          for (int c = 0; c < 16; ++c) d2[o + c * plane] = v[c];
        store_half<CHUNK>(S.a, r * PW + lane, h, v);
      }
    }
    zero_tail(S.a, tid);
    umma::fence_smem();
    umma::fence_before();
    __syncthreads();
    if (warp == 0 && umma::elect()) {
      umma::fence_after();
      conv32_issue(S, tmem, 0);
      conv32_issue(S, tmem, 1);
    }
    __syncwarp();
    const int gy = oy + warp, gx = ox + lane;
    const bool in = lane < DW && gy < G.H && gx < G.W;
    float v[32];
    bool ok = conv32_read(S, tmem, warp, phase, G.wait_ns, v);
    if (in) {
      const size_t o = (size_t)n * 32 * plane + (size_t)gy * G.W + gx;
#pragma unroll
      for (int h = 0; h < 32; h += 16) {
        float m[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) m[c] = __ldg(a1 + o + (h + c) * plane);
#pragma unroll
        for (int c = 0; c < 16; ++c)
          d1[o + (h + c) * plane] = !ok ? __int_as_float(0x7fc00000) : m[c] > 0.0f ? v[h + c] : 0.0f;
      }
    }
    for (int t = 0; t < M2 / 128; ++t) ok = ok && umma::bar_wait(&S.bar[t], phase, G.wait_ns);
    if (!ok) S.failed = 1;
    umma::fence_before();
    __syncthreads();
    umma::fence_after();
    if (S.failed) break;
  }
  __syncthreads();
  // the tiles that a block leaves out keep an earlier pass's d1 and d2: the
  // gradients formed from them (layers 1 and 2) are marked as missing
  if (S.failed)
    for (int i = tid; i < OFF_W3; i += TILE_THREADS) atomicAdd(&grad[i], __int_as_float(0x7fc00000));
  if (warp == 0 && S.failed) umma::drain(&S.drained);
  if (warp == 0) umma::tmem_free(tmem, 256);
}

// ---------------------------------------------------------------- weight gradients
// dW[o][i][k] = sum over pixels p of D[o][p] X[i][p + k - 1]: a GEMM whose
// contraction runs over the pixels, both operands MN-major with their pieces
// stacked along M and N, so one MMA forms all nine products of the pieces.
// The tile is `tr` rows of `sw` columns flattened with a pitch of sw + 2: D is
// zero in the two columns between the rows, X has the halo there.
constexpr int WG_THREADS = 512;
constexpr int WG_K = 256;                   // pixels of a tile, at most
struct WgradGrid {
  int n, H, W, sw, tr, tx, ty;
  uint32_t inv;      // 2^16 / (sw + 2), rounded up
  uint32_t wait_ns;  // limit of a wait
  int64_t tiles;
};
constexpr int WG_X = 392;                   // input pixels of a tile: 256 + 2 * pitch + 3 at most, pitch <= 64

// Stages 32 channels of `src` (rows from oy, columns from ox, `rows` x `cols`
// of a pitch, zero elsewhere up to `len` pixels) as 12 planes of `stride` bytes.
// IT rounds of a chunk (8 channels of a pixel) per thread; `inv` = 2^16 /
// pitch rounded up (exact quotients: pixels < 512, pitch <= 64), a
// warp's lanes in one chunk.
template <int IT>
__device__ __forceinline__ void stage32(unsigned char* a, uint32_t stride, const float* __restrict__ src, size_t plane,
                                        int H, int W, int oy, int ox, int rows, int cols, int pitch, uint32_t inv,
                                        int len, int tid) {
  const int warps = (len + 31) / 32;
  float v[IT][8];  // every round's loads are under way before the first is split
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int wi = (tid >> 5) + it * (WG_THREADS / 32), c = wi / warps, m = (wi - c * warps) * 32 + (tid & 31);
    const int r = (int)((uint32_t)m * inv >> 16), q = m - r * pitch;
    const int gy = oy + r, gx = ox + q;
    const bool in = c < 4 && r < rows && q < cols && gy >= 0 && gy < H && gx >= 0 && gx < W;
    const float* sp = src + (size_t)(8 * c) * plane + (size_t)gy * W + gx;
#pragma unroll
    for (int e = 0; e < 8; ++e) v[it][e] = in ? __ldg(sp + e * plane) : 0.0f;
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int wi = (tid >> 5) + it * (WG_THREADS / 32), c = wi / warps, m = (wi - c * warps) * 32 + (tid & 31);
    uint4 p[3];
    umma::split8(v[it], p);
    if (c < 4 && m < len)
#pragma unroll
      for (int k = 0; k < 3; ++k) *reinterpret_cast<uint4*>(a + (k * 4 + c) * stride + m * 16) = p[k];
  }
}

template <int XP>
struct alignas(16) WgradSmem {
  unsigned char d[16 * WG_K * 16];          // 12 planes of D and 4 of zeros: M = 128
  unsigned char x[XP * WG_X * 16];          // layer 2: 12 planes of X, ones, zeros; layers 1, 3: one chunk
  uint32_t tmem;
  int failed;
  uint64_t full[2], empty[2], drained;
};
static_assert(sizeof(WgradSmem<14>) <= 227 * 1024 && sizeof(WgradSmem<1>) <= 227 * 1024, "one block per SM");

// Layer 2: 32 x 32 channels. The tensor core cuts the low bits of its sums,
// so they stay short: a stage is two taps over a third of the tile's pixels
// (at most six K steps), in one of two TMEM buffers; the warps of the lane
// quarters 0-2 (the pieces of D) add it to FP32 registers while the next stage
// runs, issued by warp 3. The ninth tap's stage has a plane of ones beside the
// planes of X: its column is the bias gradient.
constexpr int WG_CHAINS = 3;
constexpr int WG_ROW = 289;  // an output channel's 288 sums, padded to another bank per lane
__global__ void __launch_bounds__(WG_THREADS, 1)
    wgrad32_kernel(const float* __restrict__ x, const float* __restrict__ dy, float* __restrict__ dw,
                   float* __restrict__ db, const WgradGrid G) {
  extern __shared__ __align__(16) unsigned char smem[];
  WgradSmem<14>& S = *reinterpret_cast<WgradSmem<14>*>(smem);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const size_t plane = (size_t)G.H * G.W;
  const int pitch = G.sw + 2, klen = (G.tr * pitch + 15) / 16 * 16, xlen = klen + 2 * pitch + 2;
  const int kstep = (klen / 16 + WG_CHAINS - 1) / WG_CHAINS * 16, chains = (klen + kstep - 1) / kstep;
  for (int i = tid; i < 4 * WG_K; i += WG_THREADS)
    *reinterpret_cast<uint4*>(S.d + (12 * WG_K + i) * 16) = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < 2 * WG_X; i += WG_THREADS)
    *reinterpret_cast<uint4*>(S.x + (12 * WG_X + i) * 16) = make_uint4(i < WG_X ? 0x3f80u : 0u, 0, 0, 0);
  if (tid == 0) {
    S.failed = 0;
    for (int i = 0; i < 2; ++i) {
      umma::bar_init(&S.full[i]);
      umma::bar_init(&S.empty[i], 12);
    }
    umma::bar_init(&S.drained);
    umma::bar_init_fence();
  }
  if (warp == 0) umma::tmem_alloc(&S.tmem, 512);
  umma::fence_before();
  __syncthreads();
  umma::fence_after();
  const uint32_t tmem = S.tmem;
  const int piece = warp & 3, i0 = (warp >> 2) * 8;  // a thread's row of D is (piece, lane), its columns i0 ..
  const uint32_t tq = tmem + ((uint32_t)piece << 21);
  float acc[9][8], bias = 0.0f;
#pragma unroll
  for (int j = 0; j < 9; ++j)
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[j][c] = 0.0f;
  uint32_t stage = 0;
  bool ok = true;
  for (int64_t tile = blockIdx.x; tile < G.tiles; tile += gridDim.x) {
    int64_t t = tile;
    const int ox = (int)(t % G.tx) * G.sw;
    t /= G.tx;
    const int oy = (int)(t % G.ty) * G.tr, n = (int)(t / G.ty);
    stage32<2>(S.d, WG_K * 16, dy + (size_t)n * 32 * plane, plane, G.H, G.W, oy, ox, G.tr, G.sw, pitch, G.inv, klen, tid);
    stage32<4>(S.x, WG_X * 16, x + (size_t)n * 32 * plane, plane, G.H, G.W, oy - 1, ox - 1, G.tr + 2, pitch, pitch, G.inv,
               xlen, tid);
    umma::fence_smem();
    __syncthreads();
    if (warp == 3) {
      const uint64_t a0 = umma::desc_mn(umma::smem_addr(S.d), WG_K * 16), b0 = umma::desc_mn(umma::smem_addr(S.x), WG_X * 16);
#pragma unroll 1
      for (int g = 0; g < 5; ++g)
#pragma unroll 1
        for (int ch = 0; ch < chains; ++ch, ++stage) {
          // both buffers start empty
          if (stage >= 2) ok = ok && umma::bar_wait(&S.empty[stage & 1], (stage >> 1) - 1 & 1, G.wait_ns);
          umma::fence_after();
          if (ok && umma::elect()) {
            const int k0 = ch * kstep, k1 = min(klen, k0 + kstep);
#pragma unroll 1
            for (int tap = 2 * g; tap < 2 * g + 2 && tap < 9; ++tap) {
              const uint32_t d = tmem + (stage & 1) * 256 + (tap & 1) * 96;
              const uint32_t id = tap == 8 ? umma::idesc(128, 112, true) : umma::idesc(128, 96, true);
              const uint64_t bt = b0 + (tap / 3) * pitch + tap % 3;
              for (int k = k0; k < k1; k += 16) umma::mma(d, a0 + k, bt + k, id, k > k0);
            }
            umma::commit(&S.full[stage & 1]);
          }
          __syncwarp();
        }
      // the tile's planes are free once its last MMA is done
      ok = ok && umma::bar_wait(&S.full[(stage - 1) & 1], (stage - 1) >> 1 & 1, G.wait_ns);
    } else if (piece < 3) {
#pragma unroll
      for (int g = 0; g < 5; ++g)
#pragma unroll 1
        for (int ch = 0; ch < chains; ++ch, ++stage) {
          ok = ok && umma::bar_wait(&S.full[stage & 1], stage >> 1 & 1, G.wait_ns);
          umma::fence_after();
          const uint32_t col = tq + (stage & 1) * 256 + i0;
          // row 32 piece + o, column 32 piece' + i
#pragma unroll
          for (int j = 0; j < 2; ++j)
            if (2 * g + j < 9) {
              float v[8], u[8], s[8];
              umma::tmem_ld8(col + j * 96, v);
              umma::tmem_ld8(col + j * 96 + 32, u);
              umma::tmem_ld8(col + j * 96 + 64, s);
#pragma unroll
              for (int c = 0; c < 8; ++c) acc[2 * g + j < 9 ? 2 * g + j : 8][c] += v[c] + (u[c] + s[c]);
            }
          if (g == 4 && i0 == 0) {
            float v[8];
            umma::tmem_ld8(col + 96, v);
            bias += v[0];
          }
          umma::fence_before();
          __syncwarp();
          if (lane == 0 && ok) umma::bar_arrive(&S.empty[stage & 1]);
        }
    }
    if (!ok) S.failed = 1;
    __syncthreads();
    if (S.failed) break;
  }
  if (S.failed && warp == 3) umma::drain(&S.drained);
  // the pieces of D are added in shared memory, in turn, then once per block in global memory
  float* sum = reinterpret_cast<float*>(S.x);
  const float bad = S.failed ? __int_as_float(0x7fc00000) : 0.0f;
#pragma unroll 1
  for (int p = 2; p >= 0; --p) {
    __syncthreads();
    if (piece == p) {
#pragma unroll
      for (int j = 0; j < 9; ++j)
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          float* q = &sum[lane * WG_ROW + (i0 + c) * 9 + j];
          *q = (p == 2 ? bad : *q) + acc[j][c];
        }
      if (i0 == 0) sum[32 * WG_ROW + lane] = (p == 2 ? bad : sum[32 * WG_ROW + lane]) + bias;
    }
  }
  umma::fence_before();
  __syncthreads();
  for (int i = tid; i < NW2; i += WG_THREADS) atomicAdd(&dw[i], sum[i + i / 288]);
  if (tid < 32) atomicAdd(&db[tid], sum[32 * WG_ROW + tid]);
  if (warp == 0) umma::tmem_free(tmem, 512);
}

// Layers 1 and 3 (block y of the grid), the side with 32 channels as D:
//  layer 1: D = d1, X = the network input (both channels in one chunk of
//           pieces; element 6 is one: the bias gradient);
//  layer 3: D = a2, X = dz, whose taps are reversed (dW3[i][k] = sum over q
//           of a2[i][q] dz[q - k + 1]); its bias gradient is bce_kernel's.
// X's chunks of a row of taps are neighbouring pixels, 16 bytes apart: one MMA
// takes the three (and an unused fourth, N = 32). Each fifth of the tile's
// pixels has its own accumulators (short sums, see wgrad32_kernel). The next
// tile is read while the MMAs of this one run. 32 x 64 x 64 pixels: 26 us.
constexpr int IO_CHAINS = 5;
__global__ void __launch_bounds__(WG_THREADS, 1)
    wgrad_io_kernel(const float* __restrict__ x, const float* __restrict__ d1, const float* __restrict__ dz,
                    const float* __restrict__ a2, float* __restrict__ grad, const WgradGrid G) {
  extern __shared__ __align__(16) unsigned char smem[];
  WgradSmem<1>& S = *reinterpret_cast<WgradSmem<1>*>(smem);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const size_t plane = (size_t)G.H * G.W;
  const bool l3 = blockIdx.y != 0;
  const int pitch = G.sw + 2, klen = (G.tr * pitch + 15) / 16 * 16, xlen = klen + 2 * pitch + 3;
  const int kstep = (klen / 16 + IO_CHAINS - 1) / IO_CHAINS * 16, chains = (klen + kstep - 1) / kstep;
  for (int i = tid; i < 4 * WG_K; i += WG_THREADS)
    *reinterpret_cast<uint4*>(S.d + (12 * WG_K + i) * 16) = make_uint4(0, 0, 0, 0);
  if (tid == 0) {
    S.failed = 0;
    umma::bar_init(&S.full[0]);
    umma::bar_init(&S.drained);
    umma::bar_init_fence();
  }
  if (warp == 0) umma::tmem_alloc(&S.tmem, 512);
  umma::fence_before();
  __syncthreads();
  umma::fence_after();
  const uint32_t tmem = S.tmem;
  // taps of a thread's warp: grp, grp + 4, and for the first group 8
  const int piece = warp & 3, grp = warp >> 2;
  const uint32_t tq = tmem + ((uint32_t)piece << 21);
  float acc[3][8];
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[j][c] = 0.0f;
  // a thread's pixel of X, and its two chunks of D (rounds of 16 warps over 4 chunks of warps_d warps)
  const int warps_d = (klen + 31) / 32;
  float xv[2], dv[2][8];
  auto fetch = [&](int64_t t) {
    const bool live = t < G.tiles;
    const int ox = (int)(t % G.tx) * G.sw;
    t /= G.tx;
    const int oy = (int)(t % G.ty) * G.tr, n = (int)(t / G.ty);
    {
      const int r = (int)((uint32_t)tid * G.inv >> 16), gy = oy - 1 + r, gx = ox - 1 + tid - r * pitch;
      const bool in = live && r < G.tr + 2 && gy >= 0 && gy < G.H && gx >= 0 && gx < G.W;
      const float* p = (l3 ? dz + (size_t)n * plane : x + (size_t)n * 2 * plane) + (size_t)gy * G.W + gx;
      xv[0] = in ? __ldg(p) : 0.0f;
      xv[1] = in && !l3 ? __ldg(p + plane) : 0.0f;
    }
    const float* src = (l3 ? a2 : d1) + (size_t)n * 32 * plane;
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int wi = warp + it * (WG_THREADS / 32), c = wi / warps_d, m = (wi - c * warps_d) * 32 + lane;
      const int r = (int)((uint32_t)m * G.inv >> 16), q = m - r * pitch, gy = oy + r, gx = ox + q;
      const bool in = live && c < 4 && r < G.tr && q < G.sw && gy < G.H && gx < G.W;
      const float* p = src + (size_t)(8 * c) * plane + (size_t)gy * G.W + gx;
#pragma unroll
      for (int e = 0; e < 8; ++e) dv[it][e] = in ? __ldg(p + e * plane) : 0.0f;
    }
  };
  fetch(blockIdx.x);
  uint32_t phase = 0;
  for (int64_t tile = blockIdx.x; tile < G.tiles; tile += gridDim.x, phase ^= 1) {
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int wi = warp + it * (WG_THREADS / 32), c = wi / warps_d, m = (wi - c * warps_d) * 32 + lane;
      uint4 p[3];
      umma::split8(dv[it], p);
      if (c < 4 && m < klen)
#pragma unroll
        for (int k = 0; k < 3; ++k) *reinterpret_cast<uint4*>(S.d + ((k * 4 + c) * WG_K + m) * 16) = p[k];
    }
    if (tid < xlen) {
      uint32_t h0, m0, l0;
      umma::split2(xv[0], xv[1], &h0, &m0, &l0);
      *reinterpret_cast<uint4*>(S.x + tid * 16) = make_uint4(__byte_perm(h0, m0, 0x5410), __byte_perm(l0, h0, 0x7610),
                                                             __byte_perm(m0, l0, 0x7632), 0x3f80u);
    }
    umma::fence_smem();
    __syncthreads();
    if (warp == 3 && umma::elect()) {
      const uint64_t a0 = umma::desc_mn(umma::smem_addr(S.d), WG_K * 16), b0 = umma::desc_mn(umma::smem_addr(S.x), 16);
      constexpr uint32_t id = umma::idesc(128, 32, true);
#pragma unroll 1
      for (int ch = 0; ch < chains; ++ch)
        for (int k = ch * kstep; k < min(klen, (ch + 1) * kstep); k += 16)
#pragma unroll
          for (int ky = 0; ky < 3; ++ky)
            umma::mma(tmem + ch * 96 + ky * 32, a0 + k, b0 + k + ky * pitch, id, k > ch * kstep);
      umma::commit(&S.full[0]);
    }
    __syncwarp();
    fetch(tile + gridDim.x);
    if (!umma::bar_wait(&S.full[0], phase, G.wait_ns)) S.failed = 1;
    umma::fence_after();
    if (piece < 3) {
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int tap = grp + 4 * j;
        if (tap < 9)
#pragma unroll 1
          for (int ch = 0; ch < chains; ++ch) {
            float v[8];
            umma::tmem_ld8(tq + ch * 96 + (tap / 3) * 32 + (tap % 3) * 8, v);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[j][c] += v[c];
          }
      }
    }
    umma::fence_before();
    __syncthreads();
    umma::fence_after();
    if (S.failed) break;
  }
  if (S.failed && warp == 3) umma::drain(&S.drained);
  // sums over the pieces of X, then over those of D in shared memory, then one atomic per block
  float* sum = reinterpret_cast<float*>(S.d);  // [32][19]: 18 weights and the bias of a channel
  const float bad = S.failed ? __int_as_float(0x7fc00000) : 0.0f;
#pragma unroll 1
  for (int p = 2; p >= 0; --p) {
    __syncthreads();
    if (piece == p)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int tap = grp + 4 * j;
        if (tap >= 9) break;
        const float* v = acc[j];
        float* q = sum + lane * 19;
        const float o[3] = {v[0] + (v[1] + v[2]), v[3] + (v[4] + v[5]), v[6]};
        const int at[3] = {l3 ? 8 - tap : tap, 9 + tap, 18};
#pragma unroll
        for (int e = 0; e < 3; ++e)
          if (e < 2 || tap == 4) q[at[e]] = (p == 2 ? bad : q[at[e]]) + o[e];
      }
  }
  umma::fence_before();
  __syncthreads();
  for (int i = tid; i < 32 * 19; i += WG_THREADS) {
    const int c = i / 19, e = i - 19 * c;
    if (l3) {
      if (e < 9) atomicAdd(&grad[OFF_W3 + c * 9 + e], sum[i]);
    } else {
      atomicAdd(&grad[e < 18 ? OFF_W1 + c * 18 + e : OFF_B1 + c], sum[i]);
    }
  }
  if (warp == 0) umma::tmem_free(tmem, 512);
}

// Logit -> probability, and the BCE loss / logit gradient:
// loss = w y softplus(-z) + (1 - y) softplus(z), averaged over pixels; db: sum
// of the logit gradients (layer 3's bias gradient).
constexpr int BCE_THREADS = 256;
__global__ void __launch_bounds__(BCE_THREADS) bce_kernel(const float* __restrict__ z, const float* __restrict__ yl, int64_t n, float pos_w,
                           float* __restrict__ dz, float* __restrict__ loss, float* __restrict__ db) {
  float acc = 0.0f, dsum = 0.0f;
  const float inv = 1.0f / (float)n;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float zi = z[i], yi = yl[i];
    float sp_pos = fmaxf(zi, 0.0f) + log1pf(expf(-fabsf(zi)));  // softplus(z)
    float sp_neg = sp_pos - zi;                                  // softplus(-z)
    acc += pos_w * yi * sp_neg + (1.0f - yi) * sp_pos;
    float s = 1.0f / (1.0f + expf(-zi));
    const float d = (-pos_w * yi * (1.0f - s) + (1.0f - yi) * s) * inv;
    dz[i] = d;
    dsum += d;
  }
  __shared__ float red[2][BCE_THREADS / 32];
  for (int o = 16; o > 0; o >>= 1) {
    acc += __shfl_down_sync(0xffffffffu, acc, o);
    dsum += __shfl_down_sync(0xffffffffu, dsum, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = acc;
    red[1][threadIdx.x >> 5] = dsum;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    float t = 0.0f;
    for (int i = 0; i < BCE_THREADS / 32; ++i) t += red[threadIdx.x][i];
    atomicAdd(threadIdx.x ? db : loss, threadIdx.x ? t : t * inv);
  }
}

__global__ void adam_kernel(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ g, __nv_bfloat16* __restrict__ wb, int n, float lr, float b1,
                            float b2, float eps, float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    float gi = g[i];
    float mi = b1 * m[i] + (1.0f - b1) * gi;
    float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    store_weight(wb, i, wi);
  }
}

__global__ void to_bf16_kernel(const float* __restrict__ w, __nv_bfloat16* __restrict__ wb, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    store_weight(wb, i, w[i]);
}

// Launches a persistent tile kernel with its shared memory on `per_sm` blocks per SM.
template <class K, class... Args>
int launch_tiles(K kern, int threads, size_t smem, int per_sm, int gy, int64_t tiles, cudaStream_t s, Args... args) {
  int dev = 0, sms = 0;
  QSL_CHECK_CUDA(cudaGetDevice(&dev));
  QSL_CHECK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  QSL_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int64_t blocks = std::min<int64_t>(tiles, std::max(1, sms * per_sm / gy));
  kern<<<dim3((unsigned)blocks, gy), threads, smem, s>>>(args...);
  qsl::count_launch();
  QSL_CHECK_CUDA(cudaGetLastError());
  return QSL_OK;
}

TileGrid tile_grid(int n, int H, int W, int w, int h, uint32_t wait_ns) {
  TileGrid G;
  G.wait_ns = wait_ns;
  G.n = n;
  G.H = H;
  G.W = W;
  G.tx = (W + w - 1) / w;
  G.ty = (H + h - 1) / h;
  G.tiles = (int64_t)n * G.tx * G.ty;
  return G;
}

template <int CIN, int COUT, bool RELU>
int launch_conv(const float* x, const __nv_bfloat16* w, const float* b, float* y, int n, int H, int W, cudaStream_t s) {
  const size_t smem = sizeof(float) * (CIN * TH * TH + COUT * CIN * 9);
  auto kern = conv3x3_kernel<CIN, COUT, RELU>;
  QSL_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int tx = (int)(((int64_t)W + T - 1) / T), ty = (int)(((int64_t)H + T - 1) / T);
  kern<<<(unsigned)((int64_t)n * tx * ty), CONV_THREADS, smem, s>>>(x, w, b, y, H, W, tx, ty);
  qsl::count_launch();
  QSL_CHECK_CUDA(cudaGetLastError());
  return QSL_OK;
}

// Segment width (the one that wastes least of a row), equal output columns per
// task, and the rows per task that let the blocks, two per SM, finish soonest
// (a task computes four rows more than it yields).
FwdGrid fwd_grid(int n, int H, int W, int slots, uint32_t wait_ns) {
  FwdGrid G;
  G.wait_ns = wait_ns;
  G.H = H;
  G.W = W;
  int64_t best = INT64_MAX;
  for (int P = 32; P <= SP; P *= 2) {
    const int64_t tx = ((int64_t)W + P - 7) / (P - 6), cost = tx * P;
    if (cost < best) {
      best = cost;
      G.P = P;
      G.tx = (int)tx;
    }
  }
  G.nseg = SP / G.P;
  G.zw = (int)(((int64_t)W + G.tx - 1) / G.tx);
  int64_t time = INT64_MAX;
  for (int ty = 1; ty <= std::min(H, 1024); ++ty) {
    const int h = (int)(((int64_t)H + ty - 1) / ty);
    const int64_t groups = ((int64_t)n * G.tx * ty + G.nseg - 1) / G.nseg, t = (groups + slots - 1) / slots * (h + 4);
    if (t < time) {
      time = t;
      G.h = h;
      G.ty = (int)(((int64_t)H + h - 1) / h);
    }
  }
  G.tasks = (int64_t)n * G.tx * G.ty;
  G.groups = (G.tasks + G.nseg - 1) / G.nseg;
  return G;
}

// Strips of equal width, at most 62 columns, and as many rows as 256 pixels hold.
WgradGrid wgrad_grid(int n, int H, int W, uint32_t wait_ns) {
  WgradGrid G;
  G.wait_ns = wait_ns;
  G.n = n;
  G.H = H;
  G.W = W;
  const int strips = (W + 61) / 62;
  G.sw = (W + strips - 1) / strips;
  G.inv = 65536u / (G.sw + 2) + 1;
  G.tr = std::min(H, WG_K / (G.sw + 2));
  G.tx = (W + G.sw - 1) / G.sw;
  G.ty = (H + G.tr - 1) / G.tr;
  G.tiles = (int64_t)n * G.tx * G.ty;
  return G;
}

}  // namespace

struct qsl_cnn {
  float* w = nullptr;            // FP32 master parameters
  __nv_bfloat16* wb = nullptr;   // BF16 copy used by the passes, and the operand layouts
  float* m = nullptr;            // Adam moments
  float* v = nullptr;
  int64_t steps = 0;
  float* act = nullptr;          // activations of the largest batch seen (floats)
  size_t act_cap = 0;
};

namespace {

int ensure_act(qsl_cnn* c, size_t need, cudaStream_t s) {
  if (need <= c->act_cap) return QSL_OK;
  if (c->act) QSL_CHECK_CUDA(cudaFreeAsync(c->act, s));
  c->act = nullptr;
  c->act_cap = 0;
  QSL_CHECK_CUDA(qsl::alloc_async((void**)&c->act, need * sizeof(float), s));
  c->act_cap = need;
  return QSL_OK;
}

bool dims_ok(int n, int H, int W) { return n >= 1 && H >= 1 && W >= 1 && (int64_t)n * H * W <= (1ll << 31); }

// Network input of each z-slice of a coarse volume:
// channel 0 the FLEDGE map over its largest finite value in the slice
// (non-finite entries 0), channel 1 (log10 Q - 2) / 2 clamped to [-2, 3], a
// missing Q (NaN) counted as the floor Q = 2 and an infinite one as the top
// of the range.
// A slice belongs to a cluster of CL blocks that share its maximum. Clusters are
// placed at about 20 per us, a block goes over a slice at about 0.7 pixels per ns:
// one block per slice for small slices and for many middling ones (one_block).
// Slices x pixels, one block and 8 (and one block of the kernel before): 600 of
// 32^2 6.2 and 32 us (6.2), 64 of 48^2 6.2 and 7.8 (6.2), 16 of 48^2 6.2 and 5.8,
// 300 of 64^2 8.2 and 21 (10), 64 of 96^2 14 and 9.2, 300 of 128^2 35 and 29, 1,200
// of 128^2 90 and 123, 150 of 256^2 227 and 59 (230).
constexpr int FEAT_CLUSTER = 8;
bool one_block(int slices, int64_t plane) { return plane <= 1024 || (plane <= 16384 && plane <= 40 * (int64_t)slices); }
template <int CL, int THREADS>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(THREADS)
    features_kernel(const float* __restrict__ S, const float* __restrict__ Q, int64_t plane, float* __restrict__ X) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ float red[THREADS / 32], block_max;
  const int z = blockIdx.x / CL, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t first = (int64_t)(CL > 1 ? cluster.block_rank() : 0) * THREADS + threadIdx.x, step = CL * THREADS;
  const float* s = S + (size_t)z * plane;
  const float* q = Q + (size_t)z * plane;
  float m = 0.0f;
#pragma unroll 4
  for (int64_t i = first; i < plane; i += step) {
    const float v = s[i];
    if (isfinite(v) && v > m) m = v;
  }
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) red[warp] = m;
  __syncthreads();
  if (warp == 0) {
    m = lane < THREADS / 32 ? red[lane] : 0.0f;
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) block_max = m;
  }
  if constexpr (CL > 1) {
    cluster.sync();
    m = 0.0f;
    for (int r = 0; r < CL; ++r) m = fmaxf(m, *cluster.map_shared_rank(&block_max, r));
    cluster.sync();  // no block leaves while another reads its maximum
  } else {
    __syncthreads();
    m = block_max;
  }
  const float smax = fmaxf(m, 1e-12f);
  float* x0 = X + (size_t)z * 2 * plane;
  float* x1 = x0 + plane;
#pragma unroll 2
  for (int64_t i = first; i < plane; i += step) {
    const float v = s[i] / smax;
    x0[i] = isfinite(v) ? v : 0.0f;
    float qv = q[i];
    if (isnan(qv) || (isinf(qv) && qv < 0)) qv = 2.0f;  // no Q: the floor Q = 2
    x1[i] = isinf(qv) ? 3.0f : fminf(fmaxf((log10f(fmaxf(qv, 2.0f)) - 2.0f) * 0.5f, -2.0f), 3.0f);
  }
}

// out = 1 where any cell of the 3 x 3 x 3 neighbourhood (clipped to the
// volume; 3 x 3 for one slice) of `in` is nonzero.
__global__ void dilate_kernel(const uint8_t* __restrict__ in, int nz, int ny, int nx, uint8_t* __restrict__ out) {
  const int64_t n = (int64_t)nz * ny * nx;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % nx), y = (int)((i / nx) % ny), z = (int)(i / ((int64_t)nx * ny));
    uint8_t v = 0;
    for (int dz = -1; dz <= 1 && !v; ++dz) {
      const int zz = z + dz;
      if (zz < 0 || zz >= nz) continue;
      for (int dy = -1; dy <= 1 && !v; ++dy) {
        const int yy = y + dy;
        if (yy < 0 || yy >= ny) continue;
        for (int dx = -1; dx <= 1; ++dx) {
          const int xx = x + dx;
          if (xx < 0 || xx >= nx) continue;
          if (in[((int64_t)zz * ny + yy) * nx + xx]) {
            v = 1;
            break;
          }
        }
      }
    }
    out[i] = v;
  }
}

// Limit of a kernel's waits: WAIT_NS, or none at all for a kernel of the set
// `kernels` (qsl_check_cnn_waits; 0 in the passes).
uint32_t wait_of(int kernels, int kernel) { return kernels & kernel ? 0 : umma::WAIT_NS; }

int forward_pass(qsl_cnn* c, const float* x, int n, int H, int W, float* prob, int kernels, cudaStream_t s) {
  int dev = 0, sms = 0;
  QSL_CHECK_CUDA(cudaGetDevice(&dev));
  QSL_CHECK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const FwdGrid G = fwd_grid(n, H, W, 2 * sms, wait_of(kernels, QSL_CNN_FORWARD));
  // setmaxnreg.inc waits for registers of the launch: 128 x 72 + 128 x 120 + 32 x n <= 288 x n
  cudaFuncAttributes at;
  QSL_CHECK_CUDA(cudaFuncGetAttributes(&at, forward_kernel));
  if (at.numRegs < 96) {
    qsl::set_error("the forward kernel was built with %d registers, its split needs 96", at.numRegs);
    return QSL_ECUDA;
  }
  return launch_tiles(forward_kernel, FWD_THREADS, sizeof(FwdSmem), 2, 1, G.groups, s, x, c->wb, c->w, prob, G);
}

int loss_grad_pass(qsl_cnn* c, const float* x, const float* y, int n, int H, int W, float pos_weight, float* loss,
                   float* grad, int kernels, cudaStream_t s) {
  size_t P = (size_t)n * H * W;
  int rc = ensure_act(c, P * (4 * 32 + 2), s);  // a1, a2, d2, d1 (32 channels each), z, dz
  if (rc) return rc;
  float *a1 = c->act, *a2 = a1 + P * 32, *d2 = a2 + P * 32, *d1 = d2 + P * 32, *z = d1 + P * 32, *dz = z + P;
  QSL_CHECK_CUDA(cudaMemsetAsync(loss, 0, sizeof(float), s));
  QSL_CHECK_CUDA(cudaMemsetAsync(grad, 0, NPAR * sizeof(float), s));
  const TileGrid GD = tile_grid(n, H, W, DW, DH, wait_of(kernels, QSL_CNN_DGRAD));
  if ((rc = launch_conv<C1, C2, true>(x, c->wb + OFF_W1, c->w + OFF_B1, a1, n, H, W, s))) return rc;
  if ((rc = launch_conv<C2, C2, true>(a1, c->wb + OFF_W2, c->w + OFF_B2, a2, n, H, W, s))) return rc;
  if ((rc = launch_conv<C2, 1, false>(a2, c->wb + OFF_W3, c->w + OFF_B3, z, n, H, W, s)))
    return rc;
  bce_kernel<<<(int)std::min<size_t>((P + BCE_THREADS - 1) / BCE_THREADS, 1024), BCE_THREADS, 0, s>>>(z, y, (int64_t)P, pos_weight, dz, loss,
                                                                          grad + OFF_B3);
  qsl::count_launch();
  QSL_CHECK_CUDA(cudaGetLastError());
  if ((rc = launch_tiles(dgrad_kernel, TILE_THREADS, sizeof(TileSmem), 2, 1, GD.tiles, s, dz, c->wb, a1, a2, d1, d2, grad, GD)))
    return rc;
  WgradGrid GW = wgrad_grid(n, H, W, wait_of(kernels, QSL_CNN_WGRAD2));
  if ((rc = launch_tiles(wgrad32_kernel, WG_THREADS, sizeof(WgradSmem<14>), 1, 1, GW.tiles, s, a1, d2, grad + OFF_W2,
                         grad + OFF_B2, GW)))
    return rc;
  GW.wait_ns = wait_of(kernels, QSL_CNN_WGRAD13);
  return launch_tiles(wgrad_io_kernel, WG_THREADS, sizeof(WgradSmem<1>), 1, 2, GW.tiles, s, x, d1, dz, a2, grad, GW);
}

}  // namespace

extern "C" {

int qsl_cnn_features(const float* S, const float* Q, int nz, int ny, int nx, float* X, void* stream_) {
  if (!S || !Q || !X || nz < 1 || ny < 1 || nx < 1) {
    qsl::set_error("qsl_cnn_features: bad arguments");
    return QSL_EINVAL;
  }
  const int64_t plane = (int64_t)ny * nx;
  constexpr int MAX_SLICES = 1 << 24;  // per launch
  for (int z = 0; z < nz; z += std::min(MAX_SLICES, nz - z)) {
    const int slices = std::min(MAX_SLICES, nz - z);
    const bool one = one_block(slices, plane);
    (one ? features_kernel<1, 256> : features_kernel<FEAT_CLUSTER, 512>)
        <<<slices*(one ? 1 : FEAT_CLUSTER), one ? 256 : 512, 0, (cudaStream_t)stream_>>>(
            S + z * plane, Q + z * plane, plane, X + 2 * z * plane);
    qsl::count_launch();
    QSL_CHECK_CUDA(cudaGetLastError());
  }
  return QSL_OK;
}

int qsl_mask_dilate(const uint8_t* in, int nz, int ny, int nx, uint8_t* out, void* stream_) {
  if (!in || !out || in == out || nz < 1 || ny < 1 || nx < 1) {
    qsl::set_error("qsl_mask_dilate: bad arguments (in and out must differ)");
    return QSL_EINVAL;
  }
  const int64_t n = (int64_t)nz * ny * nx;
  int blocks = (int)((n + 255) / 256);
  if (blocks > 152 * 32) blocks = 152 * 32;
  dilate_kernel<<<blocks, 256, 0, (cudaStream_t)stream_>>>(in, nz, ny, nx, out);
  qsl::count_launch();
  QSL_CHECK_CUDA(cudaGetLastError());
  return QSL_OK;
}

int qsl_cnn_create(const float* params, qsl_cnn** out) {
  if (!params || !out) {
    qsl::set_error("NULL argument");
    return QSL_EINVAL;
  }
  qsl_cnn* c = new qsl_cnn();
  cudaError_t e = cudaMalloc((void**)&c->w, NPAR * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc((void**)&c->wb, NWB * sizeof(__nv_bfloat16));
  if (e == cudaSuccess) e = cudaMalloc((void**)&c->m, NPAR * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc((void**)&c->v, NPAR * sizeof(float));
  if (e == cudaSuccess) e = cudaMemcpy(c->w, params, NPAR * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(c->wb, 0, NWB * sizeof(__nv_bfloat16));  // the operands' unused elements
  if (e == cudaSuccess) e = cudaMemset(c->m, 0, NPAR * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(c->v, 0, NPAR * sizeof(float));
  if (e != cudaSuccess) {
    qsl::set_error("CNN allocation failed: %s", cudaGetErrorString(e));
    qsl_cnn_free(c);
    return QSL_ENOMEM;
  }
  to_bf16_kernel<<<(NPAR + 255) / 256, 256>>>(c->w, c->wb, NPAR);
  qsl::count_launch();
  if ((e = cudaDeviceSynchronize()) != cudaSuccess) {
    qsl::set_error("CNN init failed: %s", cudaGetErrorString(e));
    qsl_cnn_free(c);
    return QSL_ECUDA;
  }
  *out = c;
  return QSL_OK;
}

int qsl_cnn_params(const qsl_cnn* c, float* params) {
  if (!c || !params) {
    qsl::set_error("NULL argument");
    return QSL_EINVAL;
  }
  QSL_CHECK_CUDA(cudaMemcpy(params, c->w, NPAR * sizeof(float), cudaMemcpyDeviceToHost));
  return QSL_OK;
}

int qsl_cnn_forward(qsl_cnn* c, const float* x, int n, int H, int W, float* prob, void* stream_) {
  // a task may hang over the image by its rows (H / 1000 at these heights) or 128
  // columns: coordinates stay 32-bit
  constexpr int MAX_SIDE = INT32_MAX - (1 << 22);
  if (!c || !x || !prob || !dims_ok(n, H, W) || H > MAX_SIDE || W > MAX_SIDE) {
    qsl::set_error("bad CNN forward arguments (n h w at most 2^31, h and w at most 2^31 - 2^22 - 1)");
    return QSL_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream_;
  // prob may lie over x: blocks read and write at different times, so the pass
  // then writes beside it
  const size_t P = (size_t)n * H * W;
  const uintptr_t xa = (uintptr_t)x, pa = (uintptr_t)prob;
  if (pa >= xa + 2 * P * sizeof(float) || xa >= pa + P * sizeof(float)) return forward_pass(c, x, n, H, W, prob, 0, s);
  int rc = ensure_act(c, P, s);
  if (rc || (rc = forward_pass(c, x, n, H, W, c->act, 0, s))) return rc;
  QSL_CHECK_CUDA(cudaMemcpyAsync(prob, c->act, P * sizeof(float), cudaMemcpyDeviceToDevice, s));
  return QSL_OK;
}

int qsl_cnn_loss_grad(qsl_cnn* c, const float* x, const float* y, int n, int H, int W, float pos_weight, float* loss,
                      float* grad, void* stream_) {
  if (!c || !x || !y || !loss || !grad || !dims_ok(n, H, W) || !(pos_weight > 0)) {
    qsl::set_error("bad CNN loss/gradient arguments");
    return QSL_EINVAL;
  }
  return loss_grad_pass(c, x, y, n, H, W, pos_weight, loss, grad, 0, (cudaStream_t)stream_);
}

int qsl_check_cnn_waits(qsl_cnn* c, const float* x, const float* y, int n, int H, int W, float* prob, float* loss,
                        float* grad, int kernels, void* stream_) {
  if (!c || !x || !y || !prob || !loss || !grad || !dims_ok(n, H, W)) {
    qsl::set_error("bad CNN check arguments");
    return QSL_EINVAL;
  }
  const int rc = forward_pass(c, x, n, H, W, prob, kernels, (cudaStream_t)stream_);
  return rc ? rc : loss_grad_pass(c, x, y, n, H, W, 1.0f, loss, grad, kernels, (cudaStream_t)stream_);
}

int qsl_cnn_adam_step(qsl_cnn* c, const float* grad, float lr, float beta1, float beta2, float eps, void* stream_) {
  cudaStream_t s = (cudaStream_t)stream_;
  if (!c || !grad || !(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0)) {
    qsl::set_error("bad Adam arguments");
    return QSL_EINVAL;
  }
  c->steps += 1;
  float c1 = 1.0f - powf(beta1, (float)c->steps), c2 = 1.0f - powf(beta2, (float)c->steps);
  adam_kernel<<<(NPAR + 255) / 256, 256, 0, s>>>(c->w, c->m, c->v, grad, c->wb, NPAR, lr, beta1, beta2, eps, c1, c2);
  qsl::count_launch();
  QSL_CHECK_CUDA(cudaGetLastError());
  return QSL_OK;
}

void qsl_cnn_free(qsl_cnn* c) {
  if (!c) return;
  if (c->act) cudaFree(c->act);
  cudaFree(c->w);
  cudaFree(c->wb);
  cudaFree(c->m);
  cudaFree(c->v);
  delete c;
}

int qsl_cnn_nparams(void) { return NPAR; }

}  // extern "C"

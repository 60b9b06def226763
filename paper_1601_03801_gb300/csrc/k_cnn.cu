// Learned warm start of the smoothing solve: a 3-layer 3x3x3 convolutional network
// 4 -> 32 -> 32 -> 4 (ReLU after the first two) on the averaging mesh, trained on
// the GPU by these kernels.  Weights and activations are stored in bfloat16,
// products accumulate in FP32.  Fields are channels-last [voxel][channel]; a tap
// outside the mesh wraps on periodic axes and reads zero otherwise.
//
// Parameter order (shared with the FP64 reference network of the tests):
//   w1[32][4][27] b1[32] w2[32][32][27] b2[32] w3[4][32][27] b3[4],
//   tap t = (kz*3 + ky)*3 + kx at offset (kx-1, ky-1, kz-1).
// Backward: data gradients are the same convolutions with mirrored taps and
// transposed weights; weight gradients are per-tap voxel sums (per-block partials
// reduced in a fixed order); gradients are FP32 words; loss = mean (y - target)^2; Adam on
// FP32 master weights.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"

namespace sedi {

namespace {

struct Grid3 {
  int nx, ny, nz;
  int per[3];
  int64_t n;
};

// the cell at (x, y, z), each from -1 to beyond the last cell: wrapped where the axis is
// periodic and the place one cell outside, else -1
__device__ __forceinline__ int64_t nb_of(const Grid3& g, int x, int y, int z) {
  int c[3] = {x, y, z};
  const int n[3] = {g.nx, g.ny, g.nz};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (c[a] == -1 && g.per[a]) c[a] = n[a] - 1;
    else if (c[a] == n[a] && g.per[a]) c[a] = 0;
    if (c[a] < 0 || c[a] >= n[a]) return -1;
  }
  return ((int64_t)c[2] * g.ny + c[1]) * g.nx + c[0];
}

// ---------------------------------------------------------------- tensor-core kernels
// Both products of a layer, the convolution and the weight gradient, are implicit GEMMs
// on mma.sync m16n8k16 (bf16 in, FP32 accumulate) over tiles of 8 x 8 x 4 or 8 x 4 x 4
// voxels that are staged with a halo of one voxel in shared memory: a tap is an offset
// of the staged row, and every fragment is one ldmatrix of rows of 8 voxels along x.
// FP32 gradients take part as three bf16 planes, the top, middle and low 8 bits of the
// significand: their sum is the FP32 word (see split3), and each product with a bf16
// weight or activation is exact, so the operands are the FP32 ones.  The tensor cores' accumulation
// does not round to nearest, so the top planes' products are summed in chains of two
// instructions that are then added in FP32, and the lower planes' (2^-8 of them) apart.
// The two layers whose outputs are rounded to bf16 keep one order of summation, tap after
// tap and channel after channel: layer 1 on the FP32 pipe (k_conv1) and layer 2 as one
// chain of instructions, since a last bit there can move an activation by 2^-9.
//
// Rows: x [v][16] (4 fields, 12 zeros), a1 and a2 [v][32], the output gradient
// gy [v][3 planes x 4, 4 zeros], hidden gradients g2 and g1 [v][3 planes][32].
// In shared memory the 16-byte parts of a row are permuted by the row's number, so that
// the 8 rows of an ldmatrix meet every bank once.
constexpr int kTX = 8;              // voxels of a tile along x, all of them a fragment's rows
constexpr int kHX = kTX + 2;
constexpr int kConvTY = 8, kConvTZ = 4, kConvThreads = 256;
constexpr int kWgTY = 4, kWgTZ = 4;
constexpr int kWgMaxBlocks = 160;   // partial weight gradients at most

// byte of 16-byte part c of row r, rows of 2 KC bytes
template <int KC>
__device__ __forceinline__ uint32_t row_at(int r, int c) {
  if (KC == 32) return (uint32_t)(r * 64 + ((c ^ ((r >> 1) & 3)) << 4));
  return (uint32_t)(r * 32 + ((c ^ ((r >> 2) & 1)) << 4));
}

__device__ __forceinline__ void ldsm4(uint32_t* r, uint32_t at) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(at)
               : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t* r, uint32_t at) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(at)
               : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t* r, uint32_t at) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(at)
               : "memory");
}
// 16 bytes to shared memory, zeros where `src` is not to be read
__device__ __forceinline__ void cp16(uint32_t to, const void* src, bool ok) {
  const int bytes = ok ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void mma_bf16_16816(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// g = p[0] + p[1] + p[2], exactly from 2^-110 up (below, the low plane can lie under bf16's least
// word, 2^-133); infinities and NaN stay in p[0]
__device__ __forceinline__ void split3(float g, __nv_bfloat16* p) {
  const uint32_t u = __float_as_uint(g);
  if ((u & 0x7f800000u) == 0x7f800000u) {
    p[0] = __float2bfloat16_rn(g);
    p[1] = p[2] = __float2bfloat16_rn(0.0f);
    return;
  }
  const float hi = __uint_as_float(u & 0xffff0000u), r = g - hi;
  const float mid = __uint_as_float(__float_as_uint(r) & 0xffff0000u);
  p[0] = __float2bfloat16_rn(hi);
  p[1] = __float2bfloat16_rn(mid);
  p[2] = __float2bfloat16_rn(r - mid);
}
__device__ __forceinline__ uint32_t pair_of(__nv_bfloat16 a, __nv_bfloat16 b) {
  return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

struct Tiling {
  unsigned nx, ny;  // tiles along x and y
  unsigned n;       // tiles (a mesh has fewer than 2^31 cells)
  __device__ __forceinline__ int3 at(unsigned tile, int ty, int tz) const {
    const unsigned q = tile / nx, z = q / ny;
    return make_int3((int)(tile - q * nx) * kTX, (int)(q - z * ny) * ty, (int)z * tz);
  }
};
Tiling tiling(const Grid3& g, int ty, int tz) {
  Tiling t;
  t.nx = (g.nx + kTX - 1) / kTX;
  t.ny = (g.ny + ty - 1) / ty;
  t.n = t.nx * t.ny * ((g.nz + tz - 1) / tz);
  return t;
}

// Stage the rows (ROW 16-byte parts: planes of KC channels) of the tile at (x0, y0, z0) and
// of its halo: plane p starts at `to` + p * rows * 2 KC bytes.  Zeros outside the mesh.
template <int KC, int NP, int TY, int TZ, int THREADS>
__device__ __forceinline__ void stage_halo(uint32_t to, const __nv_bfloat16* in, const Grid3& g, int x0,
                                           int y0, int z0) {
  constexpr int HY = TY + 2, HZ = TZ + 2, HV = kHX * HY * HZ, CH = KC / 8, ROW = CH * NP;
  for (int k = threadIdx.x; k < HV * ROW; k += THREADS) {
    const int hv = k / ROW, c = k % ROW;
    const int hx = hv % kHX, hy = (hv / kHX) % HY, hz = hv / (kHX * HY);
    const int64_t q = nb_of(g, x0 + hx - 1, y0 + hy - 1, z0 + hz - 1);
    cp16(to + (uint32_t)((c / CH) * HV * 2 * KC) + row_at<KC>(hv, c % CH),
         in + (q < 0 ? 0 : q) * (NP * KC) + c * 8, q >= 0);
  }
}

// out[v][n] = bias[n] + sum_t sum_p sum_k w[t][n][k] in[v + off(t)][p][k]
// What it writes: bf16 with ReLU (OUT_RELU, [v][32]), FP32 (OUT_F32, [v][4], the first four
// of 8 columns), or three bf16 planes where mask[v][n] > 0, else zeros (OUT_SPLIT).
//
// A warp takes 2 x 16 voxels x 8 NT outputs, so that a weight fragment serves two
// products and an input fragment NT of them.  Weights stay in shared memory while the
// block takes one tile after the other.  Bound by the tensor cores' mma.sync rate and the
// ldmatrix reads before it, with the staging of a tile not overlapped.  On 64 x 32 x 64
// voxels, against a thread a voxel with FP32 operations: 32 -> 32 of three planes
// 737 -> 98 us, layer 3 228 -> 18 us, its data gradient 61 -> 26 us; layer 2, which read
// its fragments from L2 word by word, 110 -> 27 us.
enum { OUT_RELU, OUT_F32, OUT_SPLIT };

template <int KC, int NP, int NT>
constexpr int conv_smem() {
  return 27 * NT * 8 * KC * 2 + kHX * (kConvTY + 2) * (kConvTZ + 2) * KC * 2 * NP;
}

template <int KC, int NP, int NT, int OUT>
__global__ void __launch_bounds__(kConvThreads)
    k_conv(const __nv_bfloat16* in, const __nv_bfloat16* wt, const float* bias, void* out,
           const __nv_bfloat16* mask, Grid3 g, Tiling tl) {
  static_assert(NT == 4 || (NT == 1 && KC == 32), "");
  constexpr int TY = kConvTY, TZ = kConvTZ, HY = TY + 2, HV = kHX * HY * (TZ + 2);
  constexpr int W16 = 27 * NT * 8 * KC / 8;  // 16-byte words of the weights
  constexpr int KS = KC / 16;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const uint32_t sw = (uint32_t)__cvta_generic_to_shared(smem_raw);
  const uint32_t sx = sw + W16 * 16;
  for (int k = threadIdx.x; k < W16; k += kConvThreads) cp16(sw + k * 16, wt + k * 8, true);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gid = lane >> 2, tig = lane & 3;
  // the lane's row and part of an input fragment, first of the warp's two
  const int z = warp >> 1;
  const int ar = (z * HY + (warp & 1) * 4 + ((lane >> 3) & 1)) * kHX + (lane & 7), ac = lane >> 4;
  const int br = ((lane >> 4) & 1) * 8 + (lane & 7), bc = (lane >> 3) & 1;
  float bv[NT][2];
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int e = 0; e < 2; ++e) bv[n][e] = bias ? bias[n * 8 + 2 * tig + e] : 0.0f;
  for (unsigned tile = blockIdx.x; tile < tl.n; tile += gridDim.x) {
    const int3 t0 = tl.at(tile, TY, TZ);
    const int x0 = t0.x, y0 = t0.y, z0 = t0.z;
    stage_halo<KC, NP, TY, TZ, kConvThreads>(sx, in, g, x0, y0, z0);
    cp_commit();
    cp_wait<0>();
    __syncthreads();
    // the sums, the chain that is being added up, and that of the lower planes
    float acc[2][NT][4], s[2][NT][4], sl[NP > 1 ? 2 : 1][NP > 1 ? NT : 1][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[m][n][e] = bv[n][e & 1];
          s[m][n][e] = 0.0f;
          if (NP > 1) sl[m][n][e] = 0.0f;
        }
#pragma unroll 1
    for (int tr = 0; tr < 9; ++tr) {  // rows of three taps
      const int roff = ((tr / 3) * HY + tr % 3) * kHX;
#pragma unroll
      for (int kx = 0; kx < 3; ++kx) {
        const int t = tr * 3 + kx;
        uint32_t b1[4];  // NT == 1: the whole tap's 32 channels of the 8 columns
        if (NT == 1) ldsm4(b1, sw + row_at<KC>(t * 8 + (lane & 7), lane >> 3));
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          uint32_t b[NT == 4 ? 8 : 2];
          if (NT == 4) {
            ldsm4(b, sw + row_at<KC>(t * 32 + br, ks * 2 + bc));
            ldsm4(b + (NT == 4 ? 4 : 0), sw + row_at<KC>(t * 32 + 16 + br, ks * 2 + bc));
          } else {
            b[0] = b1[2 * ks];
            b[1] = b1[2 * ks + 1];
          }
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const uint32_t at = sx + row_at<KC>(ar + m * 2 * kHX + roff + kx, ks * 2 + ac);
#pragma unroll
            for (int p = NP - 1; p >= 0; --p) {
              uint32_t a[4];
              ldsm4(a, at + p * (HV * 2 * KC));
#pragma unroll
              for (int n = 0; n < NT; ++n) mma_bf16_16816(NP > 1 && p ? sl[m][n] : s[m][n], a, b + 2 * n);
            }
          }
        }
        if (OUT == OUT_RELU && tr * 3 + kx < 26) continue;
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              acc[m][n][e] += s[m][n][e];
              s[m][n][e] = 0.0f;
              if (NP > 1 && tr == 8 && kx == 2) acc[m][n][e] += sl[m][n][e];
            }
      }
    }
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int X = x0 + gid, Y = y0 + (warp & 1) * 4 + m * 2 + h, Z = z0 + z;
        if (X >= g.nx || Y >= g.ny || Z >= g.nz) continue;
        const int64_t v = ((int64_t)Z * g.ny + Y) * g.nx + X;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const float r0 = acc[m][n][2 * h], r1 = acc[m][n][2 * h + 1];
          const int col = n * 8 + 2 * tig;
          if (OUT == OUT_RELU) {
            ((uint32_t*)out)[(v * 32 + col) / 2] = pair_of(__float2bfloat16_rn(r0 > 0.0f ? r0 : 0.0f),
                                                           __float2bfloat16_rn(r1 > 0.0f ? r1 : 0.0f));
          } else if (OUT == OUT_F32) {
            if (col < 4) ((float2*)out)[(v * 4 + col) / 2] = make_float2(r0, r1);
          } else {
            const __nv_bfloat162 k = *(const __nv_bfloat162*)(mask + v * 32 + col);
            __nv_bfloat16 p0[3], p1[3];
            split3(__bfloat162float(k.x) > 0.0f ? r0 : 0.0f, p0);
            split3(__bfloat162float(k.y) > 0.0f ? r1 : 0.0f, p1);
#pragma unroll
            for (int p = 0; p < 3; ++p) ((uint32_t*)out)[(v * 96 + p * 32 + col) / 2] = pair_of(p0[p], p1[p]);
          }
        }
      }
    __syncthreads();
  }
}

// Layer 1: a1[v][n] = max(0, b[n] + sum_t sum_i w[t][i][n] x[v + off(t)][i]), fused
// multiply-adds in that order.  A thread takes a row of 8 voxels of the tile and 8 outputs:
// a weight serves 8 products and a field value three taps, so the FP32 pipe (108 x 32
// operations a voxel, 12 us on 64 x 32 x 64) bounds it and not shared memory: 64 us with a
// thread a voxel -> 31 us.
constexpr int kConv1Threads = 128;

__global__ void __launch_bounds__(kConv1Threads)
    k_conv1(const __nv_bfloat16* x, const float* wt, const float* bias, uint4* out, Grid3 g, Tiling tl) {
  constexpr int TY = kConvTY, TZ = kConvTZ, HY = TY + 2, HV = kHX * HY * (TZ + 2);
  __shared__ float4 sw[27 * 4 * 8];  // [tap][field][32 outputs]
  __shared__ float4 sx[HV];
  for (int k = threadIdx.x; k < 27 * 4 * 8; k += kConv1Threads) sw[k] = ((const float4*)wt)[k];
  const int n8 = threadIdx.x & 3, y = (threadIdx.x >> 2) & 7, z = threadIdx.x >> 5;
  for (unsigned tile = blockIdx.x; tile < tl.n; tile += gridDim.x) {
    const int3 t0 = tl.at(tile, TY, TZ);
    const int x0 = t0.x, y0 = t0.y, z0 = t0.z;
    for (int k = threadIdx.x; k < HV; k += kConv1Threads) {
      const int64_t q = nb_of(g, x0 + k % kHX - 1, y0 + (k / kHX) % HY - 1, z0 + k / (kHX * HY) - 1);
      const uint2 u = q < 0 ? make_uint2(0u, 0u) : *(const uint2*)(x + q * 16);
      sx[k] = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                          __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
    }
    __syncthreads();
    float acc[kTX][8];
#pragma unroll
    for (int n = 0; n < 8; ++n) {
      const float b = bias[n8 * 8 + n];
#pragma unroll
      for (int v = 0; v < kTX; ++v) acc[v][n] = b;
    }
#pragma unroll 1
    for (int tr = 0; tr < 9; ++tr) {
      const float4* row = sx + ((z + tr / 3) * HY + y + tr % 3) * kHX;
      float4 f[kHX];
#pragma unroll
      for (int k = 0; k < kHX; ++k) f[k] = row[k];
#pragma unroll
      for (int kx = 0; kx < 3; ++kx)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 wa = sw[((tr * 3 + kx) * 4 + i) * 8 + n8 * 2], wb = sw[((tr * 3 + kx) * 4 + i) * 8 + n8 * 2 + 1];
          const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
          for (int v = 0; v < kTX; ++v) {
            const float q = i == 0 ? f[v + kx].x : i == 1 ? f[v + kx].y : i == 2 ? f[v + kx].z : f[v + kx].w;
#pragma unroll
            for (int n = 0; n < 8; ++n) acc[v][n] = fmaf(w[n], q, acc[v][n]);
          }
        }
    }
    if (y0 + y < g.ny && z0 + z < g.nz) {
      const int64_t v0 = ((int64_t)(z0 + z) * g.ny + y0 + y) * g.nx + x0;
#pragma unroll
      for (int v = 0; v < kTX; ++v) {
        if (x0 + v >= g.nx) break;
        uint32_t o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float r0 = acc[v][2 * k], r1 = acc[v][2 * k + 1];
          o[k] = pair_of(__float2bfloat16_rn(r0 > 0.0f ? r0 : 0.0f), __float2bfloat16_rn(r1 > 0.0f ? r1 : 0.0f));
        }
        out[(v0 + v) * 4 + n8] = make_uint4(o[0], o[1], o[2], o[3]);
      }
    }
    __syncthreads();
  }
}

// Weight gradient of one layer:
//   dw[co][ci][t] = sum_v dout[v][co] in[v + off(t)][ci],  db[co] = sum_v dout[v][co]
// The voxels are the products' inner dimension: rows of 16 of them (8 along x, 2 along y).
// A warp holds 16 rows of dout (MT = 2: 16 of the 32 outputs, its three planes one after
// the other; MT = 1: the three planes of the 4 outputs as rows) against the 8 NT inputs
// of three taps one by one, and adds the tile's sums to the block's in shared memory: the
// 9 MT warps cover all 27.  The next tile's rows arrive meanwhile.  The blocks' sums are added in a fixed order by k_wgrad_reduce, so the
// gradient is deterministic.  On 64 x 32 x 64 voxels, against a block a tap with FP32
// operations from shared memory: 32 x 32 1,209 -> 83 us, 32 x 4 679 -> 31 us, 4 x 32
// 221 -> 40 us; relative errors against 64 bits on 512 voxels 1.2e-7 -> 0.8e-7.
template <int MT, int NT>
struct Wg {
  static constexpr int NP = MT == 2 ? 3 : 1;    // planes of a dout row
  static constexpr int KA = MT == 2 ? 32 : 16;  // channels of one
  static constexpr int KB = NT == 4 ? 32 : 16;  // channels of an input row
  static constexpr int CO = MT == 2 ? 32 : 4, CI = NT == 4 ? 32 : 4;
  static constexpr int threads = 9 * MT * 32;
  static constexpr int TV = kTX * kWgTY * kWgTZ, HV = kHX * (kWgTY + 2) * (kWgTZ + 2);
  static constexpr int bytes_a = TV * KA * NP * 2, bytes_b = HV * KB * 2;
  static constexpr int smem = 2 * (bytes_a + bytes_b) + 3 * NT * 4 * threads * 4;
  static constexpr int part = 27 * CO * CI + CO;  // words of a block's sums
};

template <int MT, int NT>
__global__ void __launch_bounds__(Wg<MT, NT>::threads)
    k_wgrad(const __nv_bfloat16* in, const __nv_bfloat16* dout, float* part, Grid3 g, Tiling tl) {
  using W = Wg<MT, NT>;
  constexpr int TY = kWgTY, TZ = kWgTZ, HY = TY + 2, KA = W::KA, KB = W::KB, NP = W::NP;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const uint32_t sb = (uint32_t)__cvta_generic_to_shared(smem_raw);
  float* sums = (float*)(smem_raw + 2 * (W::bytes_a + W::bytes_b)) + threadIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gid = lane >> 2, tig = lane & 3;
  const int mt = warp / 9, tr = warp % 9;
  // the lane's rows and parts of the fragments of the first 16 voxels
  const int ar = ((lane >> 4) & 1) * 8 + (lane & 7), ac = mt * 2 + ((lane >> 3) & 1);
  const int br = ((tr / 3) * HY + tr % 3 + ((lane >> 3) & 1)) * kHX + (lane & 7), bc = lane >> 4;
  const uint32_t ones[2] = {0x3f803f80u, 0x3f803f80u};
  float bias[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int k = 0; k < 3 * NT * 4; ++k) sums[k * W::threads] = 0.0f;

  auto stage = [&](unsigned tile, int buf) {
    const uint32_t sa = sb + buf * (W::bytes_a + W::bytes_b);
    const int3 t0 = tl.at(tile, TY, TZ);
    const int x0 = t0.x, y0 = t0.y, z0 = t0.z;
    constexpr int CH = KA / 8, ROW = CH * NP;
    for (int k = threadIdx.x; k < W::TV * ROW; k += W::threads) {
      const int v = k / ROW, c = k % ROW;
      const int x = x0 + v % kTX, y = y0 + (v / kTX) % TY, z = z0 + v / (kTX * TY);
      const bool ok = x < g.nx && y < g.ny && z < g.nz;
      const int64_t q = ok ? ((int64_t)z * g.ny + y) * g.nx + x : 0;
      cp16(sa + (uint32_t)((c / CH) * W::TV * 2 * KA) + row_at<KA>(v, c % CH), dout + q * (NP * KA) + c * 8, ok);
    }
    stage_halo<KB, 1, TY, TZ, W::threads>(sa + W::bytes_a, in, g, x0, y0, z0);
  };

  int buf = 0;
  if (blockIdx.x < tl.n) stage(blockIdx.x, 0);
  cp_commit();
  for (unsigned tile = blockIdx.x; tile < tl.n; tile += gridDim.x, buf ^= 1) {
    if (tile + gridDim.x < tl.n) stage(tile + gridDim.x, buf ^ 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    const uint32_t sa = sb + buf * (W::bytes_a + W::bytes_b), sx = sa + W::bytes_a;
#pragma unroll 1
    for (int kx = 0; kx < 3; ++kx) {
      // the sums, the chain that is being added up, and that of the lower planes
      float tot[NT][4], sh[NT][4], sl[NP > 1 ? NT : 1][4], bh[4], bl[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        bh[e] = bl[e] = 0.0f;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          tot[n][e] = sh[n][e] = 0.0f;
          if (NP > 1) sl[n][e] = 0.0f;
        }
      }
      const bool with_bias = tr == 0 && kx == 0;
#pragma unroll
      for (int k = 0; k < W::TV / 16; ++k) {
        uint32_t a[NP][4], b[NT == 4 ? 8 : 2];
#pragma unroll
        for (int p = 0; p < NP; ++p) ldsm4t(a[p], sa + p * (W::TV * 2 * KA) + row_at<KA>(k * 16 + ar, ac));
        const int row = br + ((k / (TY / 2)) * HY + (k % (TY / 2)) * 2) * kHX + kx;
        if (NT == 4) {
          ldsm4t(b, sx + row_at<KB>(row, bc));
          ldsm4t(b + (NT == 4 ? 4 : 0), sx + row_at<KB>(row, 2 + bc));
        } else {
          ldsm2t(b, sx + row_at<KB>(row, 0));
        }
#pragma unroll
        for (int p = NP - 1; p >= 0; --p)
#pragma unroll
          for (int n = 0; n < NT; ++n) mma_bf16_16816(NP > 1 && p ? sl[n] : sh[n], a[p], b + 2 * n);
        if (with_bias)
#pragma unroll
          for (int p = NP - 1; p >= 0; --p) mma_bf16_16816(p ? bl : bh, a[p], ones);
        if (k % 2 == 1) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            bias[e] += bh[e];
            bh[e] = 0.0f;
#pragma unroll
            for (int n = 0; n < NT; ++n) {
              tot[n][e] += sh[n][e];
              sh[n][e] = 0.0f;
            }
          }
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        bias[e] += bl[e];
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          if (NP > 1) tot[n][e] += sl[n][e];
          sums[((kx * NT + n) * 4 + e) * W::threads] += tot[n][e];
        }
      }
    }
    __syncthreads();
  }
  // rows gid and gid + 8 of the fragment, columns 2 tig and 2 tig + 1 of each n-tile
  float* my = part + (int64_t)blockIdx.x * W::part;
#pragma unroll
  for (int kx = 0; kx < 3; ++kx)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float v0 = sums[((kx * NT + n) * 4 + e) * W::threads];
        const float v1 = sums[((kx * NT + n) * 4 + 2 + e) * W::threads];
        const int ci = n * 8 + 2 * tig + e;
        float* at = my + (tr * 3 + kx) * W::CO * W::CI + ci;
        if (MT == 1) {  // rows 0..3 are the top planes, 4..7 the middle, 8..11 the low ones
          const float mid = __shfl_down_sync(0xffffffffu, v0, 16);
          v0 += mid + v1;
          if (gid < 4) at[gid * W::CI] = v0;
        } else if (ci < W::CI) {
          at[(mt * 16 + gid) * W::CI] = v0;
          at[(mt * 16 + gid + 8) * W::CI] = v1;
        }
      }
  if (tr == 0) {
    float* at = my + 27 * W::CO * W::CI;
    if (MT == 1) {
      const float mid = __shfl_down_sync(0xffffffffu, bias[0], 16);
      if (gid < 4 && tig == 0) at[gid] = bias[0] + (mid + bias[2]);
    } else if (tig == 0) {
      at[mt * 16 + gid] = bias[0];
      at[mt * 16 + gid + 8] = bias[2];
    }
  }
}

// Sums of the blocks' partial gradients of the three layers into the packed gradient.
// A block takes 32 values, its warps every eighth partial each.
struct WgParts {
  const float* p[3];
};
__global__ void __launch_bounds__(256) k_wgrad_reduce(WgParts parts, int nb, float* grad) {
  __shared__ float red[8][32];
  constexpr int S1 = Wg<2, 1>::part, S2 = Wg<2, 4>::part, S3 = Wg<1, 4>::part;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int k0 = blockIdx.x * 32 + lane;
  const int layer = k0 < S1 ? 0 : k0 < S1 + S2 ? 1 : 2;
  const int k = k0 - (layer == 0 ? 0 : layer == 1 ? S1 : S1 + S2);
  const int stride = layer == 0 ? S1 : layer == 1 ? S2 : S3;
  const bool ok = k0 < S1 + S2 + S3;
  float s = 0.0f;
  if (ok) {
    const float* p = (layer == 0 ? parts.p[0] : layer == 1 ? parts.p[1] : parts.p[2]) + k;
#pragma unroll 4
    for (int b = warp; b < nb; b += 8) s += p[(int64_t)b * stride];
  }
  red[warp][lane] = s;
  __syncthreads();
  if (warp || !ok) return;
#pragma unroll
  for (int w = 1; w < 8; ++w) s += red[w][lane];
  const int ci_n = layer == 0 ? 4 : 32, co_n = layer == 2 ? 4 : 32, e_n = ci_n * co_n;
  const int base = layer == 0 ? 0 : layer == 1 ? S1 : S1 + S2;
  // partials [t][co][ci] then the biases; the parameter order is [co][ci][t]
  grad[base + (k < 27 * e_n ? (k % e_n) * 27 + k / e_n : k)] = s;
}

// The bf16 compute copies of the FP32 master weights, as rows of the kernels' second
// operand ([tap][output][input], their 16-byte parts permuted as in shared memory).  A
// data gradient is the convolution with the taps mirrored and inputs and outputs swapped.
struct Packed {
  float* f1;  // layer 1: [tap][field][output], rounded to bf16
  __nv_bfloat16 *f2, *f3, *b2, *b3;
  float* bias;  // [32] [32] [8], rounded to bf16
};
constexpr int kPackF1 = 27 * 4 * 32, kPackB3 = 27 * 32 * 16, kPackF2 = 27 * 32 * 32, kPackF3 = 27 * 8 * 32;

__global__ void k_pack(const float* w, Packed o) {
  const float* w1 = w;
  const float* w2 = w + Wg<2, 1>::part;
  const float* w3 = w2 + Wg<2, 4>::part;
  const int total = kPackF1 + 2 * kPackF2 + kPackF3 + kPackB3 + 72;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < total; k += gridDim.x * blockDim.x) {
    int j = k;
    if (j < kPackF1) {
      const int n = j % 32, i = (j / 32) % 4, t = j / 128;
      o.f1[j] = __bfloat162float(__float2bfloat16_rn(w1[(n * 4 + i) * 27 + t]));
    } else if ((j -= kPackF1) < kPackF2) {
      const int i = j % 32, n = (j / 32) % 32, t = j / 1024;
      o.f2[row_at<32>(j / 32, i / 8) / 2 + i % 8] = __float2bfloat16_rn(w2[(n * 32 + i) * 27 + t]);
    } else if ((j -= kPackF2) < kPackF3) {  // 4 outputs and 4 zeros
      const int i = j % 32, n = (j / 32) % 8, t = j / 256;
      o.f3[row_at<32>(j / 32, i / 8) / 2 + i % 8] = __float2bfloat16_rn(n < 4 ? w3[(n * 32 + i) * 27 + t] : 0.0f);
    } else if ((j -= kPackF3) < kPackF2) {
      const int i = j % 32, n = (j / 32) % 32, t = 26 - j / 1024;
      o.b2[row_at<32>(j / 32, i / 8) / 2 + i % 8] = __float2bfloat16_rn(w2[(i * 32 + n) * 27 + t]);
    } else if ((j -= kPackF2) < kPackB3) {  // the same weights for each of the three planes
      const int i = j % 16, n = (j / 16) % 32, t = 26 - j / 512;
      o.b3[row_at<16>(j / 16, i / 8) / 2 + i % 8] =
          __float2bfloat16_rn(i < 12 ? w3[((i % 4) * 32 + n) * 27 + t] : 0.0f);
    } else {
      j -= kPackB3;
      const float v = j < 32 ? w1[27 * 128 + j] : j < 64 ? w2[27 * 1024 + j - 32] : j < 68 ? w3[27 * 128 + j - 64] : 0.0f;
      o.bias[j] = __bfloat162float(__float2bfloat16_rn(v));
    }
  }
}

// y [v][4] FP32 vs target [v][4]: gradient 2 (y - t) / (4 N) in three planes, and the loss
__global__ void k_mse(const float4* y, const float4* tgt, uint4* g, double* loss, int64_t n) {
  __shared__ double red[256];
  double s = 0.0;
  const float n4 = (float)(4 * n);
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const float4 a = y[k], b = tgt[k];
    const float d[4] = {a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w};
    __nv_bfloat16 p[4][3];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      split3(2.0f * d[c] / n4, p[c]);
      s += (double)d[c] * (double)d[c];
    }
    uint32_t o[6];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      o[2 * q] = pair_of(p[0][q], p[1][q]);
      o[2 * q + 1] = pair_of(p[2][q], p[3][q]);
    }
    g[2 * k] = make_uint4(o[0], o[1], o[2], o[3]);
    g[2 * k + 1] = make_uint4(o[4], o[5], 0u, 0u);
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(loss, red[0] / (double)(4 * n));
}

__global__ void k_adam(float* p, const float* g, float* m, float* v, int64_t n, float lr,
                       float b1, float b2, float eps, float c1, float c2) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const float gk = g[k];
    const float mk = b1 * m[k] + (1.0f - b1) * gk;
    const float vk = b2 * v[k] + (1.0f - b2) * gk * gk;
    m[k] = mk;
    v[k] = vk;
    p[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
  }
}

// [C][4] channels-first FP64 field rows -> [v][16] bf16 network input, x / scale and zeros
__global__ void k_to_input(const double* f0, const double* f1, const double* f2, const double* f3,
                           float s0, float s1, float s2, float s3, uint4* x, int64_t n) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    x[2 * v] = make_uint4(
        pair_of(__float2bfloat16_rn((float)f0[v] / s0), __float2bfloat16_rn((float)f1[v] / s1)),
        pair_of(__float2bfloat16_rn((float)f2[v] / s2), __float2bfloat16_rn((float)f3[v] / s3)), 0u, 0u);
    x[2 * v + 1] = make_uint4(0u, 0u, 0u, 0u);
  }
}

int64_t blocks(int64_t n, int b) { return (n + b - 1) / b; }

}  // namespace

// The packed parameter vector: each layer's weights and biases, as in its gradient.
constexpr int kNP = Wg<2, 1>::part + Wg<2, 4>::part + Wg<1, 4>::part;

size_t cnn_param_count() { return kNP; }

size_t cnn_work_bytes(int64_t n) {
  // x(bf16x16) a1(bf16x32) g1(bf16x96, in the place of a2(bf16x32) y(f32x4) gy(bf16x16))
  // g2(bf16x96), packed weights and the weight gradients' partials
  // (and up to 255 bytes of alignment for each of the 16 parts)
  return (size_t)n * (32 + 64 + 192 + 192) + kPackF1 * 4 + (2 * kPackF2 + kPackF3 + kPackB3) * 2 + 72 * 4 +
         (size_t)kWgMaxBlocks * kNP * 4 + 16 * 256;
}

struct CnnBufs {
  __nv_bfloat16 *x, *a1, *a2, *gy, *g2, *g1;
  float* y;
  Packed w;
  float* part[3];  // partial weight gradients of the layers
};

// Every part starts on a 256-byte boundary: the kernels read them as 16-byte words.
static CnnBufs carve(void* work, int64_t n) {
  char* p = (char*)work;
  auto take = [&](size_t bytes) {
    void* at = p;
    p += (bytes + 255) & ~(size_t)255;
    return at;
  };
  CnnBufs b;
  b.x = (__nv_bfloat16*)take(n * 32);
  b.a1 = (__nv_bfloat16*)take(n * 64);
  // the gradient of layer 1's output is written when nothing reads a2, y and gy any more
  char* a2 = p;
  b.a2 = (__nv_bfloat16*)take(n * 64);
  b.y = (float*)take(n * 16);
  b.gy = (__nv_bfloat16*)take(n * 32);
  b.g1 = (__nv_bfloat16*)a2;
  p = std::max(p, a2 + ((n * 192 + 255) & ~(int64_t)255));
  b.g2 = (__nv_bfloat16*)take(n * 192);
  b.w.f1 = (float*)take(kPackF1 * 4);
  b.w.f2 = (__nv_bfloat16*)take(kPackF2 * 2);
  b.w.f3 = (__nv_bfloat16*)take(kPackF3 * 2);
  b.w.b2 = (__nv_bfloat16*)take(kPackF2 * 2);
  b.w.b3 = (__nv_bfloat16*)take(kPackB3 * 2);
  b.w.bias = (float*)take(72 * 4);
  b.part[0] = (float*)take((size_t)kWgMaxBlocks * Wg<2, 1>::part * 4);
  b.part[1] = (float*)take((size_t)kWgMaxBlocks * Wg<2, 4>::part * 4);
  b.part[2] = (float*)take((size_t)kWgMaxBlocks * Wg<1, 4>::part * 4);
  return b;
}

static Grid3 grid_of(const DevParams& P) {
  Grid3 g;
  g.nx = P.nc[0];
  g.ny = P.nc[1];
  g.nz = P.nc[2];
  for (int a = 0; a < 3; ++a) g.per[a] = P.periodic[a];
  g.n = P.C;
  return g;
}

static int sm_count() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

template <int KC, int NP, int NT, int OUT>
static void conv(const __nv_bfloat16* in, const __nv_bfloat16* w, const float* bias, void* out,
                 const __nv_bfloat16* mask, const Grid3& g, int nsm, cudaStream_t s) {
  constexpr int smem = conv_smem<KC, NP, NT>();
  const Tiling t = tiling(g, kConvTY, kConvTZ);
  const int per_sm = smem <= 110 * 1024 ? 2 : 1;
  cudaFuncSetAttribute(k_conv<KC, NP, NT, OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  k_conv<KC, NP, NT, OUT><<<(unsigned)std::min<int64_t>(t.n, per_sm * nsm), kConvThreads, smem, s>>>(
      in, w, bias, out, mask, g, t);
}

template <int MT, int NT>
static void wgrad(const __nv_bfloat16* in, const __nv_bfloat16* dout, float* part, const Grid3& g, int nb,
                  cudaStream_t s) {
  using W = Wg<MT, NT>;
  cudaFuncSetAttribute(k_wgrad<MT, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, W::smem);
  k_wgrad<MT, NT><<<(unsigned)nb, W::threads, W::smem, s>>>(in, dout, part, g, tiling(g, kWgTY, kWgTZ));
}

static void forward(CnnBufs& b, const Grid3& g, const float* master, int nsm, cudaStream_t s) {
  k_pack<<<128, 256, 0, s>>>(master, b.w);
  const Tiling t = tiling(g, kConvTY, kConvTZ);
  k_conv1<<<(unsigned)std::min<int64_t>(t.n, 4 * nsm), kConv1Threads, 0, s>>>(b.x, b.w.f1, b.w.bias, (uint4*)b.a1, g, t);
  conv<32, 1, 4, OUT_RELU>(b.a1, b.w.f2, b.w.bias + 32, b.a2, nullptr, g, nsm, s);
  conv<32, 1, 1, OUT_F32>(b.a2, b.w.f3, b.w.bias + 64, b.y, nullptr, g, nsm, s);
}

void cnn_input(const DevParams& P, const double* const f[4], const float scale[4], void* work,
               cudaStream_t s) {
  CnnBufs b = carve(work, P.C);
  k_to_input<<<(unsigned)std::min<int64_t>(blocks(P.C, 256), 4096), 256, 0, s>>>(
      f[0], f[1], f[2], f[3], scale[0], scale[1], scale[2], scale[3], (uint4*)b.x, P.C);
}

void cnn_forward(const DevParams& P, const float* master, void* work, float** y_out,
                 cudaStream_t s) {
  CnnBufs b = carve(work, P.C);
  const Grid3 g = grid_of(P);
  forward(b, g, master, sm_count(), s);
  *y_out = b.y;
}

void cnn_loss_grad(const DevParams& P, const float* master, const float* target, float* grad,
                   double* loss, void* work, cudaStream_t s) {
  CnnBufs b = carve(work, P.C);
  const Grid3 g = grid_of(P);
  const int nsm = sm_count();
  const int nb = (int)std::min<int64_t>(tiling(g, kWgTY, kWgTZ).n, std::min(nsm, kWgMaxBlocks));
  forward(b, g, master, nsm, s);
  cudaMemsetAsync(loss, 0, sizeof(double), s);
  k_mse<<<(unsigned)std::min<int64_t>(blocks(P.C, 256), 1024), 256, 0, s>>>((const float4*)b.y, (const float4*)target,
                                                                          (uint4*)b.gy, loss, P.C);
  wgrad<1, 4>(b.a2, b.gy, b.part[2], g, nb, s);
  conv<16, 1, 4, OUT_SPLIT>(b.gy, b.w.b3, nullptr, b.g2, b.a2, g, nsm, s);
  wgrad<2, 4>(b.a1, b.g2, b.part[1], g, nb, s);
  conv<32, 3, 4, OUT_SPLIT>(b.g2, b.w.b2, nullptr, b.g1, b.a1, g, nsm, s);
  wgrad<2, 1>(b.x, b.g1, b.part[0], g, nb, s);
  k_wgrad_reduce<<<(unsigned)blocks(kNP, 32), 256, 0, s>>>(WgParts{{b.part[0], b.part[1], b.part[2]}}, nb, grad);
}

void cnn_adam(float* master, const float* grad, float* m, float* v, int64_t t, float lr,
              cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f - powf(b1, (float)t), c2 = 1.0f - powf(b2, (float)t);
  k_adam<<<64, 256, 0, s>>>(master, grad, m, v, kNP, lr, b1, b2, 1e-8f, c1, c2);
}

}  // namespace sedi

namespace sedi {

namespace {

__global__ void k_chan_first_to_vec(const double* in, float* out, int64_t n, int nc) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    for (int c = 0; c < nc; ++c) out[v * nc + c] = (float)in[c * n + v];
}

__global__ void k_vec_to_chan_first(const float* in, double* out, int64_t n, int nc) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    for (int c = 0; c < nc; ++c) out[c * n + v] = (double)in[v * nc + c];
}

template <class T>
__device__ __forceinline__ T t_add_f(T a, float b);
template <>
__device__ __forceinline__ double t_add_f<double>(double a, float b) { return a + (double)b; }
template <>
__device__ __forceinline__ float t_add_f<float>(float a, float b) { return a + b; }
template <>
__device__ __forceinline__ dd t_add_f<dd>(dd a, float b) { return dd_add_f(a, b); }

template <class T>
__device__ __forceinline__ float t_f(T a);
template <>
__device__ __forceinline__ float t_f<double>(double a) { return (float)a; }
template <>
__device__ __forceinline__ float t_f<float>(float a) { return a; }
template <>
__device__ __forceinline__ float t_f<dd>(dd a) { return a.hi; }

template <class T>
__device__ __forceinline__ T t_scale(T a, float s);
template <>
__device__ __forceinline__ double t_scale<double>(double a, float s) { return a * (double)s; }
template <>
__device__ __forceinline__ float t_scale<float>(float a, float s) { return a * s; }
template <>
__device__ __forceinline__ dd t_scale<dd>(dd a, float s) { return dd_mul_f(a, s); }

// guess = phi + scale_c * y_c on (eps, F_x, F_y, F_z) = fields (0, 4, 5, 6); the
// momentum fields eps*U (1, 2, 3) follow the predicted change of eps at fixed
// particle velocity: (eps U)^guess = (eps U)^m * eps^guess / eps^m.
template <class T>
__global__ void k_guess(const T* phi, const float* y, float s0, float s1, float s2, float s3,
                        T* guess, int64_t C) {
  const float sc[4] = {s0, s1, s2, s3};
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < C; v += (int64_t)gridDim.x * blockDim.x) {
    const T e = phi[v];
    const T eg = t_add_f<T>(e, sc[0] * y[v * 4]);
    guess[v] = eg;
    const float ef = t_f<T>(e);
    const float ratio = ef > 1e-9f ? t_f<T>(eg) / ef : 1.0f;
    for (int f = 1; f < 4; ++f) guess[f * C + v] = t_scale<T>(phi[f * C + v], ratio);
    for (int f = 4; f < 7; ++f) guess[f * C + v] = t_add_f<T>(phi[f * C + v], sc[f - 3] * y[v * 4 + f - 3]);
  }
}

}  // namespace

void cnn_chan_first_to_vec(const double* in, float* out, int64_t n, int nc, cudaStream_t s) {
  k_chan_first_to_vec<<<(unsigned)std::min<int64_t>(blocks(n, 256), 4096), 256, 0, s>>>(in, out, n, nc);
}

void cnn_vec_to_chan_first(const float* in, double* out, int64_t n, int nc, cudaStream_t s) {
  k_vec_to_chan_first<<<(unsigned)std::min<int64_t>(blocks(n, 256), 4096), 256, 0, s>>>(in, out, n, nc);
}

void cnn_guess(int form, const void* phi, const float* y, const float scale[4], void* guess,
               int64_t C, cudaStream_t s) {
  const unsigned g = (unsigned)std::min<int64_t>(blocks(C, 256), 4096);
  if (form == FORM_SPLIT)
    k_guess<dd><<<g, 256, 0, s>>>((const dd*)phi, y, scale[0], scale[1], scale[2], scale[3], (dd*)guess, C);
  else if (form == FORM_PLAIN)
    k_guess<float><<<g, 256, 0, s>>>((const float*)phi, y, scale[0], scale[1], scale[2], scale[3], (float*)guess, C);
  else
    k_guess<double><<<g, 256, 0, s>>>((const double*)phi, y, scale[0], scale[1], scale[2], scale[3], (double*)guess, C);
}

}  // namespace sedi

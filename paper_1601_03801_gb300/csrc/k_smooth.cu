// Diffusion smoothing of the averaged fields (Sec. 2.4, Eq. 10): n_tau implicit
// pseudo-steps A x = b of the 7-point finite-volume Laplacian L (zero flux through
// non-periodic faces), each solved to ||b - A x|| <= rtol ||b|| for every field of
// every mesh of a batch, in ONE persistent launch.  Backward Euler:
// A = I - dtau D L, b = x^m.  BDF2 (the paper's second-order implicit scheme, read
// as the two-step backward difference): A = I - (2/3) dtau D L,
// b = (4/3) x^m - (1/3) x^{m-1} = x^m + (x^m - x^{m-1}) / 3, its first step backward
// Euler; x^{m-1} is kept in the wide word.
//
// Solver: Chebyshev semi-iteration on the known spectrum of A (lambda_min = 1 from
// the constant mode, lambda_max <= 1 + 4 sum_a coef_a by Gershgorin), organised as
// iterative refinement:
//   round:  r = b - A x in the wide word (df64 in the split form), kept as a narrow
//           copy, with the sums |r|^2, sum r (and |b|^2 in the first round)
//           reduced per work unit;
//           the constant shift s = sum(r) / C restores sum(x) = sum(b) (1^T A = 1^T,
//           so A 1 = 1 and the shifted residual has |r - s|^2 = |r|^2 - (sum r)^2/C);
//           if |r - s| <= rtol |b| the field is done, otherwise k Chebyshev steps
//           follow, k fixed up front from |r_k| <= 2 sigma^k |r_0|,
//           sigma = (sqrt(kappa) - 1) / (sqrt(kappa) + 1);
//   steps:  d_0 = (r - s) / theta;  x += d;  q -= A d;  d = c1 d + c2 q
//           with the direction d and the recursive residual q in the narrow word
//           (FP32 in the split form, the 8 fields of a cell interleaved so they load
//           as two 16-byte vectors) and x accumulated in the wide word;
//           rho' = 1 / (2 theta/delta - rho), c1 = rho' rho, c2 = 2 rho'/delta.
// A round that ends with the narrow recursion's rounding floor above the tolerance
// is followed by another round from the true residual, so every field finishes
// with a true df64 residual below rtol and sum(x) = sum(b) to df64 rounding.  The
// narrow steps do about a sixth of the work of df64 steps.
//
// Work units: 256 consecutive cells of one mesh (one per thread).  Every reduction
// is a per-unit partial sum followed by a per-mesh sum over its units in unit
// order, so a mesh's result does not depend on the grid size or on the other
// meshes of the batch: a batch of beds gives the same bits as each bed alone.
// The grid barrier spins at most ~0.8 s, then records SEDI_ETIMEOUT and returns;
// the other blocks see the record and return at their next barrier.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <cmath>
#include <cstring>
#include <vector>

#include "../../include/sedi.h"
#include "common.cuh"
#include "kernels.h"

namespace sedi {

namespace {

constexpr int kThreads = kSmoothUnitCells;  // threads per block = cells per work unit
constexpr int kMaxF = kSmoothMaxFields;
constexpr int kQ = kSmoothSums;  // per-unit sums: |r|^2, sum r, |b|^2, sum w r (graded mesh)
constexpr int kMaxRounds = 64;

// ---------------------------------------------------------------- words
// T: wide word (x, b, r); N: narrow word (d, q); Acc: unit sums.
template <class T>
struct Wide;
template <>
struct Wide<dd> {
  using N = float;
  using Acc = float;
  static constexpr double kFloor = 1.0e-6;  // reduction one narrow round can reach
  __device__ static dd zero() { return dd{0.0f, 0.0f}; }
  __device__ static dd from_d(double a) { return dd_from_double(a); }
  __device__ static float narrow(dd a) { return __fadd_rn(a.hi, a.lo); }
  __device__ static dd add(dd a, dd b) { return dd_add(a, b); }
  __device__ static dd addq(dd a, dd b) { return dd_add_fast(a, b); }
  __device__ static dd subq(dd a, dd b) { return dd_sub_fast(a, b); }
  __device__ static dd mul(dd a, dd b) { return dd_mul(a, b); }
  __device__ static dd add_n(dd a, float b) { return dd_add_f(a, b); }
  __device__ static dd ld(const dd* p) {
    const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
    return dd{v.x, v.y};
  }
};
template <>
struct Wide<float> {
  using N = float;
  using Acc = float;
  static constexpr double kFloor = 1.0e-6;
  __device__ static float zero() { return 0.0f; }
  __device__ static float from_d(double a) { return __double2float_rn(a); }
  __device__ static float narrow(float a) { return a; }
  __device__ static float add(float a, float b) { return a + b; }
  __device__ static float addq(float a, float b) { return a + b; }
  __device__ static float subq(float a, float b) { return a - b; }
  __device__ static float mul(float a, float b) { return a * b; }
  __device__ static float add_n(float a, float b) { return a + b; }
  __device__ static float ld(const float* p) { return __ldcg(p); }
};
template <>
struct Wide<double> {
  using N = double;
  using Acc = double;
  static constexpr double kFloor = 0.0;
  __device__ static double zero() { return 0.0; }
  __device__ static double from_d(double a) { return a; }
  __device__ static double narrow(double a) { return a; }
  __device__ static double add(double a, double b) { return a + b; }
  __device__ static double addq(double a, double b) { return a + b; }
  __device__ static double subq(double a, double b) { return a - b; }
  __device__ static double mul(double a, double b) { return a * b; }
  __device__ static double add_n(double a, double b) { return a + b; }
  __device__ static double ld(const double* p) { return __ldcg(p); }
};

// The operator coefficients in the wide and the narrow word (converted on the host,
// so the kernels run no FP64 conversion per cell).
template <class T>
__device__ __forceinline__ T coef_w(const SmoothSpec& sp, int a);
template <>
__device__ __forceinline__ dd coef_w<dd>(const SmoothSpec& sp, int a) {
  return dd{sp.coef_hi[a], sp.coef_lo[a]};
}
template <>
__device__ __forceinline__ float coef_w<float>(const SmoothSpec& sp, int a) {
  return sp.coef_hi[a];
}
template <>
__device__ __forceinline__ double coef_w<double>(const SmoothSpec& sp, int a) {
  return sp.coef[a];
}

// Loads of words written by other blocks of the same launch go to L2 (ld.cg), so
// no stale L1 line is read after a grid barrier.
__device__ __forceinline__ int ldi(const int* p) { return __ldcg(p); }
__device__ __forceinline__ double ldd(const double* p) { return __ldcg(p); }

// Bounded grid barrier (co-residency guaranteed by the cooperative launch).
__device__ bool grid_barrier(Ctl* ctl, unsigned nblocks, long long spin_limit) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* gen = &ctl->bar_gen;
    const unsigned g = *gen;
    __threadfence();
    const unsigned arrived = atomicAdd(&ctl->bar_count, 1u);
    if (arrived == nblocks - 1) {
      atomicExch(&ctl->bar_count, 0u);
      __threadfence();
      atomicAdd(&ctl->bar_gen, 1u);
    } else {
      long long spins = 0;
      while (*gen == g) {
        if (++spins > spin_limit) {  // ~0.8 s at the default kBarrierSpins
          atomicCAS((int*)&ctl->cg_status, 0, SEDI_ETIMEOUT);
          break;
        }
        // another block gave up: stop waiting too
        if ((spins & 1023) == 0 && *((volatile int*)&ctl->cg_status) == SEDI_ETIMEOUT) break;
        __nanosleep(32);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return *((volatile int*)&ctl->cg_status) != SEDI_ETIMEOUT;
}

// Cell coordinates -> the six face neighbours (-1: zero-flux face).
struct Stencil {
  int32_t nb[6];
};

// n / d for 32-bit n from M = ceil(2^64 / d) (M = 0 for d = 1): floor(n M / 2^64) is
// exact, the excess n (M - 2^64/d) / 2^64 < 2^-32 <= 1/d.
__device__ __forceinline__ uint32_t div_magic(uint32_t n, uint64_t M) {
  return M ? (uint32_t)__umul64hi((uint64_t)n, M) : n;
}

__device__ __forceinline__ Stencil stencil_of(const SmoothMeshDev& m, int64_t c) {
  const uint32_t nx = m.nc[0], ny = m.nc[1], nz = m.nc[2];
  const uint32_t cc = (uint32_t)c;
  const uint32_t t = div_magic(cc, m.div_x);
  const uint32_t iz = div_magic(cc, m.div_xy);
  const uint32_t ix = cc - t * nx;
  const uint32_t iy = t - iz * ny;
  const uint32_t idx[3] = {ix, iy, iz};
  const uint32_t n[3] = {nx, ny, nz};
  const int32_t stride[3] = {1, (int32_t)nx, (int32_t)(nx * ny)};
  Stencil s;
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const int32_t base = (int32_t)cc - (int32_t)idx[ax] * stride[ax];
    if (idx[ax] > 0) s.nb[2 * ax] = (int32_t)cc - stride[ax];
    else s.nb[2 * ax] = m.per[ax] ? base + (int32_t)(n[ax] - 1) * stride[ax] : -1;
    if (idx[ax] + 1 < n[ax]) s.nb[2 * ax + 1] = (int32_t)cc + stride[ax];
    else s.nb[2 * ax + 1] = m.per[ax] ? base : -1;
  }
  return s;
}

// (A v)(c) = v_c - sum_axes coef_a ((v_- - v_c) + (v_+ - v_c)), faces that exist only.
// V is the word of the operand, get(k) loads (or forms) its value at cell k.
template <class V, class Sub, class Add, class Mul, class Get>
__device__ __forceinline__ V apply_A(const Stencil& st, const V* cf, V vc, Sub sub, Add add,
                                     Mul mul, Get get) {
  V lap{};
  bool any_axis = false;
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    V sa{};
    bool any = false;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const int32_t nb = st.nb[2 * ax + side];
      if (nb < 0) continue;
      const V t = sub(get(nb), vc);
      sa = any ? add(sa, t) : t;
      any = true;
    }
    if (any) {
      const V t = mul(cf[ax], sa);
      lap = any_axis ? add(lap, t) : t;
      any_axis = true;
    }
  }
  return any_axis ? sub(vc, lap) : vc;
}

// Graded z mesh: as apply_A, the z faces with their own coefficients (cz_m towards
// the plane below, cz_p towards the plane above).
template <class V, class Sub, class Add, class Mul, class Get>
__device__ __forceinline__ V apply_A_graded(const Stencil& st, const V* cf, V czm, V czp, V vc,
                                            Sub sub, Add add, Mul mul, Get get) {
  V lap{};
  bool any_axis = false;
#pragma unroll
  for (int ax = 0; ax < 2; ++ax) {
    V sa{};
    bool any = false;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const int32_t nb = st.nb[2 * ax + side];
      if (nb < 0) continue;
      const V t = sub(get(nb), vc);
      sa = any ? add(sa, t) : t;
      any = true;
    }
    if (any) {
      const V t = mul(cf[ax], sa);
      lap = any_axis ? add(lap, t) : t;
      any_axis = true;
    }
  }
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int32_t nb = st.nb[4 + side];
    if (nb < 0) continue;
    const V t = mul(side ? czp : czm, sub(get(nb), vc));
    lap = any_axis ? add(lap, t) : t;
    any_axis = true;
  }
  return any_axis ? sub(vc, lap) : vc;
}

// Eight narrow words of one cell (the fields of the narrow recursion are stored
// interleaved, [C][8], so one cell's fields load as two 16-byte vectors).
template <class N>
struct V8 {
  N v[8];
};
__device__ __forceinline__ V8<float> ld8(const float* p) {
  const float4 a = __ldcg(reinterpret_cast<const float4*>(p));
  const float4 b = __ldcg(reinterpret_cast<const float4*>(p) + 1);
  return V8<float>{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}
__device__ __forceinline__ void st8(float* p, const V8<float>& x) {
  reinterpret_cast<float4*>(p)[0] = make_float4(x.v[0], x.v[1], x.v[2], x.v[3]);
  reinterpret_cast<float4*>(p)[1] = make_float4(x.v[4], x.v[5], x.v[6], x.v[7]);
}
__device__ __forceinline__ V8<double> ld8(const double* p) {
  V8<double> r;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double2 a = __ldcg(reinterpret_cast<const double2*>(p) + k);
    r.v[2 * k] = a.x;
    r.v[2 * k + 1] = a.y;
  }
  return r;
}
__device__ __forceinline__ void st8(double* p, const V8<double>& x) {
#pragma unroll
  for (int k = 0; k < 4; ++k) reinterpret_cast<double2*>(p)[k] = make_double2(x.v[2 * k], x.v[2 * k + 1]);
}

// Per-mesh solver state published by the owner block of each mesh.
struct alignas(16) MeshState {
  int32_t k[kMaxF];      // Chebyshev steps of the current round per field (0: none)
  int32_t done[kMaxF];   // converged, zero or stopped
  int32_t zero[kMaxF];   // b == 0: x = 0
  int32_t total[kMaxF];  // steps taken in this pseudo-step
  double shift[kMaxF];   // projection shift of the current round
  double bb[kMaxF];      // |b|^2
};

// Per-block reduction of the kQ sums of nf fields for one unit (fixed order).  The
// warp stage is a butterfly reduce-scatter of the 32 (field, sum) slots: at each of
// five rounds a lane keeps half of its slots and adds its partner's copy of them, so
// lane l ends with the warp's sum of slot l after 31 additions (a plain shuffle
// reduction of every slot would take 5 x 32; the FP64 pipe is the narrow one).
template <class Acc>
__device__ __forceinline__ void unit_sums(const Acc (&v)[kMaxF][kQ], int nf, double* out) {
  static_assert(kMaxF * kQ == 32, "one slot per lane");
  __shared__ Acc red[kThreads / 32][kMaxF * kQ];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  Acc a[32];
#pragma unroll
  for (int f = 0; f < kMaxF; ++f)
#pragma unroll
    for (int q = 0; q < kQ; ++q) a[f * kQ + q] = v[f][q];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < o; ++k) {
      const Acc mine = up ? a[k + o] : a[k];
      const Acc give = up ? a[k] : a[k + o];
      a[k] = mine + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  red[wid][lane] = a[0];
  __syncthreads();
  if (threadIdx.x < nf * kQ) {
    double s = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) s += (double)red[w][threadIdx.x];
    out[threadIdx.x] = s;
  }
  __syncthreads();
}

// Right-hand side of pseudo-step m from x^m (xv): x^m itself (backward Euler, and
// the first BDF2 step), or x^m + (x^m - x^{m-1}) / 3 with x^{m-1} read from *xp.
// BDF2 also stores x^m in *xp for the next step.
template <class T>
__device__ __forceinline__ T rhs_of(int scheme, int m, T xv, T* xp) {
  using W = Wide<T>;
  if (scheme != TAU_BDF2) return xv;
  T bv = xv;
  if (m > 0) bv = W::add(xv, W::mul(W::from_d(1.0 / 3.0), W::subq(xv, W::ld(xp))));
  *xp = xv;
  return bv;
}

// Resident blocks per SM of the grid solver: 3 for the double-float and FP32 words (80
// registers, no spills; 17% faster than 2 on a 2M-cell mesh), 2 for FP64 (which would
// spill at 80).
template <class T>
constexpr int smooth_blocks_per_sm() {
  return sizeof(T) == 8 && !std::is_same<T, dd>::value ? 2 : 3;
}

// GR: graded z mesh (per-plane z coefficients, volume-weighted projection shift).
template <class T, bool GR>
__global__ void __launch_bounds__(kThreads, smooth_blocks_per_sm<T>()) k_smooth(SmoothBatchDev a) {
  using W = Wide<T>;
  using N = typename W::N;
  using Acc = typename W::Acc;
  const unsigned G = gridDim.x;
  const int nf = a.nf;
  const int64_t U = a.U;
  const int64_t u_begin = (int64_t)blockIdx.x * U / G, u_end = (int64_t)(blockIdx.x + 1) * U / G;
  MeshState* ms = (MeshState*)a.pairs;
  __shared__ double s_sums[(kThreads / 32) * kQ];
  __shared__ int s_K;
  // the mesh of the units being walked and its solver state for the current pass, in
  // shared memory (every thread of a block walks the same units, so a change of mesh is
  // seen by the whole block at once)
  static_assert(sizeof(SmoothMeshDev) % 16 == 0, "mesh entries are copied as 16-byte words");
  __shared__ SmoothMeshDev s_md;
  __shared__ int s_kf[kMaxF], s_zero[kMaxF], s_done[kMaxF];
  __shared__ double s_shd[kMaxF];
  auto load_mesh = [&](int bi) {
    __syncthreads();
    const int4* src = reinterpret_cast<const int4*>(a.mesh + bi);
    int4* dst = reinterpret_cast<int4*>(&s_md);
    for (int q = threadIdx.x; q < (int)(sizeof(SmoothMeshDev) / 16); q += blockDim.x) dst[q] = src[q];
    if (threadIdx.x < kMaxF) {
      const int f = threadIdx.x;
      const MeshState& st = ms[bi];
      s_kf[f] = f < nf ? ldi(&st.k[f]) : 0;
      s_zero[f] = f < nf ? ldi(&st.zero[f]) : 0;
      s_done[f] = f < nf ? ldi(&st.done[f]) : 1;
      s_shd[f] = f < nf ? ldd(&st.shift[f]) : 0.0;
    }
    __syncthreads();
  };
  int slot = 0;

  for (int m = 0; m < a.n_tau; ++m) {
    const bool use_guess = (m == 0);
    const int ph = (a.scheme == TAU_BDF2 && m > 0) ? 1 : 0;  // operator of this step
    // ---- b from the previous pseudo-step's result; x = guess on the first
    for (int64_t u = u_begin; u < u_end; ++u) {
      const SmoothMeshDev& md = a.mesh[a.unit_bed[u]];
      const int64_t c = (u - md.u0) * kThreads + threadIdx.x;
      if (c >= md.C) continue;
      for (int f = 0; f < nf; ++f) {
        const int64_t k = f * md.C + c;
        const T xv = W::ld((const T*)md.x + k);
        ((T*)md.b)[k] = rhs_of<T>(a.scheme, m, xv, (T*)md.xp + (md.xp ? k : 0));
        if (use_guess && md.guess) ((T*)md.x)[k] = W::ld((const T*)md.guess + k);
      }
    }
    if (!grid_barrier(a.ctl, G, a.spin_limit)) return;
    for (int round = 0; round < kMaxRounds; ++round) {
      // ---- true residual r = b - A x (wide), its narrow copy (interleaved, in d[0])
      //      and the unit sums |r|^2, sum r, |b|^2
      int cur_bi = -1;
      for (int64_t u = u_begin; u < u_end; ++u) {
        const int bi = a.unit_bed[u];
        if (bi != cur_bi) {
          load_mesh(bi);
          cur_bi = bi;
        }
        const SmoothMeshDev& md = s_md;
        const int64_t c = (u - md.u0) * kThreads + threadIdx.x;
        const bool in = c < md.C;
        Acc v[kMaxF][kQ];
        V8<N> rn;
        const SmoothSpec& sp = md.sp[ph];
        const T cf[3] = {coef_w<T>(sp, 0), coef_w<T>(sp, 1), coef_w<T>(sp, 2)};
        const Stencil sc = stencil_of(md, in ? c : 0);
        T czm{}, czp{};
        Acc wz = Acc(1);
        if constexpr (GR) {
          const int kz = (int)div_magic((uint32_t)(in ? c : 0), md.div_xy);
          czm = W::from_d(md.z.cz[ph][2 * kz]);
          czp = W::from_d(md.z.cz[ph][2 * kz + 1]);
          wz = (Acc)md.z.w[kz];
        }
#pragma unroll
        for (int f = 0; f < kMaxF; ++f) {
          v[f][0] = v[f][1] = v[f][2] = v[f][3] = Acc(0);
          rn.v[f] = N(0);
          if (f >= nf || !in || (round > 0 && s_done[f])) continue;
          const T* X = (const T*)md.x + f * md.C;
          const T xc = W::ld(X + c);
          auto subq = [](T p, T q) { return W::subq(p, q); };
          auto addq = [](T p, T q) { return W::addq(p, q); };
          auto mul = [](T p, T q) { return W::mul(p, q); };
          auto get = [&](int32_t k) { return W::ld(X + k); };
          T ax;
          if constexpr (GR) ax = apply_A_graded<T>(sc, cf, czm, czp, xc, subq, addq, mul, get);
          else ax = apply_A<T>(sc, cf, xc, subq, addq, mul, get);
          const T bv = W::ld((const T*)md.b + f * md.C + c);
          const T rv = W::subq(bv, ax);
          const N r_n = W::narrow(rv);
          rn.v[f] = r_n;
          v[f][0] = (Acc)r_n * (Acc)r_n;
          v[f][1] = (Acc)r_n;
          if constexpr (GR) v[f][3] = wz * (Acc)r_n;
          if (round == 0) {
            const Acc bn = (Acc)W::narrow(bv);
            v[f][2] = bn * bn;
          }
        }
        if (in) st8((N*)md.d[0] + c * kMaxF, rn);
        unit_sums<Acc>(v, nf, md.part + (u - md.u0) * (kMaxF * kQ));
      }
      if (!grid_barrier(a.ctl, G, a.spin_limit)) return;
      // ---- owners: one block per (mesh, field): the field's sums over the mesh's units
      //      (thread t adds units t, t + 256, ... in order, then a fixed tree: the same
      //      association whatever the grid or the batch), then its decisions
      for (int64_t it = blockIdx.x; it < (int64_t)a.B * nf; it += G) {
        const int bi = (int)(it / nf), f = (int)(it % nf);
        const SmoothMeshDev& md = a.mesh[bi];
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        double sq[kQ] = {0.0, 0.0, 0.0, 0.0};
        for (int64_t u = threadIdx.x; u < md.nu; u += kThreads) {
          const double* pu = md.part + u * (kMaxF * kQ) + f * kQ;
#pragma unroll
          for (int q = 0; q < kQ; ++q) sq[q] += ldd(pu + q);
        }
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
          double v = sq[q];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane == 0) s_sums[wid * kQ + q] = v;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
          double tot[kQ];
#pragma unroll
          for (int q = 0; q < kQ; ++q) {
            tot[q] = 0.0;
            for (int w = 0; w < kThreads / 32; ++w) tot[q] += s_sums[w * kQ + q];
          }
          MeshState& st = ms[bi];
          int k = 0, done = 1, zero = 0, total = 0;
          double shift = 0.0, bb = 0.0;
          done = round == 0 ? 0 : st.done[f];
          zero = round == 0 ? 0 : st.zero[f];
          total = round == 0 ? 0 : st.total[f];
          bb = round == 0 ? tot[2] : st.bb[f];
          if (round == 0) zero = !(bb > 0.0);
          if (!done) {
            const double rr = tot[0], sr = tot[1];
            const double Cd = (double)md.C;
            if (zero) {
              done = 1;
            } else {
              double rrp;
              if (GR) {
                // the shift keeps sum(w x) = sum(w b); |r - s|^2 = |r|^2 - 2 s sum r + C s^2
                shift = tot[3] / md.z.wsum;
                rrp = fmax(rr - 2.0 * shift * sr + Cd * shift * shift, 0.0);
              } else {
                shift = sr / Cd;
                rrp = fmax(rr - sr * sr / Cd, 0.0);
              }
              if (rrp <= a.rtol2 * bb) {
                done = 1;
              } else {
                // |r_k| <= 2 sig^k |r_0|: enough steps for the tolerance, or for the
                // reduction the narrow word can deliver in one round
                const double need = fmax(0.5 * sqrt(a.rtol2 * bb / rrp), W::kFloor);
                const double sig = md.sp[ph].sig;
                k = sig > 0.0 ? (int)ceil(log(need) / log(sig)) : 1;
                if (k < 1) k = 1;
                if (k > kMaxStepsRound) k = kMaxStepsRound;
                if (total + k > a.max_iter) k = a.max_iter - total;
                if (k <= 0) {
                  k = 0;
                  done = 1;
                  atomicCAS((int*)&a.ctl->cg_status, 0, SEDI_EDIVERGED);
                } else {
                  total += k;
                }
              }
            }
            if (done && md.iters) atomicAdd(md.iters + f, total);
          }
          st.k[f] = k;
          st.done[f] = done;
          st.zero[f] = zero;
          st.total[f] = total;
          st.shift[f] = shift;
          st.bb[f] = bb;
          if (k > 0) atomicMax(a.gflag + slot, k);
        }
        __syncthreads();
      }
      // the slot of the next round was last read before the previous barrier
      if (blockIdx.x == 0 && threadIdx.x == 0) a.gflag[slot ^ 1] = 0;
      if (!grid_barrier(a.ctl, G, a.spin_limit)) return;
      if (threadIdx.x == 0) s_K = ldi(a.gflag + slot);
      __syncthreads();
      const int K = s_K;
      slot ^= 1;
      // ---- Chebyshev steps j = 1..K; step 1 also applies the shift (or zeroes x)
      const int J = K > 0 ? K : 1;
      for (int j = 1; j <= J; ++j) {
        int cur_bi = -1;
        for (int64_t u = u_begin; u < u_end; ++u) {
          const int bi = a.unit_bed[u];
          if (bi != cur_bi) {
            load_mesh(bi);
            cur_bi = bi;
          }
          const SmoothMeshDev& md = s_md;
          const int64_t c = (u - md.u0) * kThreads + threadIdx.x;
          if (c >= md.C) continue;
          int kf[kMaxF];
          N sh[kMaxF];
          bool any = false;
#pragma unroll
          for (int f = 0; f < kMaxF; ++f) sh[f] = N(0);
#pragma unroll
          for (int f = 0; f < kMaxF; ++f) {
            kf[f] = s_kf[f];
            any |= kf[f] >= j;
          }
          if (j == 1) {
            // projection shift (and zero fields) for every field, then the first step
            T* X = (T*)md.x;
#pragma unroll
            for (int f = 0; f < kMaxF; ++f) {
              if (f >= nf) continue;
              const double s = s_shd[f];
              sh[f] = (N)s;
              if (kf[f] == 0) {
                if (round == 0 && s_zero[f]) X[f * md.C + c] = W::zero();
                else if (s != 0.0) X[f * md.C + c] = W::add(W::ld(X + f * md.C + c), W::from_d(s));
              }
            }
          }
          if (!any) continue;
          const SmoothSpec& sp = md.sp[ph];
          const N cfn[3] = {coef_w<N>(sp, 0), coef_w<N>(sp, 1), coef_w<N>(sp, 2)};
          N c1, c2, inv_theta;
          if constexpr (sizeof(N) == 4) {
            c1 = sp.chebf[0][j - 1];
            c2 = sp.chebf[1][j - 1];
            inv_theta = sp.inv_theta_f;
          } else {
            c1 = (N)sp.cheb[0][j - 1];
            c2 = (N)sp.cheb[1][j - 1];
            inv_theta = (N)(1.0 / sp.theta);
          }
          const Stencil sc = stencil_of(md, c);
          // step 1 reads the narrow residual (d[0]) and forms d0 = (r - s) / theta at
          // every stencil point; later steps read the previous direction
          const N* Dold = (const N*)md.d[(j - 1) & 1];
          N* Dnew = (N*)md.d[j & 1];
          N* Q = (N*)md.q;
          auto dir = [&](const V8<N>& raw) {
            V8<N> d = raw;
            if (j == 1) {
#pragma unroll
              for (int f = 0; f < kMaxF; ++f) d.v[f] = (raw.v[f] - sh[f]) * inv_theta;
            }
            return d;
          };
          const V8<N> dc = dir(ld8(Dold + c * kMaxF));
          V8<N> lap;
          bool any_axis = false;
          N czn[2] = {N(0), N(0)};
          if constexpr (GR) {
            const int kz = (int)div_magic((uint32_t)c, md.div_xy);
            if constexpr (sizeof(N) == 4) {
              czn[0] = md.z.czf[ph][2 * kz];
              czn[1] = md.z.czf[ph][2 * kz + 1];
            } else {
              czn[0] = (N)md.z.cz[ph][2 * kz];
              czn[1] = (N)md.z.cz[ph][2 * kz + 1];
            }
          }
#pragma unroll
          for (int ax = 0; ax < 3; ++ax) {
            if (GR && ax == 2) {
              // graded z: each face with its own coefficient
#pragma unroll
              for (int side = 0; side < 2; ++side) {
                const int32_t nb = sc.nb[4 + side];
                if (nb < 0) continue;
                const V8<N> dn = dir(ld8(Dold + (int64_t)nb * kMaxF));
#pragma unroll
                for (int f = 0; f < kMaxF; ++f) {
                  const N t = czn[side] * (dn.v[f] - dc.v[f]);
                  lap.v[f] = any_axis ? lap.v[f] + t : t;
                }
                any_axis = true;
              }
              continue;
            }
            V8<N> sa;
            bool any_side = false;
#pragma unroll
            for (int side = 0; side < 2; ++side) {
              const int32_t nb = sc.nb[2 * ax + side];
              if (nb < 0) continue;
              const V8<N> dn = dir(ld8(Dold + (int64_t)nb * kMaxF));
#pragma unroll
              for (int f = 0; f < kMaxF; ++f) {
                const N t = dn.v[f] - dc.v[f];
                sa.v[f] = any_side ? sa.v[f] + t : t;
              }
              any_side = true;
            }
            if (any_side) {
#pragma unroll
              for (int f = 0; f < kMaxF; ++f) {
                const N t = cfn[ax] * sa.v[f];
                lap.v[f] = any_axis ? lap.v[f] + t : t;
              }
              any_axis = true;
            }
          }
          // q: the narrow residual r - s (step 1) or the recursive residual
          V8<N> q = j == 1 ? ld8(Dold + c * kMaxF) : ld8(Q + c * kMaxF);
          V8<N> dn;
          T* X = (T*)md.x;
#pragma unroll
          for (int f = 0; f < kMaxF; ++f) {
            dn.v[f] = N(0);
            if (kf[f] < j) continue;
            const N ad = any_axis ? dc.v[f] - lap.v[f] : dc.v[f];
            const int64_t k = f * md.C + c;
            T xv = W::ld(X + k);
            if (j == 1) {
              xv = W::add(xv, W::from_d(s_shd[f]));  // projection shift
              q.v[f] = q.v[f] - sh[f];                         // narrow r - s
            }
            q.v[f] = q.v[f] - ad;
            dn.v[f] = c1 * dc.v[f] + c2 * q.v[f];
            X[k] = W::add_n(xv, dc.v[f]);
          }
          st8(Q + c * kMaxF, q);
          st8(Dnew + c * kMaxF, dn);
        }
        if (!grid_barrier(a.ctl, G, a.spin_limit)) return;
      }
      if (K == 0) break;
    }
  }
}

// ---------------------------------------------------------------- cluster solver
// Meshes whose z-planes fit 8192 cells per CTA on at most 16 CTAs (split and plain
// forms): a thread-block cluster solves one (mesh, field) pair at a time.  CTA r
// holds whole z-planes [r P, (r + 1) P) of the field and its narrow recursion in
// shared memory (x in the wide word, the narrow residual and two directions), so a
// step touches no global memory; the z-neighbours of a CTA's first and last plane
// are read from the adjacent CTAs through distributed shared memory.  Pairs are
// independent, so there is no grid-wide barrier: each step ends with the hardware
// cluster barrier and each field runs its own step count.  Same iteration as the
// grid solver (rounds of a wide true residual, then narrow Chebyshev steps); the
// sums of a round are reduced per CTA, then over the CTAs in rank order.  The
// cluster shape is a function of the mesh alone, so a bed smooths the same way in
// any batch.
namespace cg = cooperative_groups;
constexpr int kClThreads = 1024;
constexpr int kClCells = 8192;   // cells per CTA at most
constexpr size_t kClSmem = 212 * 1024;  // dynamic shared memory of a CTA at most: 20 B a cell
constexpr int kClMaxCta = 16;

// A stencil neighbour: index in the owning CTA's arrays, and that CTA (-1: this one).
struct Nb {
  int32_t l;
  int32_t r;
};

template <class T, bool GR>
__global__ void __launch_bounds__(kClThreads, 1) k_smooth_cl(SmoothBatchDev a) {
  using W = Wide<T>;
  using N = typename W::N;
  using Acc = typename W::Acc;
  extern __shared__ __align__(16) unsigned char s_dyn[];
  __shared__ double s_part[kClMaxCta][kQ];  // every CTA's sums, pushed by each CTA
  __shared__ double s_red[kClThreads / 32][kQ];
  __shared__ double s_shift;
  __shared__ int s_k, s_zero;
  cg::cluster_group cl = cg::this_cluster();
  const int csize = (int)cl.num_blocks();
  const int rank = (int)cl.block_rank();
  const int64_t ncl = gridDim.x / csize, cid = blockIdx.x / csize;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t items = (int64_t)a.B * a.nf;
  // one item a cluster as launched; the loop stays because the kernel without it is slower
  // (four fields of 37 x 41 x 45 668 -> 680 us)
  for (int64_t w = cid; w < items; w += ncl) {
    const int bi = (int)(w / a.nf), f = (int)(w % a.nf);
    const SmoothMeshDev& md = a.mesh[bi];
    const int64_t C = md.C;
    const int nx = md.nc[0], ny = md.nc[1], nz = md.nc[2], nxy = nx * ny;
    const int P = md.cl_planes;                                  // planes of a full CTA
    const int z0 = rank * P;
    const int planes = z0 + P <= nz ? P : nz - z0;               // this CTA's planes
    const int last_planes = nz - (csize - 1) * P;
    const int ncell = planes * nxy;
    const int64_t c0 = (int64_t)z0 * nxy;
    T* Xs = (T*)s_dyn;                      // [P nxy] x
    N* dA = (N*)(Xs + P * nxy);             // narrow true residual, then even directions
    N* dB = dA + P * nxy;                   // odd directions
    N* Qs = dB + P * nxy;                   // recursive residual

    T* Xg = (T*)md.x + f * C;
    T* Bg = (T*)md.b + f * C;
    T* XPg = md.xp ? (T*)md.xp + f * C : nullptr;
    // Work layout: thread t owns the (x, y) columns t, t + kClThreads, ... of the plane
    // and walks each column through this CTA's planes with a rolling window in z, so
    // the in-plane neighbours are fixed offsets per column and only the first and
    // last plane read a z-neighbour from another CTA (distributed shared memory,
    // both loaded before the walk).
    const bool pz = md.per[2] != 0;
    // z-neighbour below plane 0 / above the last plane of column s in array `arr`
    // (has = false: zero-flux face)
    auto z_below = [&](auto* arr, int s, bool& has) {
      using V = typename std::remove_const<typename std::remove_pointer<decltype(arr)>::type>::type;
      has = true;
      if (z0 > 0) return (V)cl.map_shared_rank(arr, (unsigned)(rank - 1))[(P - 1) * nxy + s];
      if (pz) {
        if (csize > 1) return (V)cl.map_shared_rank(arr, (unsigned)(csize - 1))[(last_planes - 1) * nxy + s];
        return (V)arr[(planes - 1) * nxy + s];
      }
      has = false;
      return V{};
    };
    auto z_above = [&](auto* arr, int s, bool& has) {
      using V = typename std::remove_const<typename std::remove_pointer<decltype(arr)>::type>::type;
      has = true;
      if (z0 + planes < nz) return (V)cl.map_shared_rank(arr, (unsigned)(rank + 1))[s];
      if (pz) {
        if (csize > 1) return (V)cl.map_shared_rank(arr, 0u)[s];
        return (V)arr[s];
      }
      has = false;
      return V{};
    };
    // in-plane neighbour offsets of column s (has[k] = false: zero-flux face)
    struct Col {
      int off[4];
      bool has[4];
    };
    auto col_of = [&](int sidx) {
      Col c;
      const int ix = sidx % nx, iy = sidx / nx;
      c.has[0] = ix > 0 || md.per[0];
      c.off[0] = ix > 0 ? -1 : nx - 1;
      c.has[1] = ix < nx - 1 || md.per[0];
      c.off[1] = ix < nx - 1 ? 1 : -(nx - 1);
      c.has[2] = iy > 0 || md.per[1];
      c.off[2] = iy > 0 ? -nx : (ny - 1) * nx;
      c.has[3] = iy < ny - 1 || md.per[1];
      c.off[3] = iy < ny - 1 ? nx : -(ny - 1) * nx;
      return c;
    };
    for (int m = 0; m < a.n_tau; ++m) {
      const int ph = (a.scheme == TAU_BDF2 && m > 0) ? 1 : 0;
      const SmoothSpec& sp = md.sp[ph];
      const T cf[3] = {coef_w<T>(sp, 0), coef_w<T>(sp, 1), coef_w<T>(sp, 2)};
      const N cfn[3] = {coef_w<N>(sp, 0), coef_w<N>(sp, 1), coef_w<N>(sp, 2)};
      N inv_theta;
      if constexpr (sizeof(N) == 4) inv_theta = sp.inv_theta_f;
      else inv_theta = (N)(1.0 / sp.theta);
      // ---- b (global) from the previous pseudo-step's result; x (or the guess)
      //      into shared memory
      for (int l = threadIdx.x; l < ncell; l += kClThreads) {
        const T xv = W::ld(Xg + c0 + l);
        Bg[c0 + l] = rhs_of<T>(a.scheme, m, xv, XPg ? XPg + c0 + l : nullptr);
        Xs[l] = (m == 0 && md.guess) ? W::ld((const T*)md.guess + f * C + c0 + l) : xv;
      }
      cl.sync();
      int total = 0, zero = 0;
      double bb = 0.0;
      for (int round = 0; round < kMaxRounds; ++round) {
        // ---- true residual (wide), its narrow copy in dA, sums
        Acc v[kQ] = {Acc(0), Acc(0), Acc(0), Acc(0)};
        // (A x)(c) = x_c - sum_a coef_a ((x_- - x_c) + (x_+ - x_c)), faces that exist
        auto wpair = [](bool h0, T v0, bool h1, T v1, T c) {
          if (h0 && h1) return W::addq(W::subq(v0, c), W::subq(v1, c));
          if (h0) return W::subq(v0, c);
          if (h1) return W::subq(v1, c);
          return W::zero();
        };
        for (int sidx = threadIdx.x; sidx < nxy; sidx += kClThreads) {
          const Col col = col_of(sidx);
          bool hb, hl;
          // both remote z-neighbours of the column are loaded before the walk
          T below = z_below(Xs, sidx, hb);
          const T top = z_above(Xs, sidx, hl);
          T cur = Xs[sidx];
          for (int izl = 0; izl < planes; ++izl) {
            const int l = izl * nxy + sidx;
            const bool ha = izl + 1 < planes || hl;
            const T above = izl + 1 < planes ? Xs[l + nxy] : top;
            const T sx = wpair(col.has[0], col.has[0] ? Xs[l + col.off[0]] : cur, col.has[1],
                               col.has[1] ? Xs[l + col.off[1]] : cur, cur);
            const T sy = wpair(col.has[2], col.has[2] ? Xs[l + col.off[2]] : cur, col.has[3],
                               col.has[3] ? Xs[l + col.off[3]] : cur, cur);
            T zt;
            if constexpr (GR) {
              // graded z: each face with its plane's own coefficient
              const double* cz = md.z.cz[ph] + 2 * (z0 + izl);
              zt = W::zero();
              if (hb) zt = W::mul(W::from_d(cz[0]), W::subq(below, cur));
              if (ha) zt = W::addq(zt, W::mul(W::from_d(cz[1]), W::subq(above, cur)));
            } else {
              zt = W::mul(cf[2], wpair(hb, below, ha, above, cur));
            }
            const T lap = W::addq(W::addq(W::mul(cf[0], sx), W::mul(cf[1], sy)), zt);
            const T ax = W::subq(cur, lap);
            const T bv = W::ld(Bg + c0 + l);
            const N rn = W::narrow(W::subq(bv, ax));
            dA[l] = rn;
            v[0] += (Acc)rn * (Acc)rn;
            v[1] += (Acc)rn;
            if constexpr (GR) v[3] += (Acc)md.z.w[z0 + izl] * (Acc)rn;
            if (round == 0) {
              const Acc bn = (Acc)W::narrow(bv);
              v[2] += bn * bn;
            }
            below = cur;
            hb = true;
            cur = above;
          }
        }
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
          // warp sums in the accumulation word (as the grid solver's units), the
          // CTA's sum of the 32 warp sums in FP64
          Acc t = v[q];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
          if (lane == 0) s_red[wid][q] = (double)t;
        }
        __syncthreads();
        // this CTA's sums, pushed into every CTA's shared memory (stores do not wait)
        if (threadIdx.x < csize * kQ) {
          const int r = threadIdx.x / kQ, q = threadIdx.x % kQ;
          double t = 0.0;
          for (int k = 0; k < kClThreads / 32; ++k) t += s_red[k][q];
          cl.map_shared_rank(&s_part[0][0], (unsigned)r)[rank * kQ + q] = t;
        }
        cl.sync();
        // one thread of every CTA sums the parts in rank order and decides: every CTA
        // takes the same decision
        if (threadIdx.x == 0) {
          double tot[kQ] = {0.0, 0.0, 0.0, 0.0};
          for (int r = 0; r < csize; ++r)
#pragma unroll
            for (int q = 0; q < kQ; ++q) tot[q] += s_part[r][q];
          if (round == 0) {
            bb = tot[2];
            zero = !(bb > 0.0);
          }
          const double Cd = (double)C;
          double shift, rrp;
          if (GR) {
            // the shift keeps sum(w x) = sum(w b); |r - s|^2 = |r|^2 - 2 s sum r + C s^2
            shift = zero ? 0.0 : tot[3] / md.z.wsum;
            rrp = fmax(tot[0] - 2.0 * shift * tot[1] + Cd * shift * shift, 0.0);
          } else {
            shift = zero ? 0.0 : tot[1] / Cd;
            rrp = fmax(tot[0] - tot[1] * tot[1] / Cd, 0.0);
          }
          int k = 0;
          if (!zero && !(rrp <= a.rtol2 * bb)) {
            // the step count only has to be about right (the next round checks the true
            // residual), so it is formed in FP32
            const float need = fmaxf(0.5f * sqrtf((float)(a.rtol2 * bb / rrp)), (float)W::kFloor);
            k = sp.sig > 0.0 ? (int)ceilf(logf(need) / logf((float)sp.sig)) : 1;
            if (k < 1) k = 1;
            if (k > kMaxStepsRound) k = kMaxStepsRound;
            if (total + k > a.max_iter) k = a.max_iter - total;
            if (k <= 0) {
              k = 0;
              if (rank == 0) atomicCAS((int*)&a.ctl->cg_status, 0, SEDI_EDIVERGED);
            }
          }
          s_k = k;
          s_shift = shift;
          s_zero = zero;
        }
        __syncthreads();
        const int k = s_k;
        const double shift = s_shift;
        zero = s_zero;
        total += k;
        if (k == 0) {
          // converged (or zero, or stopped): apply the projection shift, write x back
          const T sw = W::from_d(shift);
          for (int l = threadIdx.x; l < ncell; l += kClThreads) {
            T xv = Xs[l];
            if (zero) xv = W::zero();
            else if (shift != 0.0) xv = W::add(xv, sw);
            Xg[c0 + l] = xv;
          }
          break;
        }
        const N shn = (N)shift;
        const T sw = W::from_d(shift);
        // ---- Chebyshev steps (step 1 applies the shift and forms d0 = (r - s) / theta)
        for (int j = 1; j <= k; ++j) {
          N* Dold = (j & 1) ? dA : dB;
          N* Dnew = (j & 1) ? dB : dA;
          N c1s, c2s;
          if constexpr (sizeof(N) == 4) {
            c1s = sp.chebf[0][j - 1];
            c2s = sp.chebf[1][j - 1];
          } else {
            c1s = (N)sp.cheb[0][j - 1];
            c2s = (N)sp.cheb[1][j - 1];
          }
          // One step over this CTA's columns.  FIRST (step 1) reads the narrow true
          // residual r and forms d0 = (r - s) / theta at every point it touches; x and
          // the recursion take the shift.  FULL: all four in-plane faces exist (the
          // common case), so the loop has no per-face selects.
          auto step = [&](auto first_tag, auto full_tag, int sidx, const Col& col) {
            constexpr bool FIRST = decltype(first_tag)::value;
            constexpr bool FULL = decltype(full_tag)::value;
            auto tr = [&](N raw) {
              if constexpr (FIRST) return (raw - shn) * inv_theta;
              else return raw;
            };
            auto face = [&](bool h, int l, int off, N cur) {
              if constexpr (FULL) return tr(Dold[l + off]) - cur;
              else return h ? tr(Dold[l + off]) - cur : N(0);
            };
            bool hb, hl;
            // both remote z-neighbours of the column are loaded before the walk
            N below = tr(z_below(Dold, sidx, hb));
            const N top = tr(z_above(Dold, sidx, hl));
            N cur = tr(Dold[sidx]);
            for (int izl = 0; izl < planes; ++izl) {
              const int l = izl * nxy + sidx;
              const bool up = izl + 1 < planes;
              const N above = up ? tr(Dold[l + nxy]) : top;
              const N sx = face(col.has[0], l, col.off[0], cur) + face(col.has[1], l, col.off[1], cur);
              const N sy = face(col.has[2], l, col.off[2], cur) + face(col.has[3], l, col.off[3], cur);
              N zt;
              if constexpr (GR) {
                const float* cz = md.z.czf[ph] + 2 * (z0 + izl);
                zt = (hb ? (N)cz[0] * (below - cur) : N(0)) + ((up || hl) ? (N)cz[1] * (above - cur) : N(0));
              } else {
                zt = cfn[2] * ((hb ? below - cur : N(0)) + ((up || hl) ? above - cur : N(0)));
              }
              const N ad = cur - ((cfn[0] * sx + cfn[1] * sy) + zt);
              T xv = Xs[l];
              N q;
              if constexpr (FIRST) {
                xv = W::add(xv, sw);
                q = Dold[l] - shn;
              } else {
                q = Qs[l];
              }
              q = q - ad;
              Qs[l] = q;
              Dnew[l] = c1s * cur + c2s * q;
              Xs[l] = W::add_n(xv, cur);
              below = cur;
              hb = true;
              cur = above;
            }
          };
          for (int sidx = threadIdx.x; sidx < nxy; sidx += kClThreads) {
            const Col col = col_of(sidx);
            const bool full = col.has[0] && col.has[1] && col.has[2] && col.has[3];
            if (j == 1) {
              if (full) step(std::true_type{}, std::true_type{}, sidx, col);
              else step(std::true_type{}, std::false_type{}, sidx, col);
            } else {
              if (full) step(std::false_type{}, std::true_type{}, sidx, col);
              else step(std::false_type{}, std::false_type{}, sidx, col);
            }
          }
          cl.sync();
        }
      }
      if (rank == 0 && threadIdx.x == 0 && md.iters) atomicAdd(md.iters + f, total);
    }
  }
}

// ---------------------------------------------------------------- resident solver
// A group of CTAs solves one (mesh, field) pair at a time with the whole field on chip:
// CTA (ix, iy, iz) of the group holds a brick of bx x by x bz cells.
// x (wide) and the recursive residual q live in registers (a thread owns chunks of
// kRsZ cells along z), the direction d in shared memory, double-buffered, with halos.
// Same iteration as the solvers above, operation for operation; the sums of a round are theirs
// too (rs_sums), so are all bits of a result.
// Halos between CTAs go through global memory (they stay in L2) as 8-byte words of a value
// and the exchange's number, so a receiver polls the data itself: no fence, no flag and no
// barrier between a store and its use.  A round's sums travel the same way.  Every wait is
// bounded and every CTA of a group resident (cooperative launch); a field in one CTA
// needs neither.  Several groups work on the mesh's fields at once when they fit.
// A missing face (zero flux) is a halo that repeats the boundary cell: its difference is
// exactly zero, so there are no per-face branches.
//
// A direction buffer: the chunks [zc][y + 1][x + 1] as 4-cell vectors, with a halo chunk
// on each x and y side (an odd number a row, so a column of chunks meets no bank twice),
// then the planes below and above the brick, [y][x] words each, where z is cut.  A step
// reads a chunk and its four neighbours as vectors and two more words: 7 loads for 4
// cells.  A cut across z costs a word a cell of halo traffic, one across x or y a vector
// for four, so z is cut last.
//
// What bounds it: the exchange and the issue of a step.  On 128 x 64 x 128 a step takes
// 8 us for 6,900 cells a CTA (rounds included), of which the FP32 pipe accounts for 0.9 us
// (29 operations a cell at 128 a clock and SM; packed f32x2 instructions run at the same
// operation rate), one way between SMs through L2 for 0.8 us.
// Seven fields of random values, microseconds a call, streaming grid solver -> here:
// 128 x 64 x 128 9,760 -> 5,990, 256 x 128 x 64 10,190 -> 7,360, 96 x 96 x 24
// 2,030 -> 1,140; 10 x 10 x 20 in one CTA 440 -> 250; FP64 19 x 15 x 31 4,390 -> 750 (the
// streaming solver ran it on 35 blocks).
constexpr int kRsZ = 4;              // cells of a chunk
constexpr int kRsMaxGroup = 160;     // CTAs of a group at most
constexpr int kRsSumBytes = 5120;    // shared memory of a round's sums
constexpr size_t kRsSmem = 176 * 1024;  // dynamic shared memory of a CTA at most

// Threads of a CTA, and the chunks a thread holds at most: their x and q are 12 registers
// each in the double-float form (16 in FP64) of the 128 it has.
constexpr int kRsThreads = 512;
constexpr int kRsChunks = 4;         // where they do, and in FP64
constexpr int kRsChunksBig = 7;      // larger meshes

// The four cells of a chunk as loaded from a direction buffer.
struct C4f {
  float v[kRsZ];
};
struct C4d {
  double v[kRsZ];
};
__device__ __forceinline__ C4f ld_chunk(const float* p) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  return C4f{{t.x, t.y, t.z, t.w}};
}
__device__ __forceinline__ C4d ld_chunk(const double* p) {
  const double2 t = reinterpret_cast<const double2*>(p)[0], u = reinterpret_cast<const double2*>(p)[1];
  return C4d{{t.x, t.y, u.x, u.y}};
}
__device__ __forceinline__ void st_chunk(float* p, const float (&v)[kRsZ]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st_chunk(double* p, const double (&v)[kRsZ]) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}

// x as it is published for the true residual: the double-float word split over the two
// direction buffers, the other words in the first.
template <class T>
struct Pub;
template <>
struct Pub<dd> {
  static constexpr int n = 2;
  __device__ static float word(dd v, int k) { return k ? v.lo : v.hi; }
  __device__ static dd one(const float* d0, const float* d1, int o) { return dd{d0[o], d1[o]}; }
  __device__ static void chunk(const float* d0, const float* d1, int o, dd (&t)[kRsZ]) {
    const C4f h = ld_chunk(d0 + o), l = ld_chunk(d1 + o);
#pragma unroll
    for (int z = 0; z < kRsZ; ++z) t[z] = dd{h.v[z], l.v[z]};
  }
};
template <class T>
struct Pub {
  static constexpr int n = 1;
  __device__ static T word(T v, int) { return v; }
  __device__ static T one(const T* d0, const T*, int o) { return d0[o]; }
  __device__ static void chunk(const T* d0, const T*, int o, T (&t)[kRsZ]) {
    const auto h = ld_chunk(d0 + o);
#pragma unroll
    for (int z = 0; z < kRsZ; ++z) t[z] = h.v[z];
  }
};

// True residual b - A x of a cell (wide) as the narrow word: c the cell, l r f k its x and
// y neighbours, dn up its planes; cz the z-face coefficients of a graded mesh.
template <class T>
struct Resid {
  using W = Wide<T>;
  using N = typename W::N;
  __device__ static T pair(T m, T p, T c) { return W::addq(W::subq(m, c), W::subq(p, c)); }
  __device__ static N eval(const T (&cf)[3], T c, T l, T r, T f, T k, T dn, T up, T b) {
    const T lap = W::addq(W::addq(W::mul(cf[0], pair(l, r, c)), W::mul(cf[1], pair(f, k, c))),
                          W::mul(cf[2], pair(dn, up, c)));
    return W::narrow(W::subq(b, W::subq(c, lap)));
  }
  // zz: the z faces' terms are added to each other first (the cluster solver's order)
  __device__ static N eval_z(const T (&cf)[3], const double* cz, bool zz, T c, T l, T r, T f, T k, T dn, T up, T b) {
    T lap = W::addq(W::mul(cf[0], pair(l, r, c)), W::mul(cf[1], pair(f, k, c)));
    const T tm = W::mul(W::from_d(cz[0]), W::subq(dn, c)), tp = W::mul(W::from_d(cz[1]), W::subq(up, c));
    lap = zz ? W::addq(lap, W::addq(tm, tp)) : W::addq(W::addq(lap, tm), tp);
    return W::narrow(W::subq(b, W::subq(c, lap)));
  }
};
// Words that carry their own arrival: each 8-byte word of global memory holds 32 bits of
// data and the number of the exchange that wrote it.  A 64-bit access is indivisible, so
// a reader that finds the number has the data, with no fence between them.
__device__ __forceinline__ unsigned long long tag(uint32_t w, uint32_t e) {
  return (unsigned long long)e << 32 | w;
}
__device__ __forceinline__ void put2(unsigned long long* p, uint32_t w0, uint32_t w1, uint32_t e) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(tag(w0, e)), "l"(tag(w1, e)) : "memory");
}
__device__ __forceinline__ void put1(unsigned long long* p, uint32_t w, uint32_t e) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(tag(w, e)) : "memory");
}
struct Tag2 {
  unsigned long long a, b;
  __device__ void load(const unsigned long long* p) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  }
  __device__ bool is(uint32_t e) const { return (uint32_t)(a >> 32) == e && (uint32_t)(b >> 32) == e; }
};
__device__ __forceinline__ unsigned long long get1(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
// A waiting poll: false once the limit is reached (SEDI_ETIMEOUT recorded) or another
// block gave up.
struct Spin {
  unsigned n = 0;
  __device__ bool go(Ctl* ctl, long long limit) {
    if (++n > (unsigned)limit) {
      atomicCAS((int*)&ctl->cg_status, 0, SEDI_ETIMEOUT);
      return false;
    }
    return (n & 255) != 0 || *((volatile int*)&ctl->cg_status) != SEDI_ETIMEOUT;
  }
};
__device__ __forceinline__ uint32_t as_word(float v, int) { return __float_as_uint(v); }
__device__ __forceinline__ uint32_t as_word(double v, int k) {
  return k ? (uint32_t)__double2hiint(v) : (uint32_t)__double2loint(v);
}
__device__ __forceinline__ void of_words(float& v, uint32_t a, uint32_t) { v = __uint_as_float(a); }
__device__ __forceinline__ void of_words(double& v, uint32_t a, uint32_t b) { v = __hiloint2double((int)b, (int)a); }

// The halos of a CTA from its tagged words: unit u < nu a chunk (kRsZ values), the nw units
// after them one value each, laid out in that order; pull[u] the word of the buffer that
// it fills (top bit: none).  Not inlined: a caller full of live registers would spill.
template <class N, int TH>
__device__ __noinline__ bool rs_receive(N* D, const uint32_t* pull, int nu, int nw, const unsigned long long* src,
                                        uint32_t seq, Ctl* ctl, long long spin_limit) {
  constexpr int NW = sizeof(N) / 4, K = 2;  // chunks in flight
  bool ok = true;
#pragma unroll 1
  for (int u0 = threadIdx.x; u0 < nu; u0 += K * TH) {
#pragma unroll
    for (int h = 0; h < NW; ++h) {  // FP64: two halves of a chunk
      Tag2 t[K][2];
      uint32_t e[K];
#pragma unroll
      for (int q = 0; q < K; ++q) {
        const int u = u0 + q * TH;
        e[q] = u < nu ? pull[u] : 1u << 31;
        if (e[q] >> 31) continue;
        t[q][0].load(src + (u * NW + h) * 4);
        t[q][1].load(src + (u * NW + h) * 4 + 2);
      }
#pragma unroll
      for (int q = 0; q < K; ++q) {
        if (e[q] >> 31) continue;
        Spin spin;
        while (!(t[q][0].is(seq) && t[q][1].is(seq)) && ok) {
          ok = spin.go(ctl, spin_limit);
          const int u = u0 + q * TH;
          t[q][0].load(src + (u * NW + h) * 4);
          t[q][1].load(src + (u * NW + h) * 4 + 2);
        }
        N* const to = D + e[q];
        if constexpr (NW == 1) {
          N c[kRsZ];
          of_words(c[0], (uint32_t)t[q][0].a, 0u);
          of_words(c[1], (uint32_t)t[q][0].b, 0u);
          of_words(c[2], (uint32_t)t[q][1].a, 0u);
          of_words(c[3], (uint32_t)t[q][1].b, 0u);
          st_chunk(to, c);
        } else {
          of_words(to[2 * h], (uint32_t)t[q][0].a, (uint32_t)t[q][0].b);
          of_words(to[2 * h + 1], (uint32_t)t[q][1].a, (uint32_t)t[q][1].b);
        }
      }
    }
  }
  const unsigned long long* const ws = src + (size_t)nu * kRsZ * NW;
#pragma unroll 1
  for (int u0 = threadIdx.x; u0 < nw; u0 += 4 * TH) {
    unsigned long long t[4][NW];
    uint32_t e[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int u = u0 + q * TH;
      e[q] = u < nw ? pull[nu + u] : 1u << 31;
      if (!(e[q] >> 31))
#pragma unroll
        for (int k = 0; k < NW; ++k) t[q][k] = get1(ws + u * NW + k);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (e[q] >> 31) continue;
#pragma unroll
      for (int k = 0; k < NW; ++k) {
        Spin spin;
        while ((uint32_t)(t[q][k] >> 32) != seq && ok) {
          ok = spin.go(ctl, spin_limit);
          t[q][k] = get1(ws + (u0 + q * TH) * NW + k);
        }
      }
      of_words(D[e[q]], (uint32_t)t[q][0], (uint32_t)t[q][NW - 1]);
    }
  }
  return ok;
}

// The sums of a round, in the order of the solver that takes this mesh otherwise, so neither the
// choice of solver nor a cut changes a bit of a result (an averaged solid fraction that
// rounds to another FP32 word would change the drag and a trajectory with it).

// A mesh of one CTA (FP32 words), which the cluster solver would hold in one too: thread t of its 1,024
// adds columns t, t + 1,024, ..., a warp its threads, the CTA its 32 warps in FP64.  The
// residuals are in shared memory.
template <class T, bool GR>
__device__ __forceinline__ void rs_sums_one(const SmoothMeshDev& md, const float* r, const T* b, bool first, float* sl,
                                         double* tot) {
  using W = Wide<T>;
  constexpr int TH = kRsThreads;
  const int tid = threadIdx.x, lane = tid & 31;
  const int nxy = md.nc[0] * md.nc[1], nz = md.nc[2];
  __syncthreads();
#pragma unroll 1
  for (int t = tid; t < kClThreads; t += TH) {
    float v[kQ] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int s = t; s < nxy; s += kClThreads) {
      constexpr int kAhead = 8;  // planes whose loads are under way together
      for (int za = 0; za < nz; za += kAhead) {
        float rn[kAhead];
        T bv[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
          const int64_t c = (int64_t)(za + k) * nxy + s;
          rn[k] = za + k < nz ? r[c] : 0.0f;
          bv[k] = W::zero();
          if (first) bv[k] = za + k < nz ? W::ld(b + c) : W::zero();
        }
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
          if (za + k >= nz) continue;
          v[0] += rn[k] * rn[k];
          v[1] += rn[k];
          if constexpr (GR) v[3] += (float)md.z.w[za + k] * rn[k];
          const float bn = W::narrow(bv[k]);
          v[2] += bn * bn;
        }
      }
    }
    // a butterfly from 16 down for each value: 0 and 2 in the lower half of the lanes, 1
    // and 3 in the upper
    const bool up = lane & 16;
    float a = up ? v[1] : v[0], c = up ? v[3] : v[2];
    a += __shfl_xor_sync(0xffffffffu, up ? v[0] : v[1], 16);
    if (first || GR) c += __shfl_xor_sync(0xffffffffu, up ? v[2] : v[3], 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      if (first || GR) c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if ((lane & 15) == 0) {
      float* const to = sl + (t >> 5) * kQ;
      to[up ? 1 : 0] = a;
      to[up ? 3 : 2] = c;
    }
  }
  __syncthreads();
  if (tid < kQ) {
    double t = 0.0;
    for (int w = 0; w < kClThreads / 32; ++w) t += (double)sl[w * kQ + tid];
    tot[tid] = t;
  }
  __syncthreads();
}

// A group's tagged words of the sums: a flag a CTA (its residuals are in place), then the
// pieces below, each for two parities.
constexpr int kRsPieces = kThreads;
static_assert(kThreads == 256, "");
__host__ __device__ constexpr size_t rs_sum_words(int G) { return 2 * ((size_t)G + 2 * kRsPieces * kQ); }

// One CTA: as above.  Several CTAs, a mesh that the streaming solver would take: its thread t of 256
// adds units t, t + 256, ... of 256 cells in FP64, a piece.  Piece p is formed by CTA p % G
// from the residuals in global memory and goes to every CTA as tagged words.  This costs two
// exchanges and a read of the residuals from L2 a round: 1,000 of the 5,990 us of seven
// 128 x 64 x 128 fields, twelve rounds each.
template <class T, bool GR>
__device__ __noinline__ bool rs_sums(const SmoothMeshDev& md, const typename Wide<T>::N* r, const T* b, bool first,
                                     int G, int rank, typename Wide<T>::N* sl, unsigned long long* words, uint32_t seq, double* tot, int* s_ok,
                                     Ctl* ctl, long long spin_limit) {
  using W = Wide<T>;
  using N = typename W::N;
  constexpr int TH = kRsThreads, kWarps = TH / 32, kUnits = kRsSumBytes / (8 * kQ * sizeof(N));
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nxy = md.nc[0] * md.nc[1];
  const int64_t C = md.C;
  if constexpr (sizeof(N) == 4) {
    if (G == 1) {
      rs_sums_one<T, GR>(md, r, b, first, sl, tot);
      return true;
    }
  }
  unsigned long long* const flags = words + (size_t)(seq & 1) * G;
  unsigned long long* const pieces = words + 2 * (size_t)G + (size_t)(seq & 1) * 2 * kRsPieces * kQ;
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    put1(flags + rank, 0u, seq);
  }
  if (tid < G) {
    Spin spin;
    while ((uint32_t)(get1(flags + tid) >> 32) != seq)
      if (!spin.go(ctl, spin_limit)) {
        *s_ok = 0;
        break;
      }
    __threadfence();
  }
  __syncthreads();
  if (!*s_ok) return false;
  bool ok = true;
  auto get_piece = [&](int p, int q) {
    const unsigned long long* const at = pieces + ((size_t)p * kQ + q) * 2;
    Tag2 v;
    v.load(at);
    Spin spin;
    while (!v.is(seq) && ok) {
      ok = spin.go(ctl, spin_limit);
      v.load(at);
    }
    double d;
    of_words(d, (uint32_t)v.a, (uint32_t)v.b);
    return d;
  };
  // warp sums of the 8 warps of a unit, two values each: the same butterflies as a
  // reduce-scatter, a lane keeps half of its sums at every step
  auto unit_warps = [&](N (&v)[2][8], N* to) {
    N a[8];
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      const bool up = lane & 16;
      a[w] = (up ? v[1][w] : v[0][w]) + __shfl_xor_sync(0xffffffffu, up ? v[0][w] : v[1][w], 16);
    }
#pragma unroll
    for (int o = 8; o > 1; o >>= 1) {
      const bool up = lane & o;
#pragma unroll
      for (int w = 0; w < o / 2; ++w)
        a[w] = (up ? a[w + o / 2] : a[w]) + __shfl_xor_sync(0xffffffffu, up ? a[w] : a[w + o / 2], o);
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    if (!(lane & 1)) to[lane >> 1] = a[0];  // [value][warp]
  };
  const int nu = (int)md.nu, np = nu < kRsPieces ? nu : kRsPieces;
  const int mine = rank < np ? (np - rank + G - 1) / G : 0;  // this CTA's pieces rank, rank + G, ...
  const int all = mine * ((nu + kRsPieces - 1) / kRsPieces);
  double acc = 0.0;  // of piece tid / kQ of them (128 at most), sum tid % kQ
  for (int i0 = 0; i0 < all; i0 += kUnits) {  // units in order for every piece
    const int n = all - i0 < kUnits ? all - i0 : kUnits;
#pragma unroll 1
    for (int s = wid; s < n; s += kWarps) {  // a warp takes the 8 warps of a unit
      const int i = i0 + s, u = rank + i % mine * G + i / mine * kRsPieces;
      const int64_t c0 = (int64_t)u * kThreads + lane;
      N rn[8], v[2][8];
      T bv[8];
#pragma unroll
      for (int w = 0; w < 8; ++w) {  // every load before the first use
        const int64_t c = c0 + w * 32;
        const bool in = u < nu && c < C;
        rn[w] = in ? __ldcg(r + c) : N(0);
        bv[w] = W::zero();
        if (first) bv[w] = in ? W::ld(b + c) : W::zero();
      }
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        v[0][w] = rn[w] * rn[w];
        v[1][w] = rn[w];
      }
      unit_warps(v, sl + s * (8 * kQ));
      if (GR || first) {
#pragma unroll
        for (int w = 0; w < 8; ++w) {
          const N bn = W::narrow(bv[w]);
          v[0][w] = bn * bn;
          v[1][w] = N(0);
          if constexpr (GR) {
            const int c = (int)c0 + w * 32;
            if (u < nu && c < C) v[1][w] = (N)md.z.w[c / nxy] * rn[w];
          }
        }
        unit_warps(v, sl + s * (8 * kQ) + 16);
      }
    }
    __syncthreads();
    if (tid < n * kQ && (GR || first || tid % kQ < 2)) {  // a unit's sum, in the place of its warps'
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < 8; ++w) t += (double)sl[tid * 8 + w];
      ((double*)sl)[tid * sizeof(N)] = t;
    }
    __syncthreads();
    if (tid < mine * kQ) {
      const int j = tid / kQ, q = tid % kQ;
      for (int k = ((j - i0) % mine + mine) % mine; k < n; k += mine)
        if (rank + j * G + (i0 + k) / mine * kRsPieces < nu) acc += ((double*)sl)[(k * kQ + q) * sizeof(N)];
    }
    __syncthreads();
  }
  double* const ws = (double*)sl;  // sums of 32 pieces
  if (tid < mine * kQ)
    put2(pieces + ((size_t)(rank + tid / kQ * G) * kQ + tid % kQ) * 2, as_word(acc, 0), as_word(acc, 1), seq);
#pragma unroll
  for (int k = wid; k < 8 * kQ; k += kWarps) {
    const int p = k / kQ * 32 + lane, q = k % kQ;
    double v = p < np ? get_piece(p, q) : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) ws[k] = v;
  }
  if (!ok) *s_ok = 0;
  __syncthreads();
  if (tid < kQ) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += ws[w * kQ + tid];
    tot[tid] = t;
  }
  __syncthreads();
  return *s_ok;
}

template <class T, bool GR, int M>
__global__ void __launch_bounds__(kRsThreads, 1) k_smooth_rs(SmoothBatchDev a) {
  using W = Wide<T>;
  using N = typename W::N;
  using P = Pub<T>;
  constexpr int TH = kRsThreads;
  constexpr int NW = sizeof(N) / 4;  // 32-bit words of a narrow value
  // a chunk's first word: index of its first cell, valid cells, chunk along z; its second
  // word: the indexes of the cells below and above it
  constexpr int kCnt = 18, kZc = 21;
  extern __shared__ __align__(16) unsigned char s_dyn[];
  __shared__ double s_part[kRsSumBytes / 8];  // rs_sums
  __shared__ double s_tot[kQ], s_shift;
  __shared__ uint2 s_info[M * TH];
  __shared__ int s_cell[M * TH];  // first cell of a chunk in the mesh
  __shared__ int s_k, s_zero, s_ok;
  // the item's neighbours and pointers (registers hold the field)
  __shared__ struct {
    int nb[6];             // neighbour CTAs below / above along x, y and z (-1: none)
    int dst[6];            // x, y: words from a boundary cell to the halo that takes it;
                           // z: the halo plane that takes it
    T *x, *b, *xp;
    const T* guess;
    N* r;                  // the narrow true residual between its pass and the step loop (FP32
                           // words in one CTA: in shared memory)
    unsigned long long* halo;  // grid: the group's tagged halo words, [CTA][parity][channel][hw]
    unsigned long long* sums;  // grid: the group's tagged words of the sums (rs_sums)
  } s_g;
  const int tid = threadIdx.x;
  const int G = a.rs_G, rank = (int)(blockIdx.x % (unsigned)G);
  const int64_t grp = blockIdx.x / (unsigned)G, ngrp = gridDim.x / (unsigned)G;
  uint32_t seq = 0, rseq = 0;  // halo exchanges and reductions so far
  if (tid == 0) s_ok = 1;
  const int64_t items = (int64_t)a.B * a.nf;
  for (int64_t w = grp; w < items; w += ngrp) {
    const int bi = (int)(w / a.nf), f = (int)(w % a.nf);
    const SmoothMeshDev& md = a.mesh[bi];
    const int64_t C = md.C;
    const int nx = md.nc[0], ny = md.nc[1], nz = md.nc[2], nxy = nx * ny;
    const int px = md.rs_px, py = md.rs_py, pz = md.rs_pz;
    const int ix = rank % px, iy = rank / px % py, iz = rank / (px * py);
    // first cell of part i of n cells cut in p
    auto cut = [](int i, int n, int p) { return (int)((int64_t)i * n / p); };
    const int x0 = cut(ix, nx, px), bx = cut(ix + 1, nx, px) - x0;
    const int y0 = cut(iy, ny, py), by = cut(iy + 1, ny, py) - y0;
    const int z0 = cut(iz, nz, pz), bz = cut(iz + 1, nz, pz) - z0;
    const int bxm = (nx + px - 1) / px, bym = (ny + py - 1) / py;
    const int nzcm = ((nz + pz - 1) / pz + kRsZ - 1) / kRsZ;
    const bool zcut = pz > 1 || md.per[2];              // halo planes are exchanged
    const int pr = ((bxm + 2) | 1) * kRsZ;              // words of a row
    const int cs = (bym + 2) * pr;                      // words of a chunk layer
    const int zlo = nzcm * cs, zhi = zlo + (zcut ? bym * bxm : 0);   // halo planes
    const int words = (zhi + (zcut ? bym * bxm : 0) + 3) & ~3;      // of a buffer
    const int bxy = bx * by, nzc = (bz + kRsZ - 1) / kRsZ, nch = bxy * nzc;
    const bool part = bz % kRsZ != 0;
    [[maybe_unused]] const bool zz = md.cl_size > 0;    // order of a graded mesh's z terms
    // grid: room for the halo words of a CTA and channel
    const int hw = 2 * (nzcm * kRsZ * (bxm + bym) + (zcut ? bxm * bym : 0));
    const int nu = 2 * nzc * (bx + by), nw = zcut ? 2 * bxy : 0;  // halo units: chunks, words
    N* const D0 = (N*)s_dyn;
    N* const D1 = D0 + words;
    N* const s_cz = D1 + words;  // [bz][2] z-face coefficients (graded mesh)
    // halo units: {word of the boundary cell | kLocal, target}: a word of this CTA's buffer
    // (local) or a tagged word of the neighbour's; and the word of this CTA's halo that
    // unit u of its own tagged words fills (kLocal: none)
    uint2* const s_push = (uint2*)(s_cz + (GR ? 2 * nzcm * kRsZ : 0));
    const int nu_max = 2 * nzcm * (bxm + bym) + (zcut ? 2 * bxm * bym : 0);
    uint32_t* const s_pull = (uint32_t*)(s_push + nu_max);
    constexpr uint32_t kLocal = 1u << 31;

    __syncthreads();  // the previous item's readers of s_g and s_info are done
    if (tid == 0) {
      auto rank_of = [&](int jx, int jy, int jz) { return (jz * py + jy) * px + jx; };
      // the neighbour on each side, or -1 at a face without flux; a missing x or y face
      // pushes the boundary cells to this CTA's own halo on that side, a missing z face
      // needs none (the cell below or above is the boundary cell itself)
      const int p3[3] = {px, py, pz};
      for (int s = 0; s < 6; ++s) {
        const int ax = s >> 1, up = s & 1;
        int j[3] = {ix, iy, iz};
        j[ax] += up ? 1 : -1;
        const bool in = j[ax] >= 0 && j[ax] < p3[ax];
        if (!in) j[ax] = up ? 0 : p3[ax] - 1;
        s_g.nb[s] = in || md.per[ax] ? rank_of(j[0], j[1], j[2]) : -1;
        const int n = ax == 0 ? nx : ny, mine = ax == 0 ? bx : by, step = ax == 0 ? kRsZ : pr;
        if (ax < 2) {
          const int theirs = cut(j[ax] + 1, n, p3[ax]) - cut(j[ax], n, p3[ax]);
          s_g.dst[s] = s_g.nb[s] < 0 ? (up ? step : -step) : (up ? -mine * step : theirs * step);
        } else {
          s_g.dst[s] = up ? zlo : zhi;
        }
      }
      s_g.x = (T*)md.x + f * C;
      s_g.b = (T*)md.b + f * C;
      s_g.xp = md.xp ? (T*)md.xp + f * C : nullptr;
      s_g.guess = md.guess ? (const T*)md.guess + f * C : nullptr;
      s_g.r = G == 1 ? (N*)(s_pull + nu_max) : (N*)md.q + f * C;
      s_g.sums = (unsigned long long*)md.tags + (size_t)grp * rs_sum_words(G);
      s_g.halo = (unsigned long long*)md.tags + (size_t)ngrp * rs_sum_words(G) + (size_t)grp * G * 2 * P::n * hw * NW;
    }
    __syncthreads();
#pragma unroll 1
    for (int m = 0; m < M; ++m) {
      const int c = tid + m * TH;
      uint2 in = make_uint2(0u, 0u);
      int g = 0;
      if (c < nch) {
        const int zc = c / bxy, r = c - zc * bxy, y = r / bx, x = r - y * bx;
        const int cnt = bz - zc * kRsZ < kRsZ ? bz - zc * kRsZ : kRsZ;
        const int o = zc * cs + (y + 1) * pr + (x + 1) * kRsZ;
        const int ob = zc > 0 ? o - cs + kRsZ - 1 : s_g.nb[4] < 0 ? o : zlo + r;
        const int oa = zc + 1 < nzc ? o + cs : s_g.nb[5] < 0 ? o + cnt - 1 : zhi + r;
        in.x = (uint32_t)o | ((uint32_t)cnt << kCnt) | ((uint32_t)zc << kZc);
        in.y = (uint32_t)ob | ((uint32_t)oa << 16);
        g = (z0 + zc * kRsZ) * nxy + (y0 + y) * nx + x0 + x;
      }
      s_info[m * TH + tid] = in;
      s_cell[m * TH + tid] = g;
    }
    // the first unit of side s in CTA r of the group (its units are in side order); words
    // of the z sides follow the chunks
    [[maybe_unused]] auto ufirst = [&](int s, int r) {
      const int jx = r % px, jy = r / px % py, jz = r / (px * py);
      const int wx = cut(jx + 1, nx, px) - cut(jx, nx, px), wy = cut(jy + 1, ny, py) - cut(jy, ny, py);
      const int wz = (cut(jz + 1, nz, pz) - cut(jz, nz, pz) + kRsZ - 1) / kRsZ;
      const int c = s < 2 ? s * wz * wy : 2 * wz * wy + (s == 2 ? 0 : wz * wx);
      return s < 4 ? c * kRsZ : 2 * wz * (wx + wy) * kRsZ + (s - 4) * wx * wy;
    };
    // the halo units
    for (int u = tid; u < nu + nw; u += TH) {
      int s, v, src, dst, fill, far;
      if (u < nu) {
        const int nxs = nzc * by, nys = nzc * bx;
        s = u < nxs ? 0 : u < 2 * nxs ? 1 : u < 2 * nxs + nys ? 2 : 3;
        v = u - (s == 0 ? 0 : s == 1 ? nxs : s == 2 ? 2 * nxs : 2 * nxs + nys);
        const int wide = s < 2 ? by : bx, zc = v / wide, i = v - zc * wide, step = s < 2 ? pr : kRsZ;
        const int base = zc * cs + pr + kRsZ + i * step;
        src = base + (s == 1 ? (bx - 1) * kRsZ : s == 3 ? (by - 1) * pr : 0);
        fill = base + (s == 0 ? -kRsZ : s == 1 ? bx * kRsZ : s == 2 ? -pr : by * pr);
        dst = src + s_g.dst[s];
        far = s_g.nb[s] < 0 ? 0 : ufirst(s ^ 1, s_g.nb[s]) + v * (u < nu ? kRsZ : 1);
      } else {
        s = u - nu < bxy ? 4 : 5;
        v = u - nu - (s == 5 ? bxy : 0);
        const int y = v / bx;
        src = (s == 5 ? (bz - 1) / kRsZ * cs + (bz - 1) % kRsZ : 0) + (y + 1) * pr + (v - y * bx + 1) * kRsZ;
        fill = (s == 5 ? zhi : zlo) + v;
        dst = s_g.dst[s] + v;
        far = s_g.nb[s] < 0 ? 0 : ufirst(s ^ 1, s_g.nb[s]) + v * (u < nu ? kRsZ : 1);
      }
      const int nb = s_g.nb[s];
      const bool none = s >= 4 && nb < 0;  // no halo plane: the word goes nowhere
      const bool local = nb < 0 || nb == rank;
      s_push[u] = local ? make_uint2((uint32_t)src | kLocal, (uint32_t)(none ? src : dst))
                        : make_uint2((uint32_t)src, (uint32_t)(nb * 2 * P::n * hw + far));
      s_pull[u] = local ? kLocal : (uint32_t)fill;
    }
    __syncthreads();
    auto info = [&](int m) { return s_info[m * TH + tid]; };
    auto count = [&](int m) { return (int)(s_info[m * TH + tid].x >> kCnt & 7u); };
    auto cell = [&](int m) { return s_cell[m * TH + tid]; };

    // After the chunks of this CTA are in buffers b0 (and b0 ^ 1): the boundary cells go into
    // the neighbours' halos; every halo of this CTA is in place on return.  False after a
    // timeout.
    auto exchange = [&](int b0, int nchan) -> bool {
      ++seq;
      __syncthreads();
#pragma unroll 1
      for (int ch = 0; ch < nchan; ++ch) {
        N* const D = (b0 ^ ch) ? D1 : D0;
        unsigned long long* const far = s_g.halo + (size_t)((int)(seq & 1) * P::n + ch) * hw * NW;
#pragma unroll 1
        for (int u = tid; u < nu; u += TH) {
          const uint2 e = s_push[u];
          const auto c = ld_chunk(D + (e.x & 0xffffu));
          if (e.x & kLocal) {
            st_chunk(D + e.y, c.v);
          } else {
#pragma unroll
            for (int k = 0; k < kRsZ * NW; k += 2)
              put2(far + (size_t)e.y * NW + k, as_word(c.v[k / NW], k % NW), as_word(c.v[(k + 1) / NW], (k + 1) % NW), seq);
          }
        }
#pragma unroll 1
        for (int u = nu + tid; u < nu + nw; u += TH) {
          const uint2 e = s_push[u];
          const N c = D[e.x & 0xffffu];
          if (e.x & kLocal) D[e.y] = c;
          else if constexpr (NW == 1) put1(far + e.y, as_word(c, 0), seq);
          else put2(far + (size_t)e.y * NW, as_word(c, 0), as_word(c, 1), seq);
        }
      }
      if (G > 1) {
#pragma unroll 1
        for (int ch = 0; ch < nchan; ++ch)
          if (!rs_receive<N, TH>((b0 ^ ch) ? D1 : D0, s_pull, nu, nw,
                                 s_g.halo + (size_t)((rank * 2 + (int)(seq & 1)) * P::n + ch) * hw * NW, seq, a.ctl,
                                 a.spin_limit))
            s_ok = 0;
      }
      __syncthreads();
      return s_ok;

    };

    T X[M][kRsZ];
    N Q[M][kRsZ];
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
      for (int z = 0; z < kRsZ; ++z) {
        X[m][z] = W::zero();
        Q[m][z] = N(0);
      }
    for (int m_tau = 0; m_tau < a.n_tau; ++m_tau) {
      const int ph = (a.scheme == TAU_BDF2 && m_tau > 0) ? 1 : 0;
      const SmoothSpec& sp = md.sp[ph];
      if constexpr (GR) {
        for (int k = tid; k < 2 * bz; k += TH) {
          if constexpr (sizeof(N) == 4) s_cz[k] = md.z.czf[ph][2 * z0 + k];
          else s_cz[k] = (N)md.z.cz[ph][2 * z0 + k];
        }
      }
      // ---- b from the previous pseudo-step's result (in registers; the first step loads
      //      it); x, or the guess
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const int cnt = count(m);
        if (!cnt) continue;
        const int g = cell(m);
#pragma unroll
        for (int z = 0; z < kRsZ; ++z) {
          if (z >= cnt) continue;
          const int k = g + z * nxy;
          const T xv = m_tau == 0 ? W::ld(s_g.x + k) : X[m][z];
          s_g.b[k] = rhs_of<T>(a.scheme, m_tau, xv, s_g.xp ? s_g.xp + k : nullptr);
          X[m][z] = m_tau == 0 && s_g.guess ? W::ld(s_g.guess + k) : xv;
        }
      }
      int total = 0;
      double bb = 0.0;
      for (int round = 0; round < kMaxRounds; ++round) {
        // ---- x published, its halos in place
#pragma unroll
        for (int m = 0; m < M; ++m) {
          const uint2 in = info(m);
          if (!in.x) continue;
#pragma unroll
          for (int ch = 0; ch < P::n; ++ch) {
            N v[kRsZ];
#pragma unroll
            for (int z = 0; z < kRsZ; ++z) v[z] = P::word(X[m][z], ch);
            st_chunk((ch ? D1 : D0) + (in.x & 0xffffu), v);
          }
        }
        if (!exchange(0, P::n)) return;
        // ---- true residual (wide), its narrow copy to global memory; the next chunk's b is
        //      loaded ahead
        {
          const T cf[3] = {coef_w<T>(sp, 0), coef_w<T>(sp, 1), coef_w<T>(sp, 2)};
          T bn[kRsZ];
          auto load_b = [&](int m) {
            const int cnt = m < M ? count(m) : 0;
            if (!cnt) return;
            const T* const p = s_g.b + cell(m);
#pragma unroll
            for (int z = 0; z < kRsZ; ++z)
              if (z < cnt) bn[z] = W::ld(p + z * nxy);
          };
          // one chunk; out(z, r) takes its residuals
          auto chunk = [&](int m, auto&& out) {
            const uint2 in = info(m);
            const int o = (int)(in.x & 0xffffu), cnt = (int)(in.x >> kCnt & 7u);
            [[maybe_unused]] const int kz = z0 + (int)(in.x >> kZc) * kRsZ;
            T bv[kRsZ], c[kRsZ], l[kRsZ], r[kRsZ], fr[kRsZ], bk[kRsZ];
#pragma unroll
            for (int z = 0; z < kRsZ; ++z) bv[z] = bn[z];
            load_b(m + 1);
            P::chunk(D0, D1, o, c);
            P::chunk(D0, D1, o - kRsZ, l);
            P::chunk(D0, D1, o + kRsZ, r);
            P::chunk(D0, D1, o - pr, fr);
            P::chunk(D0, D1, o + pr, bk);
            T below = P::one(D0, D1, (int)(in.y & 0xffffu));
            const T top = P::one(D0, D1, (int)(in.y >> 16));
#pragma unroll
            for (int z = 0; z < kRsZ; ++z) {
              if (z < cnt) {
                const T above = z + 1 < kRsZ && z + 1 < cnt ? c[z + 1 < kRsZ ? z + 1 : z] : top;
                N rn;
                if constexpr (GR)
                  rn = Resid<T>::eval_z(cf, md.z.cz[ph] + 2 * (kz + z), zz, c[z], l[z], r[z], fr[z], bk[z], below, above, bv[z]);
                else
                  rn = Resid<T>::eval(cf, c[z], l[z], r[z], fr[z], bk[z], below, above, bv[z]);
                out(z, rn);
              }
              below = c[z];
            }
          };
          load_b(0);
          // rolled (x and q fill the registers): the residuals pass through global memory
#pragma unroll 1
          for (int m = 0; m < M && count(m); ++m) {
            N* const rg = s_g.r + cell(m);
            chunk(m, [&](int z, N rn) { rg[z * nxy] = rn; });
          }
        }
        ++rseq;
        if (!rs_sums<T, GR>(md, s_g.r, s_g.b, round == 0, G, rank, (N*)s_part, s_g.sums, rseq, s_tot, &s_ok, a.ctl,
                            a.spin_limit))
          return;
        // one thread of every CTA decides: every CTA takes the same decision
        if (tid == 0) {
          const double rr = s_tot[0], sr = s_tot[1];
          if (round == 0) bb = s_tot[2];
          const int zero = !(bb > 0.0);
          double shift, rrp;
          if (GR) {
            // the shift keeps sum(w x) = sum(w b); |r - s|^2 = |r|^2 - 2 s sum r + C s^2
            shift = zero ? 0.0 : s_tot[3] / md.z.wsum;
            rrp = fmax(rr - 2.0 * shift * sr + (double)C * shift * shift, 0.0);
          } else {
            shift = zero ? 0.0 : sr / (double)C;
            rrp = fmax(rr - sr * sr / (double)C, 0.0);
          }
          int k = 0;
          if (!zero && !(rrp <= a.rtol2 * bb)) {
            // |r_k| <= 2 sig^k |r_0|: enough steps for the tolerance, or for the reduction
            // the narrow word can deliver in one round (as the cluster solver forms the
            // count where it would take the mesh, else as the streaming one)
            if (md.cl_size > 0) {
              const float need = fmaxf(0.5f * sqrtf((float)(a.rtol2 * bb / rrp)), (float)W::kFloor);
              k = sp.sig > 0.0 ? (int)ceilf(logf(need) / logf((float)sp.sig)) : 1;
            } else {
              const double need = fmax(0.5 * sqrt(a.rtol2 * bb / rrp), W::kFloor);
              k = sp.sig > 0.0 ? (int)ceil(log(need) / log(sp.sig)) : 1;
            }
            if (k < 1) k = 1;
            if (k > kMaxStepsRound) k = kMaxStepsRound;
            if (total + k > a.max_iter) k = a.max_iter - total;
            if (k <= 0) {
              k = 0;
              if (rank == 0) atomicCAS((int*)&a.ctl->cg_status, 0, SEDI_EDIVERGED);
            }
          }
          s_k = k;
          s_shift = shift;
          s_zero = zero;
        }
        __syncthreads();
        const int k = s_k, zero = s_zero;
        const double shift = s_shift;
        total += k;
        const T sw = W::from_d(shift);
        // x back from its published copy (so it holds no registers during the residual)
#pragma unroll
        for (int m = 0; m < M; ++m) P::chunk(D0, D1, (int)(info(m).x & 0xffffu), X[m]);
        if (k == 0) {
          // converged (or zero, or stopped): the projection shift
#pragma unroll
          for (int m = 0; m < M; ++m)
#pragma unroll
            for (int z = 0; z < kRsZ; ++z) {
              if (zero) X[m][z] = W::zero();
              else if (shift != 0.0) X[m][z] = W::add(X[m][z], sw);
            }
          break;
        }
        // ---- the shift, q = r - s, and the first direction d = q / theta
        const N shn = (N)shift;
        N inv_theta;
        if constexpr (sizeof(N) == 4) inv_theta = sp.inv_theta_f;
        else inv_theta = (N)(1.0 / sp.theta);
#pragma unroll
        for (int m = 0; m < M; ++m) {
          const uint2 in = info(m);
          if (!in.x) continue;
          const int cnt = (int)(in.x >> kCnt & 7u);
          const N* const rg = s_g.r + cell(m);
          N v[kRsZ];
#pragma unroll
          for (int z = 0; z < kRsZ; ++z) {
            v[z] = N(0);
            if (z >= cnt) continue;
            Q[m][z] = rg[z * nxy] - shn;
            v[z] = Q[m][z] * inv_theta;
            X[m][z] = W::add(X[m][z], sw);
          }
          st_chunk(D0 + (in.x & 0xffffu), v);
        }
        if (!exchange(0, 1)) return;
        // ---- Chebyshev steps
        const N cfn[3] = {coef_w<N>(sp, 0), coef_w<N>(sp, 1), coef_w<N>(sp, 2)};
#pragma unroll 1
        for (int j = 1; j <= k; ++j) {
          const N* const D = (j & 1) ? D0 : D1;
          N* const Dn = (j & 1) ? D1 : D0;
          N c1, c2;
          if constexpr (sizeof(N) == 4) {
            c1 = sp.chebf[0][j - 1];
            c2 = sp.chebf[1][j - 1];
          } else {
            c1 = (N)sp.cheb[0][j - 1];
            c2 = (N)sp.cheb[1][j - 1];
          }
#pragma unroll
          for (int m = 0; m < M; ++m) {
            const uint2 in = info(m);
            if (!in.x) continue;
            const int o = (int)(in.x & 0xffffu);
            const auto c = ld_chunk(D + o), l = ld_chunk(D + o - kRsZ), r = ld_chunk(D + o + kRsZ);
            const auto fr = ld_chunk(D + o - pr), bk = ld_chunk(D + o + pr);
            N below = D[in.y & 0xffffu], v[kRsZ];
            const N top = D[in.y >> 16];
            N up[kRsZ] = {c.v[1], c.v[2], c.v[3], top};
            if (part) {  // the brick's last chunk ends before its fourth cell
              const int cnt = (int)(in.x >> kCnt & 7u);
              if (cnt == 1) up[0] = top;
              if (cnt == 2) up[1] = top;
              if (cnt == 3) up[2] = top;
            }
#pragma unroll
            for (int z = 0; z < kRsZ; ++z) {
              const N cur = c.v[z], above = up[z];
              const N sx = (l.v[z] - cur) + (r.v[z] - cur);
              const N sy = (fr.v[z] - cur) + (bk.v[z] - cur);
              N lap = cfn[0] * sx + cfn[1] * sy;
              if constexpr (GR) {
                const N* const cz = s_cz + 2 * ((int)(in.x >> kZc) * kRsZ + z);
                const N tm = cz[0] * (below - cur), tp = cz[1] * (above - cur);
                lap = zz ? lap + (tm + tp) : (lap + tm) + tp;
              } else {
                lap = lap + cfn[2] * ((below - cur) + (above - cur));
              }
              Q[m][z] = Q[m][z] - (cur - lap);
              v[z] = c1 * cur + c2 * Q[m][z];
              X[m][z] = W::add_n(X[m][z], cur);
              below = cur;
            }
            if (j < k) st_chunk(Dn + o, v);
          }
          if (j < k && !exchange(j & 1, 1)) return;
        }
        __syncthreads();  // every reader of the directions is done before x is published
      }
      if (rank == 0 && tid == 0 && md.iters) atomicAdd(md.iters + f, total);
    }
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const int cnt = count(m);
      if (!cnt) continue;
      T* const xg = s_g.x + cell(m);
#pragma unroll
      for (int z = 0; z < kRsZ; ++z)
        if (z < cnt) xg[z * nxy] = X[m][z];
    }
  }
}

__global__ void k_bar_reset(Ctl* ctl) {
  ctl->bar_count = 0u;
  ctl->bar_gen = 0u;
}

template <class T>
size_t word() {
  return sizeof(T);
}

template <class T, bool GR>
int launch_impl(const SmoothBatchDev& a, int max_blocks, cudaStream_t s) {
  int dev = 0;
  cudaGetDevice(&dev);
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_smooth<T, GR>, kThreads, 0);
  if (per_sm < 1) return -3;
  if (per_sm > smooth_blocks_per_sm<T>()) per_sm = smooth_blocks_per_sm<T>();
  int G = nsm * per_sm;
  if (G > max_blocks) G = max_blocks;
  if (G < 1) G = 1;
  k_bar_reset<<<1, 1, 0, s>>>(a.ctl);
  SmoothBatchDev args = a;
  void* p[] = {&args};
  cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_smooth<T, GR>, dim3(G), dim3(kThreads), p, 0, s);
  return e == cudaSuccess ? 0 : -3;
}

size_t align256(size_t n) { return (n + 255) & ~(size_t)255; }

}  // namespace

int64_t smooth_units(int64_t C) { return (C + kThreads - 1) / kThreads; }

bool smooth_beyond_cluster(int64_t C) { return C > (int64_t)kClMaxCta * kClCells; }

// What the direction arrays lack of 24 MB for meshes beyond a cluster (150 CTAs of 160 KB).  The
// small meshes of the FP64 form: seven groups of 21 CTAs use 0.35 MB and 30 to 60 KB for each
// cell of a brick's face, up to 4 MB more than their arrays hold; flat ones more, and take
// another cut.
size_t smooth_tag_bytes(int form, int64_t C) {
  const size_t have = 2 * align256((size_t)kMaxF * C * (form == FORM_FP64 ? 8 : 4)), want = 24 << 20;
  if (smooth_beyond_cluster(C)) return have < want ? want - have : 0;
  if (form != FORM_FP64) return 0;
  const double face = std::cbrt((double)C / 21 * (double)C / 21);
  return align256((size_t)std::min(0.4e6 + 60e3 * face, (double)kSmoothTagBytes - 256));
}

size_t smooth_tag_room(int form, int64_t C) {
  const size_t lack = smooth_tag_bytes(form, C);
  return lack ? lack + 2 * align256((size_t)kMaxF * C * (form == FORM_FP64 ? 8 : 4)) : 0;
}

size_t smooth_mesh_bytes(int form, int64_t C, int nf, int scheme, bool own_tags) {
  const size_t w = form == FORM_PLAIN ? 4 : 8;             // wide word
  const size_t n = form == FORM_FP64 ? 8 : 4;              // narrow word
  const size_t wide = align256((size_t)nf * C * w);        // b, and x^{m-1} for BDF2
  return (scheme == TAU_BDF2 ? 2 : 1) * wide + 3 * align256((size_t)kMaxF * C * n) +
         (own_tags ? smooth_tag_bytes(form, C) : 0) + align256((size_t)smooth_units(C) * kMaxF * kQ * 8) + 256;
}

size_t smooth_work_bytes(int form, int64_t C, int nf, int scheme, bool own_tags) {
  return align256(smooth_mesh_bytes(form, C, nf, scheme, own_tags)) + smooth_batch_bytes(1, smooth_units(C));
}

int launch_smooth(int form, const DevParams& P, void* phi, const void* guess, int nf, void* work,
                  const DevState& st, int* iters_dev, double rtol, int max_iter, int n_tau,
                  int scheme, const double coef[3], const SmoothZ* z, cudaStream_t s,
                  long long spin_limit, bool resident, const SmoothTags& tags) {
  SmoothMesh m{};
  m.phi = phi;
  m.guess = guess;
  m.work = work;
  m.tags = tags;
  m.iters = iters_dev;
  m.C = P.C;
  m.nf = nf;
  for (int k = 0; k < 3; ++k) {
    m.nc[k] = P.nc[k];
    m.per[k] = P.periodic[k];
    m.coef[k] = coef[k];
  }
  if (z) m.z = *z;
  void* batch = (char*)work + align256(smooth_mesh_bytes(form, P.C, nf, scheme, tags.own));
  return launch_smooth_batch(form, &m, 1, nf, batch, rtol, max_iter, n_tau, scheme, st.ctl,
                             1 << 30, s, spin_limit, nullptr, resident);
}

size_t smooth_batch_bytes(int64_t B, int64_t U) {
  return 2 * align256((size_t)B * sizeof(SmoothMeshDev)) + align256((size_t)U * 4) +
         align256((size_t)B * sizeof(MeshState)) + 256;
}

// Spectrum [1, lmax] of A = I - sum_a coef_a L_a (lmax <= 1 + 4 sum_a coef_a by
// Gershgorin; on a graded z mesh the z term is 2 max_k (c-_k + c+_k), zmax > 0) and
// the Chebyshev coefficients of steps 1..kMaxStepsRound (the same in every round):
// rho_1 = 1 / sigma1, rho' = 1 / (2 sigma1 - rho), c1 = rho' rho, c2 = 2 rho' / delta.
static void smooth_spec(const double coef[3], double scale, double zmax, SmoothSpec* sp) {
  for (int k = 0; k < 3; ++k) {
    sp->coef[k] = scale * coef[k];
    sp->coef_hi[k] = (float)sp->coef[k];
    sp->coef_lo[k] = (float)(sp->coef[k] - (double)sp->coef_hi[k]);
  }
  double lmax = zmax > 0.0 ? 1.0 + 4.0 * (sp->coef[0] + sp->coef[1]) + 2.0 * zmax
                           : 1.0 + 4.0 * (sp->coef[0] + sp->coef[1] + sp->coef[2]);
  if (lmax < 1.0 + 1e-12) lmax = 1.0 + 1e-12;
  sp->theta = 0.5 * (lmax + 1.0);
  sp->delta = 0.5 * (lmax - 1.0);
  sp->sigma1 = sp->theta / sp->delta;
  sp->inv_theta_f = (float)(1.0 / sp->theta);
  const double sq = std::sqrt(lmax);
  sp->sig = (sq - 1.0) / (sq + 1.0);
  double rho = 1.0 / sp->sigma1;
  for (int j = 0; j < kMaxStepsRound; ++j) {
    const double rho_new = 1.0 / (2.0 * sp->sigma1 - rho);
    sp->cheb[0][j] = rho_new * rho;
    sp->cheb[1][j] = 2.0 * rho_new / sp->delta;
    sp->chebf[0][j] = (float)sp->cheb[0][j];
    sp->chebf[1][j] = (float)sp->cheb[1][j];
    rho = rho_new;
  }
}

static void smooth_mesh_layout(int form, int scheme, const SmoothMesh& in, SmoothMeshDev* out) {
  const size_t w = form == FORM_PLAIN ? 4 : 8;
  const size_t n = form == FORM_FP64 ? 8 : 4;
  char* p = (char*)in.work;
  SmoothMeshDev& m = *out;
  std::memset(&m, 0, sizeof(m));
  m.x = in.phi;
  m.guess = in.guess;
  m.b = p;  // [nf][C] wide
  p += align256((size_t)in.nf * in.C * w);
  if (scheme == TAU_BDF2) {
    m.xp = p;  // [nf][C] wide
    p += align256((size_t)in.nf * in.C * w);
  }
  const size_t nar = align256((size_t)kMaxF * in.C * n);  // [C][8] narrow
  m.q = p;
  m.d[0] = p + nar;
  m.d[1] = p + 2 * nar;
  // tagged words from d[0] on: a resident launch has no other use for the direction arrays
  const size_t extra = in.tags.own ? smooth_tag_bytes(form, in.C) : 0;
  m.tags = m.d[0];
  m.tag_bytes = (int64_t)(2 * nar + extra);
  if (!in.tags.own && in.tags.n > m.tag_bytes) {
    m.tags = in.tags.p;
    m.tag_bytes = in.tags.n;
  }
  p += 3 * nar + extra;
  m.part = (double*)p;
  m.iters = in.iters;
  m.C = in.C;
  m.nu = smooth_units(in.C);
  for (int k = 0; k < 3; ++k) {
    m.nc[k] = in.nc[k];
    m.per[k] = in.per[k];
  }
  auto magic = [](uint64_t d) -> uint64_t { return d <= 1 ? 0 : ~(uint64_t)0 / d + 1; };
  m.div_x = magic((uint64_t)in.nc[0]);
  m.div_xy = magic((uint64_t)in.nc[0] * (uint64_t)in.nc[1]);
  m.z = in.z;
  const bool gr = in.z.cz[0] != nullptr;
  smooth_spec(in.coef, 1.0, gr ? in.z.zmax[0] : 0.0, &m.sp[0]);
  smooth_spec(in.coef, scheme == TAU_BDF2 ? 2.0 / 3.0 : 1.0, gr ? in.z.zmax[scheme == TAU_BDF2 ? 1 : 0] : 0.0,
              &m.sp[1]);
}

namespace {

template <class T, bool GR>
int launch_cluster(const SmoothBatchDev& a, int csize, cudaStream_t s) {
  using N = typename Wide<T>::N;
  const size_t smem = kClSmem;
  if (cudaFuncSetAttribute(k_smooth_cl<T, GR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return -3;
  if (csize > 8 && cudaFuncSetAttribute(k_smooth_cl<T, GR>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return -3;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(csize * 64);
  int ncl = 0;
  if (cudaOccupancyMaxActiveClusters(&ncl, (void*)k_smooth_cl<T, GR>, &cfg) != cudaSuccess || ncl < 1) return -3;
  // a cluster an item: clusters beyond the resident ones start as others end, so long and
  // short fields, and launches of other cluster sizes beside this one, share the SMs
  cfg.gridDim = dim3((unsigned)(csize * a.B * a.nf));
  return cudaLaunchKernelEx(&cfg, k_smooth_cl<T, GR>, a) == cudaSuccess ? 0 : -3;
}

// Cluster plan of a mesh (whole z-planes per CTA, <= kClCells cells each), or
// csize 0 when the mesh does not fit the cluster solver.
void cluster_plan(int form, const SmoothMeshDev& m, int* csize, int* planes) {
  *csize = 0;
  *planes = 0;
  if (form == FORM_FP64) return;
  const int64_t nxy = (int64_t)m.nc[0] * m.nc[1];
  // per CTA: P planes of x (8 B) and three narrow words (4 B)
  const int64_t room = (int64_t)kClSmem / 4;  // in 4-byte words
  if (room < 5 * nxy) return;
  int pmax = (int)(room / (5 * nxy));
  if ((int64_t)pmax * nxy > kClCells) pmax = (int)(kClCells / nxy);
  if (pmax < 1) return;
  const int nz = m.nc[2];
  int cs = (nz + pmax - 1) / pmax;
  if (cs > kClMaxCta) return;
  const int p = (nz + cs - 1) / cs;
  cs = (nz + p - 1) / p;  // every CTA gets at least one plane
  *csize = cs;
  *planes = p;
}

// How the resident solver cuts a mesh into px x py x pz bricks (G CTAs), or G = 0 when no
// cut fits, for nf fields.  No bit of a result depends on the cut.
struct RsPlan {
  int G = 0, px = 0, py = 0, pz = 0, groups = 0;
  int chunks = 0;             // of a thread
  size_t smem = 0, halo = 0;  // dynamic shared memory; halo words of a CTA and channel
  double us = 0.0;            // predicted time of a step of all fields
};

// Bytes of a group's tagged words: the sums, and for each CTA two parities of the halo words
// (the double-float form has two channels of 4-byte words, FP64 one of 8 bytes).
size_t rs_tag_bytes(int G, size_t halo) { return rs_sum_words(G) * 8 + (size_t)G * halo * 4 * 8; }

// Fields of FP32 words that a thread's few chunks hold go to one CTA: no exchange at all,
// and many meshes in one launch.
bool rs_one_cta(int form, const SmoothMeshDev& m) {
  return form != FORM_FP64 &&
         (int64_t)m.nc[0] * m.nc[1] * ((m.nc[2] + kRsZ - 1) / kRsZ) <= kRsThreads * kRsChunks;
}

RsPlan rs_plan(int form, const SmoothMeshDev& m, int nf, int nsm) {
  const size_t word = form == FORM_FP64 ? 8 : 4;
  const int nx = m.nc[0], ny = m.nc[1], nz = m.nc[2];
  const int T = kRsThreads, top = T * (word == 8 ? kRsChunks : kRsChunksBig);
  RsPlan best;
  double best_cost = 1e300;
  auto consider = [&](int px, int py, int pz, int groups) {
    if (px < 1 || px > nx || py > ny || pz > nz) return;
    const int G = px * py * pz;
    if (G == 1 && !rs_one_cta(form, m)) return;  // a group (rs_sums); on a device of few SMs
    const int64_t bx = (nx + px - 1) / px, by = (ny + py - 1) / py, bz = (nz + pz - 1) / pz;
    const int64_t nzc = (bz + kRsZ - 1) / kRsZ, nch = bx * by * nzc;
    if (nch > top) return;
    const bool zcut = pz > 1 || m.per[2];
    const int64_t words = (nzc * (by + 2) * ((bx + 2) | 1) * kRsZ + (zcut ? 2 * bx * by : 0) + 3) / 4 * 4;
    const int64_t nu = 2 * nzc * (bx + by) + (zcut ? 2 * bx * by : 0);
    const size_t smem = (2 * (size_t)words + 2 * (size_t)nzc * kRsZ) * word + (size_t)nu * 12 +
                        (G == 1 ? m.C * 4 : 0);
    // a chunk's word holds 16 bits of index and 11 of its place along z
    if (smem > kRsSmem || words > 0xffff || nzc > 2000) return;
    const size_t halo = 2 * (size_t)(nzc * kRsZ * (bx + by) + (zcut ? bx * by : 0));
    // time of a step, in microseconds, fitted to measured cuts of 128 x 64 x 128 and
    // 256 x 128 x 64 meshes: 0.45 for every 512 chunks (FP64: by the cells, its pipe is
    // the limit); an exchange's latency, its halo chunks and its plane words (tagged words
    // cost most: they fill L2's write path)
    const int chunks = (int)((nch + T - 1) / T);
    const double units = 2.0 * (double)(nzc * (bx + by)), planes = zcut ? 2.0 * (double)(bx * by) : 0.0;
    double t = word == 8 ? 0.006 * (double)(nch * kRsZ) : 0.45 * chunks;
    if (G > 1) {
      if ((int64_t)rs_tag_bytes(G, halo) * groups > m.tag_bytes) return;
      t += 1.5 + 0.0018 * units + 0.00015 * planes;
    }
    const double cost = t * ((nf + groups - 1) / groups);  // waves of the fields
    if (cost < best_cost) {
      best_cost = cost;
      best.G = G;
      best.px = px;
      best.py = py;
      best.pz = pz;
      best.groups = groups;
      best.chunks = chunks;
      best.smem = smem;
      best.halo = halo;
      best.us = cost;
    }
  };
  if (rs_one_cta(form, m)) {
    consider(1, 1, 1, 1);
    if (best.G) return best;
  }
  // for every number of groups at once, the largest groups
  for (int g = 1; g <= nf; ++g) {
    const int gmax = nsm / g < kRsMaxGroup ? nsm / g : kRsMaxGroup;
    for (int pz = 1; pz <= 40 && pz <= gmax; ++pz)
      for (int py = 1; py * pz <= gmax; ++py) consider(gmax / (py * pz), py, pz, g);
  }
  return best;
}

// Which FP64 meshes of a batch share a launch of the streaming solver (plan.G = 0) and which
// have the chip to themselves one after the other.  In microseconds a step, fitted to
// ensembles of equal beds, seven fields: the streaming solver takes 2 + 21 for every unit an SM has,
// one at least; a mesh on chip what its plan says and 3 for each wave of its fields.  Small
// meshes leave the chip to the latency of the exchange: 256 beds of 8^3 cells 178 ms on
// chip, 10.4 streamed, 64 of 16^3 43.0 and 17.2, 8 of 19 x 15 x 31 6.4 and 5.4; 2 of those
// 1.7 and 5.4, 4 of 48^3 17.4 and 28.7.  Small meshes are not planned where a bound of their time, their
// cells over the whole chip and the latency, settles it.
template <class Item>
void fp64_batch_plans(std::vector<Item>& items, int nf, int nsm) {
  auto stream_us = [&](int64_t units) { return 2.0 + 21.0 * std::max(1.0, (double)units / nsm); };
  auto plan = [&](Item& it) {
    it.pl = rs_plan(FORM_FP64, it.m, nf, nsm);
    return it.pl.G ? it.pl.us + 3.0 * ((nf + it.pl.groups - 1) / it.pl.groups) : 1e300;
  };
  std::vector<Item*> rest;  // not worth the chip beside a streaming launch that is full
  double sum = 0.0;
  int64_t units = 0;
  std::vector<Item*> open;  // of those, not planned yet
  for (Item& it : items) {
    const double share = 21.0 * (double)it.m.nu / nsm, bound = 4.5 + 0.006 * (double)it.m.C * nf / nsm;
    const double t = bound < share ? plan(it) : bound;
    if (bound >= share) open.push_back(&it);
    if (t < share) continue;
    rest.push_back(&it);
    sum += t;
    units += it.m.nu;
  }
  if (rest.empty()) return;
  if (sum < stream_us(units)) {
    for (Item* it : open) sum += plan(*it) - (4.5 + 0.006 * (double)it->m.C * nf / nsm);
    if (sum < stream_us(units)) return;
  }
  for (Item* it : rest) it->pl = RsPlan{};
}

// The fields of one mesh over the groups of a cooperative launch (every CTA resident, one
// per SM), or the fields of many meshes of one CTA each, an ordinary launch.
template <class T, bool GR>
int launch_rs(const SmoothBatchDev& a, const RsPlan& pl, const SmoothMeshDev& m, int nsm, cudaStream_t s) {
  auto* kern = k_smooth_rs<T, GR, kRsChunks>;
  if constexpr (!std::is_same<T, double>::value)
    if (pl.chunks > kRsChunks) kern = k_smooth_rs<T, GR, kRsChunksBig>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRsSmem) != cudaSuccess)
    return -3;
  if (pl.G == 1) {
    const int64_t items = (int64_t)a.B * a.nf;
    kern<<<(unsigned)(items < nsm ? items : nsm), kRsThreads, pl.smem, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
  }
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kRsThreads, pl.smem) != cudaSuccess) return -3;
  if ((int64_t)per_sm * nsm < (int64_t)pl.groups * pl.G) return -3;
  // no tagged word of an earlier launch may pass for this one's: exchanges count from 1
  const size_t bytes = rs_tag_bytes(pl.G, pl.halo) * pl.groups;
  if (cudaMemsetAsync(m.tags, 0, bytes, s) != cudaSuccess) return -3;
  SmoothBatchDev args = a;
  void* p[] = {&args};
  return cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)(pl.groups * pl.G)), dim3(kRsThreads), p, pl.smem, s) ==
                 cudaSuccess
             ? 0
             : -3;
}

}  // namespace

int launch_smooth_batch(int form, const SmoothMesh* meshes, int B, int nf, void* batch_work,
                        double rtol, int max_iter, int n_tau, int scheme, Ctl* ctl,
                        int max_blocks, cudaStream_t s, long long spin_limit, const SmoothSide* side,
                        bool resident) {
  if (B < 1 || B > kMaxBeds || nf < 1 || nf > kMaxF || (scheme != TAU_EULER && scheme != TAU_BDF2))
    return -1;
  // every mesh of a batch is graded or none is (one kernel instantiation per launch)
  const bool gr = meshes[0].z.cz[0] != nullptr;
  for (int b = 1; b < B; ++b)
    if ((meshes[b].z.cz[0] != nullptr) != gr) return -1;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (nsm > max_blocks) nsm = max_blocks;
  // FP32 words: fields that fit one CTA take the resident solver (10 x 10 x 20, seven fields:
  // 440 us in a cluster solver's CTA, 250 here), larger meshes that fit a cluster's shared
  // memory the cluster solver (one launch for every mesh of a cluster size), still larger
  // ones the resident solver again where a cut of the whole chip fits, else the streaming grid
  // solver.  In FP64 there is no cluster solver (several meshes: fp64_batch_plans).  No bit of a
  // result depends on the choice.
  struct Item {
    SmoothMeshDev m;
    RsPlan pl;
  };
  std::vector<SmoothMeshDev> mg, mc;
  std::vector<Item> mr;
  std::vector<Item> all(B);
  for (int b = 0; b < B; ++b) {
    Item& it = all[b];
    smooth_mesh_layout(form, scheme, meshes[b], &it.m);
    cluster_plan(form, it.m, &it.m.cl_size, &it.m.cl_planes);
    if (resident && (it.m.cl_size == 0 ? form != FORM_FP64 || B == 1 : rs_one_cta(form, it.m)))
      it.pl = rs_plan(form, it.m, nf, nsm);
  }
  if (resident && form == FORM_FP64 && B > 1) fp64_batch_plans(all, nf, nsm);
  for (Item& it : all) {
    if (it.m.cl_size > 0 && it.pl.G != 1) {
      mc.push_back(it.m);
    } else if (it.pl.G > 0) {
      it.m.rs_G = it.pl.G;
      it.m.rs_px = it.pl.px;
      it.m.rs_py = it.pl.py;
      it.m.rs_pz = it.pl.pz;
      mr.push_back(it);
    } else {
      mg.push_back(it.m);
    }
  }
  // cluster meshes grouped by cluster size (one launch per size, the largest first: the
  // small clusters fit between them), resident ones with the
  // meshes of one CTA first (one launch for all)
  std::stable_sort(mc.begin(), mc.end(),
                   [](const SmoothMeshDev& x, const SmoothMeshDev& y) { return x.cl_size > y.cl_size; });
  std::stable_sort(mr.begin(), mr.end(), [](const Item& x, const Item& y) { return (x.pl.G == 1) > (y.pl.G == 1); });
  char* p = (char*)batch_work;
  SmoothBatchDev a{};
  a.nf = nf;
  a.rtol2 = rtol * rtol;
  a.max_iter = max_iter;
  a.n_tau = n_tau;
  a.scheme = scheme;
  a.ctl = ctl;
  a.spin_limit = spin_limit > 0 ? spin_limit : 1;
  SmoothMeshDev* tab_g = (SmoothMeshDev*)p;
  p += align256((size_t)B * sizeof(SmoothMeshDev));
  SmoothMeshDev* tab_c = (SmoothMeshDev*)p;
  p += align256((size_t)B * sizeof(SmoothMeshDev));
  int rc = 0;
  if (!mc.empty() || !mr.empty()) {
    std::vector<SmoothMeshDev> tab(mc);
    for (const auto& it : mr) tab.push_back(it.m);
    if (cudaMemcpyAsync(tab_c, tab.data(), tab.size() * sizeof(SmoothMeshDev), cudaMemcpyHostToDevice, s) != cudaSuccess)
      return -3;
    // The launches of the cluster sizes run side by side where there are streams for it: a
    // GPC's SMs hold one cluster of 11 CTAs and one of 8 at once, and no launch waits
    // for the last cluster of another (48 beds of 16^3 to 48^3 cells, seven fields: 9.8 ms
    // one after the other, 8.6 side by side).
    const bool fork = side && !mc.empty() && mc.front().cl_size != mc.back().cl_size;
    if (fork && cudaEventRecord(side->fork, s) != cudaSuccess) return -3;
    unsigned used = 0;  // side streams with work
    int lane = 0;
    for (size_t i0 = 0; i0 < mc.size();) {
      size_t i1 = i0;
      while (i1 < mc.size() && mc[i1].cl_size == mc[i0].cl_size) ++i1;
      cudaStream_t on = s;
      if (fork) {
        on = side->s[lane];
        if (!(used >> lane & 1u) && cudaStreamWaitEvent(on, side->fork, 0) != cudaSuccess) return -3;
        used |= 1u << lane;
        lane = (lane + 1) % kSmoothSides;
      }
      SmoothBatchDev c = a;
      c.mesh = tab_c + i0;
      c.B = (int32_t)(i1 - i0);
      if (gr)
        rc = form == FORM_SPLIT ? launch_cluster<dd, true>(c, mc[i0].cl_size, on)
                                : launch_cluster<float, true>(c, mc[i0].cl_size, on);
      else
        rc = form == FORM_SPLIT ? launch_cluster<dd, false>(c, mc[i0].cl_size, on)
                                : launch_cluster<float, false>(c, mc[i0].cl_size, on);
      if (rc) {
        // a device without this cluster shape: these meshes take the streaming solver
        cudaGetLastError();
        for (size_t i = i0; i < i1; ++i) {
          SmoothMeshDev m = mc[i];
          m.cl_size = m.cl_planes = 0;
          mg.push_back(m);
        }
        rc = 0;
      }
      i0 = i1;
    }
    for (int k = 0; k < kSmoothSides; ++k)
      if (used >> k & 1u)
        if (cudaEventRecord(side->join[k], side->s[k]) != cudaSuccess || cudaStreamWaitEvent(s, side->join[k], 0) != cudaSuccess)
          return -3;
    for (size_t i0 = 0; i0 < mr.size();) {
      // every mesh of one CTA in one launch, the larger ones one by one
      size_t i1 = i0 + 1;
      RsPlan pl = mr[i0].pl;
      for (; pl.G == 1 && i1 < mr.size() && mr[i1].pl.G == 1; ++i1) {
        pl.smem = std::max(pl.smem, mr[i1].pl.smem);
        pl.chunks = std::max(pl.chunks, mr[i1].pl.chunks);
      }
      SmoothBatchDev c = a;
      c.mesh = tab_c + mc.size() + i0;
      c.B = (int32_t)(i1 - i0);
      c.rs_G = pl.G;
      if (form == FORM_SPLIT)
        rc = gr ? launch_rs<dd, true>(c, pl, mr[i0].m, nsm, s) : launch_rs<dd, false>(c, pl, mr[i0].m, nsm, s);
      else if (form == FORM_PLAIN)
        rc = gr ? launch_rs<float, true>(c, pl, mr[i0].m, nsm, s) : launch_rs<float, false>(c, pl, mr[i0].m, nsm, s);
      else
        rc = gr ? launch_rs<double, true>(c, pl, mr[i0].m, nsm, s) : launch_rs<double, false>(c, pl, mr[i0].m, nsm, s);
      if (rc) {
        cudaGetLastError();
        for (size_t i = i0; i < i1; ++i) {
          mg.push_back(mr[i].m);
          mg.back().cl_size = mg.back().cl_planes = 0;
        }
        rc = 0;
      }
      i0 = i1;
    }
  }
  if (!mg.empty()) {
    int64_t U = 0;
    for (auto& m : mg) {
      m.u0 = U;
      U += m.nu;
    }
    std::vector<int32_t> ub(U);
    for (size_t b = 0; b < mg.size(); ++b)
      for (int64_t u = 0; u < mg[b].nu; ++u) ub[mg[b].u0 + u] = (int32_t)b;
    a.mesh = tab_g;
    a.unit_bed = (int32_t*)p;
    p += align256((size_t)U * 4);
    a.pairs = p;
    p += align256((size_t)mg.size() * sizeof(MeshState));
    a.gflag = (int32_t*)p;
    a.B = (int32_t)mg.size();
    a.U = U;
    if (cudaMemcpyAsync(tab_g, mg.data(), mg.size() * sizeof(SmoothMeshDev), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync((void*)a.unit_bed, ub.data(), U * 4, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemsetAsync(a.gflag, 0, 2 * sizeof(int32_t), s) != cudaSuccess)
      return -3;
    switch (form) {
      case FORM_SPLIT: rc = gr ? launch_impl<dd, true>(a, max_blocks, s) : launch_impl<dd, false>(a, max_blocks, s); break;
      case FORM_PLAIN: rc = gr ? launch_impl<float, true>(a, max_blocks, s) : launch_impl<float, false>(a, max_blocks, s); break;
      default: rc = gr ? launch_impl<double, true>(a, max_blocks, s) : launch_impl<double, false>(a, max_blocks, s); break;
    }
  }
  return rc;
}

}  // namespace sedi

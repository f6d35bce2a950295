// tree_sweep.cu -- the transport / relaxation / moments sweep of tree-refined
// grids in FP32 storage (quadtrees and octrees, reading C28; bodies in the finest
// level, C29).
//
// Same arithmetic as tree_sweep_kernel in kernels.cu (which takes FP64 storage):
// finite volumes on the leaves, the van Leer slope of a leaf along an axis from
// the value on each side over the centre distances, the upwind leaf's face
// value, the mean of the face values over a side shared with finer leaves.
// Organised for GB300 around vectors of 16 bytes:
//
//   * 64 threads take a leaf, two leaves a block; a thread takes 16 bytes of a
//     row at a time (four velocities of an octree, the (h, b) pairs of two of a
//     quadtree), so every gather is a 16-byte load of consecutive addresses
//     across a warp and the faces run on packed FP32 pairs;
//   * the velocities of tree cases are stored grouped by orthant, so a vector has
//     one upwind side per axis and the structure of its stencil (levels,
//     finer leaves, ghosts, domain edges) is a branch the whole vector
//     shares; the few vectors that straddle two orthants (or end in padding)
//     are formed once per orthant and blended;
//   * a leaf with one fluid leaf of its own level on every side takes the
//     gather-first path: the leaf, its 2 D neighbours and the D far neighbours
//     upwind, all loads issued before any arithmetic (the upwind leaf's value
//     and its side towards the leaf are the leaf's side value and own value);
//   * those leaves and the others are two launches, each with the registers and
//     the shared tables that it needs.  The stencil tables are built once on the
//     host (tree.cpp) and read into shared memory per block.
//
// What bounds it: the latency of the gathers (the stalls on them are 7 of 12 warps
// per issue) and their L2 traffic (58% of its rate for the regular leaves).
// Measured per step: octree sphere of 46,584 leaves x 20^3 velocities 2.80 ms, where
// scalar gathers had taken 6.34; Ma 5 cylinder of 69,148 leaves x 60^2 1.55 ms (1.77).
// Before the relaxation came after the fluxes, at 2.85 / 1.54: both kinds of leaf in
// one launch, 80 registers: 2.91 / 1.63; blocks of four leaves, four per SM: 2.95 / 1.62; eight and
// nine blocks of two: 3.01 / 1.62 and 3.79 / 1.85; pieces of one orthant per warp
// from a table: 3.13 / 2.14; 32 threads per leaf, eight leaves: 3.12 / 1.83.
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "ctx.h"
#include "tma_sync.cuh"

namespace ibdvm {
namespace {

using namespace dev;

constexpr int kTreeThreads = 64; // threads of a leaf
constexpr int kTreeLeaves = 2;   // leaves of a block
constexpr int kTreeBlocks = 7;   // blocks per SM (72 registers: 14 warps more than at 128 hide the gathers better)
constexpr float kLog2e = 1.442695040888963407f;

struct Tree32Args {
  const float *__restrict__ f;
  float *__restrict__ fn;
  const float *__restrict__ mac;
  const float *__restrict__ xi, *__restrict__ w, *__restrict__ finf, *__restrict__ lval;
  double *__restrict__ part;       // [nchunk][NM][ncell]
  const int4 *__restrict__ sti;    // [leaf][entries][ints / 4]: stencil rows and the mutual flag
  const double2 *__restrict__ stg; // [leaf][entries][2]: 1/d-, 1/d+, h, 1/h (own entries)
  const int4 *__restrict__ lrec;   // [leaf][2]: leaves on the sides, regular flag, fluid flag
  const int *__restrict__ sched;
  long long ncell;
  int nv, nvp, per, nleaf; // per: velocities of a chunk; nleaf: leaves of this launch (sched)
  float dt;
  int qb[7]; // first stored position of the orthants 1 .. 2^D - 1 (bit a: component a < 0)
};

// the stencil of one cell along one axis (see tree_sweep_kernel)
template <int NF> struct __align__(16) Stencil {
  const float *c, *m[NF], *p[NF];
  float rdm, rdp, h;
  int mut;
};

// 16 bytes of a row as two packed pairs
struct V4 {
  float2 l, h;
};
__device__ __forceinline__ V4 ld4(const float *r, int e) {
  const float4 t = __ldg(reinterpret_cast<const float4 *>(r + e));
  return {make_float2(t.x, t.y), make_float2(t.z, t.w)};
}
__device__ __forceinline__ V4 operator-(V4 a, V4 b) { return {sub2(a.l, b.l), sub2(a.h, b.h)}; }
__device__ __forceinline__ V4 operator+(V4 a, V4 b) { return {__fadd2_rn(a.l, b.l), __fadd2_rn(a.h, b.h)}; }
__device__ __forceinline__ V4 operator*(V4 a, float s) {
  return {__fmul2_rn(a.l, dup(s)), __fmul2_rn(a.h, dup(s))};
}
__device__ __forceinline__ V4 fma4(float2 cl, float2 ch, V4 a, V4 b) {
  return {__ffma2_rn(cl, a.l, b.l), __ffma2_rn(ch, a.h, b.h)};
}
__device__ __forceinline__ V4 vl4(V4 a, V4 b) { return {vl_half2(a.l, b.l), vl_half2(a.h, b.h)}; }

// the value on one side of a cell as its slope sees it: the neighbour's, or the
// mean of the NF finer neighbours'
template <int NF> __device__ __forceinline__ V4 side4(const float *const *r, int e) {
  V4 v = ld4(r[0], e);
  if (!r[1]) return v;
#pragma unroll
  for (int j = 1; j < NF; ++j) v = v + ld4(r[j], e);
  return v * (1.f / NF);
}
// the face value on side s (+1, -1) of a cell of value f with side values m and p
template <int NF> __device__ __forceinline__ V4 face4(const Stencil<NF> &S, V4 f, V4 m, V4 p, float s) {
  const V4 v = vl4((f - m) * S.rdm, (p - f) * S.rdp);
  const float2 sh = dup(s * S.h);
  return fma4(sh, sh, v, f);
}
__device__ __forceinline__ float ex2(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void acc_add(float &a, float2 v) { a += v.x + v.y; }
__device__ __forceinline__ void acc_fma(float &a, float2 u, float2 v) { a = fmaf(u.y, v.y, fmaf(u.x, v.x, a)); }

template <int D, bool REG>
__global__ void __launch_bounds__(kTreeThreads *kTreeLeaves, kTreeBlocks) tree_sweep32_kernel(Tree32Args A) {
  constexpr int NC = (D == 2) ? 2 : 1;
  constexpr int NM = (D == 2) ? 9 : 14;
  constexpr int NF = 1 << (D - 1); // leaves at most beyond a face
  constexpr int NS = 2 * D;        // sides
  constexpr int E = tree_entries(D), EI = tree_entry_ints(D);
  constexpr int VE = 4 / NC;       // velocities of a vector
  constexpr int W = kTreeThreads / 32; // warps of a leaf
  constexpr int NL = 8, NR = NL * W; // lanes of a warp, partial sums of a leaf, that are added in FP64
  __shared__ float red[kTreeLeaves][NR][NM];
  // per leaf: its own stencil along each axis, then the upwind neighbours'
  // along axis a, side sd (0: -, 1: +), neighbour j at D + (2a + sd) NF + j
  __shared__ Stencil<NF> st[kTreeLeaves][E];
  __shared__ float s_rh[kTreeLeaves][D]; // dt / h
  // the leaf's Shakhov parameters as packed pairs: -U, the factor of c^2 in the
  // exponent (2D, base 2: -log2(e)/T; 3D: -1/T), prefactor, q, dt/tau, the
  // Shakhov factor, 2/T (read again for every vector: registers are what
  // limits the loads in flight)
  __shared__ float2 s_c[kTreeLeaves][11];
  __shared__ float s_T[kTreeLeaves]; // T / 2
  __shared__ int rec[kTreeLeaves][8];    // leaves on side 2a + sd (0 domain edge, 1, NF, 3 a ghost), regular, fluid
  const int tx = threadIdx.x, ty = threadIdx.y;
  const long long slot = (long long)blockIdx.x * kTreeLeaves + ty;
  const bool active = slot < A.nleaf;
  const long long c = active ? A.sched[slot] : 0;
  const int chunk = blockIdx.y;
  auto row = [&](int i) -> const float * {
    return (i >= 0) ? A.f + (size_t)i * A.nvp * NC
           : (i == -2) ? A.finf
           : (i <= -3) ? A.lval + (size_t)(-3 - i) * A.nvp * NC // a ghost's value for this leaf (C29)
                       : nullptr;
  };
  if (active && tx < E) {
    const int4 *I4 = A.sti + ((size_t)c * E + tx) * (EI / 4);
    int I[EI];
#pragma unroll
    for (int q = 0; q < EI / 4; ++q) {
      const int4 v = I4[q];
      I[4 * q] = v.x;
      I[4 * q + 1] = v.y;
      I[4 * q + 2] = v.z;
      I[4 * q + 3] = v.w;
    }
    const double2 g0 = A.stg[2 * ((size_t)c * E + tx)], g1 = A.stg[2 * ((size_t)c * E + tx) + 1];
    Stencil<NF> S;
    S.c = row(I[0]);
#pragma unroll
    for (int j = 0; j < NF; ++j) {
      S.m[j] = row(I[1 + j]);
      S.p[j] = row(I[1 + NF + j]);
    }
    S.mut = I[1 + 2 * NF];
    S.rdm = (float)g0.x;
    S.rdp = (float)g0.y;
    S.h = (float)g1.x;
    st[ty][tx] = S;
    if (tx < D) s_rh[ty][tx] = A.dt * (float)g1.y;
  }
  if (active && tx >= 40 && tx < 48) rec[ty][tx - 40] = reinterpret_cast<const int *>(A.lrec)[(size_t)c * 8 + tx - 40];
  if (active && tx == 63) {
    const float *M = A.mac + c * kMac;
    const float v[11] = {-M[kU0],   -M[kU0 + 1], -M[kU0 + 2], (D == 2) ? -M[kInvT] * kLog2e : -M[kInvT],
                         M[kPre],   M[kQ0],      M[kQ0 + 1],  M[kQ0 + 2],
                         M[kDtTau], M[kShA],     2.f * M[kInvT]};
#pragma unroll
    for (int i = 0; i < 11; ++i) s_c[ty][i] = dup(v[i]);
    s_T[ty] = M[kHalfT];
  }
  __syncthreads();
  float acc[NM];
#pragma unroll
  for (int m = 0; m < NM; ++m) acc[m] = 0.f;
  if (active) {
    // -U_x, -U_y, -U_z, exponent, prefactor, q_x, q_y, q_z, dt / tau, Shakhov factor, 2 / T
    const float2 *C = s_c[ty];
    const float halfT = s_T[ty];
    const float *own = A.f + (size_t)c * A.nvp * NC;
    float *dst = A.fn + (size_t)c * A.nvp * NC;
    const int k0 = chunk * A.per, k1 = min(A.nv, k0 + A.per); // the velocities of this chunk
    auto orthant = [&](int k) {
      int o = 0;
#pragma unroll
      for (int i = 0; i < (1 << D) - 1; ++i) o += k >= A.qb[i];
      return o;
    };
    // the velocities' components about U for the vector's VE velocities, in pairs
    // (3D: two pairs; 2D: one), and their weights
    constexpr int NP = VE / 2;
    struct Vel {
      float2 x[D][NP], w[NP];
    };
    auto velocities = [&](int k, Vel &v) {
#pragma unroll
      for (int a = 0; a < D; ++a) {
        if constexpr (D == 3) {
          const float4 t = __ldg(reinterpret_cast<const float4 *>(A.xi + (size_t)a * A.nvp + k));
          v.x[a][0] = make_float2(t.x, t.y);
          v.x[a][NP - 1] = make_float2(t.z, t.w);
        } else {
          v.x[a][0] = __ldg(reinterpret_cast<const float2 *>(A.xi + (size_t)a * A.nvp + k));
        }
      }
      if constexpr (D == 3) {
        const float4 t = __ldg(reinterpret_cast<const float4 *>(A.w + k));
        v.w[0] = make_float2(t.x, t.y);
        v.w[NP - 1] = make_float2(t.z, t.w);
      } else {
        v.w[0] = __ldg(reinterpret_cast<const float2 *>(A.w + k));
      }
    };
    // the flux difference d of axis a added to n
    auto flux = [&](const Vel &v, int a, V4 d, V4 n) -> V4 {
      const float h = s_rh[ty][a];
      if constexpr (D == 3) {
        return fma4(__fmul2_rn(make_float2(fabsf(v.x[a][0].x), fabsf(v.x[a][0].y)), dup(h)),
                    __fmul2_rn(make_float2(fabsf(v.x[a][NP - 1].x), fabsf(v.x[a][NP - 1].y)), dup(h)), d, n);
      } else {
        return fma4(dup(fabsf(v.x[a][0].x) * h), dup(fabsf(v.x[a][0].y) * h), d, n);
      }
    };
    // f^{n+1} of the fluxes' increment n: relaxation towards the Shakhov equilibrium
    // (Sec. 4 reduced forms in 2D, g^S in 3D) joins the increment and f comes last,
    // so that f^{n+1} is rounded once at its own size.  After the fluxes: the
    // exponentials first cost 3 and 5% (octree, cylinder)
    auto relax = [&](const Vel &v, V4 f, V4 n) -> V4 {
      V4 eq;
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        float2 c2, cq;
        const float2 cx = __fadd2_rn(v.x[0][p], C[0]), cy = __fadd2_rn(v.x[1][p], C[1]);
        c2 = __ffma2_rn(cx, cx, __fmul2_rn(cy, cy));
        cq = __ffma2_rn(cx, C[5], __fmul2_rn(cy, C[6]));
        if constexpr (D == 3) {
          const float2 cz = __fadd2_rn(v.x[D - 1][p], C[2]);
          c2 = __ffma2_rn(cz, cz, c2);
          cq = __ffma2_rn(cz, C[7], cq);
        }
        const float2 tn = __fmul2_rn(c2, C[3]);
        // 3D: expf; a base-2 exponential of the rounded product with log2(e) errs
        // by up to c^2/T units more
        const float2 e = __fmul2_rn(C[4], (D == 3) ? make_float2(expf(tn.x), expf(tn.y)) : make_float2(ex2(tn.x), ex2(tn.y)));
        const float2 mm = __fmul2_rn(e, __fmul2_rn(cq, C[9]));
        if constexpr (D == 3) {
          const float2 g = __ffma2_rn(mm, __ffma2_rn(tn, dup(-2.f), dup(-5.f)), e);
          if (p == 0) eq.l = g;
          else eq.h = g;
        } else {
          const float2 H = __ffma2_rn(mm, __ffma2_rn(c2, C[10], dup(-4.f)), e);
          const float2 B = __fmul2_rn(dup(halfT), __ffma2_rn(mm, dup(2.f), H));
          eq.l = make_float2(H.x, B.x);
          eq.h = make_float2(H.y, B.y);
        }
      }
      return fma4(C[8], C[8], eq - f, n) + f;
    };
    // the moment sums of a vector of values n about the bulk velocity
    auto moments = [&](const Vel &v, V4 n) {
      if constexpr (D == 3) {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const float2 cx = __fadd2_rn(v.x[0][p], C[0]), cy = __fadd2_rn(v.x[1][p], C[1]);
          const float2 cz = __fadd2_rn(v.x[D - 1][p], C[2]);
          const float2 wf = __fmul2_rn(v.w[p], p == 0 ? n.l : n.h);
          const float2 xw = __fmul2_rn(cx, wf), yw = __fmul2_rn(cy, wf), zw = __fmul2_rn(cz, wf);
          const float2 c2 = __ffma2_rn(cx, cx, __ffma2_rn(cy, cy, __fmul2_rn(cz, cz)));
          const float2 e2 = __fmul2_rn(c2, wf);
          acc_add(acc[0], wf);
          acc_add(acc[1], xw);
          acc_add(acc[2], yw);
          acc_add(acc[3], zw);
          acc_fma(acc[5], cx, xw);
          acc_fma(acc[6], cy, xw);
          acc_fma(acc[7], cz, xw);
          acc_fma(acc[8], cy, yw);
          acc_fma(acc[9], cz, yw);
          acc_fma(acc[10], cz, zw);
          acc_fma(acc[11], cx, e2);
          acc_fma(acc[12], cy, e2);
          acc_fma(acc[13], cz, e2);
        }
      } else {
        const float2 cx = __fadd2_rn(v.x[0][0], C[0]), cy = __fadd2_rn(v.x[1][0], C[1]);
        const float2 c2 = __ffma2_rn(cx, cx, __fmul2_rn(cy, cy));
        const float2 wh = __fmul2_rn(v.w[0], make_float2(n.l.x, n.h.x));
        const float2 e2 = __ffma2_rn(c2, wh, __fmul2_rn(v.w[0], make_float2(n.l.y, n.h.y)));
        const float2 xw = __fmul2_rn(cx, wh), yw = __fmul2_rn(cy, wh);
        acc_add(acc[0], wh);
        acc_add(acc[1], xw);
        acc_add(acc[2], yw);
        acc_add(acc[3], e2);
        acc_fma(acc[4], cx, xw);
        acc_fma(acc[5], cy, xw);
        acc_fma(acc[6], cy, yw);
        acc_fma(acc[7], cx, e2);
        acc_fma(acc[8], cy, e2);
      }
    };
    // f^{n+1} of a vector whose velocities lie in orthant o
    auto regular = [&](int o, int k, const Vel &v) -> V4 {
      const int e = k * NC;
      const V4 f = ld4(own, e);
      V4 up[D], dn[D], far[D];
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const int sd = (o >> a) & 1; // the upwind side
        const Stencil<NF> &So = st[ty][a], &Su = st[ty][D + (2 * a + sd) * NF];
        up[a] = ld4(sd ? So.p[0] : So.m[0], e);
        dn[a] = ld4(sd ? So.m[0] : So.p[0], e);
        far[a] = ld4(sd ? Su.p[0] : Su.m[0], e);
      }
      V4 n{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
      for (int a = 0; a < D; ++a) {
        // equal spacing but towards the far leaf, which may be coarser
        const int sd = (o >> a) & 1;
        const Stencil<NF> &Su = st[ty][D + (2 * a + sd) * NF];
        const V4 b = f - up[a];
        const V4 out = f + vl4(b, dn[a] - f);
        const V4 in = up[a] + vl4((up[a] - far[a]) * ((sd ? Su.rdp : Su.rdm) * Su.h), b);
        n = flux(v, a, in - out, n);
      }
      return relax(v, f, n);
    };
    auto general = [&](int o, int k, const Vel &v) -> V4 {
      const int e = k * NC;
      const V4 f = ld4(own, e);
      V4 n{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll 1
      for (int a = 0; a < D; ++a) {
        const int sd = (o >> a) & 1;
        const float s = sd ? -1.f : 1.f;
        const Stencil<NF> &So = st[ty][a], *Su = &st[ty][D + (2 * a + sd) * NF];
        const V4 fm = side4<NF>(So.m, e), fp = side4<NF>(So.p, e);
        const V4 out = face4<NF>(So, f, fm, fp, s);
        const int nu = rec[ty][2 * a + sd];
        V4 in;
        if (nu == 0) {
          in = ld4(A.finf, e); // the halo: its value, zero slope
        } else if (nu == 3) {
          in = (ld4(Su[0].c, e) + f) * 0.5f; // a ghost upwind (C29): its link value with the one-sided slope
        } else if (nu == 1 && Su[0].mut) {
          // one upwind leaf of the leaf's level: its value and its side towards
          // the leaf are the leaf's side value and own value
          const V4 far = side4<NF>(sd ? Su[0].p : Su[0].m, e);
          in = sd ? face4<NF>(Su[0], fp, f, far, s) : face4<NF>(Su[0], fm, far, f, s);
        } else {
          // the upwind leaves' face values, each over its share of the side
          in = face4<NF>(Su[0], ld4(Su[0].c, e), side4<NF>(Su[0].m, e), side4<NF>(Su[0].p, e), s);
          if (nu > 1) {
#pragma unroll 1
            for (int j = 1; j < NF; ++j)
              in = in + face4<NF>(Su[j], ld4(Su[j].c, e), side4<NF>(Su[j].m, e), side4<NF>(Su[j].p, e), s);
            in = in * (1.f / NF);
          }
        }
        const V4 d = in - out;
        // (a is a run-time index here: the components by selection)
        if (a == 0) n = flux(v, 0, d, n);
        else if (a == 1) n = flux(v, 1, d, n);
        else n = flux(v, D - 1, d, n);
      }
      return relax(v, f, n);
    };
    auto sweep = [&](auto update) {
      for (int k = k0 + VE * tx; k < k1; k += VE * kTreeThreads) {
        asm volatile("" ::: "memory"); // the shared parameters are not kept in registers across vectors
        Vel v;
        velocities(k, v);
        int o = orthant(k);
        const int o1 = orthant(min(k + VE, A.nv) - 1);
        // a straddling vector: orthants meet in it, or padding ends it (which keeps zeros)
        const bool meet = o1 != o || k + VE > A.nv;
        V4 n{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll 1
        for (;; ++o) {
          const V4 t = update(o, k, v);
          if (!meet) {
            n = t;
            break;
          }
          auto take = [&](float &x, float y, int i) {
            const int ki = k + i / NC;
            if (ki < A.nv && orthant(ki) == o) x = y;
          };
          take(n.l.x, t.l.x, 0);
          take(n.l.y, t.l.y, 1);
          take(n.h.x, t.h.x, 2);
          take(n.h.y, t.h.y, 3);
          if (o >= o1) break;
        }
        *reinterpret_cast<float4 *>(dst + k * NC) = make_float4(n.l.x, n.l.y, n.h.x, n.h.y);
        moments(v, n);
      }
    };
    if constexpr (REG) {
      sweep(regular);
    } else if (rec[ty][NS + 1] == 0) {
      // a solid leaf (C29): not updated; the moments of its stored values
      for (int k = k0 + VE * tx; k < k1; k += VE * kTreeThreads) {
        Vel v;
        velocities(k, v);
        moments(v, ld4(own, k * NC));
      }
    } else {
      sweep(general);
    }
  }
  // the moment sums of each leaf over its 64 threads (two warps): FP32 down to
  // NL lanes a warp, the largest partial sums in FP64 (in 3D the sum of w c^2 f
  // is the trace).  Random error of the density on a 20^3-velocity octree with all
  // sums of a warp in FP32 / with 2, 8 and 32 lanes in FP64: 3.4, 2.6, 1.8 and 1.5e-8
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    if (D == 3 && m == 4) continue;
    float v = acc[m];
#pragma unroll
    for (int o = 16; o >= NL; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((tx & 31) < NL) red[ty][NL * (tx >> 5) + (tx & 31)][m] = v;
  }
  __syncthreads();
  if (tx < 32) { // half of the partial sums in lanes m, half in 16 + m
    const int m = min(tx & 15, NM - 1), r0 = (tx >> 4) * (NR / 2);
    double s[NR / 2];
#pragma unroll
    for (int r = 0; r < NR / 2; ++r) s[r] = (double)red[ty][r0 + r][m];
#pragma unroll
    for (int n = NR / 4; n > 0; n >>= 1)
#pragma unroll
      for (int r = 0; r < n; ++r) s[r] += s[r + n];
    double v = s[0] + __shfl_xor_sync(0xffffffffu, s[0], 16);
    if constexpr (D == 3) {
      const double t = __shfl_sync(0xffffffffu, v, 5) + __shfl_sync(0xffffffffu, v, 8) + __shfl_sync(0xffffffffu, v, 10);
      if (tx == 4) v = t;
    }
    if (active && tx < NM) A.part[((size_t)chunk * NM + tx) * A.ncell + c] = v;
  }
}

} // namespace

cudaError_t tree_sweep32_launch(ibdvm_ctx *ctx) {
  Tree32Args A{};
  A.f = static_cast<const float *>(ctx->f[ctx->cur]);
  A.fn = static_cast<float *>(ctx->f[1 - ctx->cur]);
  A.mac = static_cast<const float *>(ctx->mac);
  A.xi = static_cast<const float *>(ctx->xiT);
  A.w = static_cast<const float *>(ctx->wT);
  A.finf = static_cast<const float *>(ctx->finf);
  A.lval = static_cast<const float *>(ctx->lval);
  A.part = ctx->part;
  A.sti = reinterpret_cast<const int4 *>(ctx->tree_sti);
  A.stg = reinterpret_cast<const double2 *>(ctx->tree_stg);
  A.lrec = reinterpret_cast<const int4 *>(ctx->tree_lrec);
  A.ncell = ctx->ncell;
  A.nv = ctx->nv;
  A.nvp = ctx->nvp;
  A.dt = (float)ctx->geom.dt;
  A.per = ctx->kloop * 64;
  for (int i = 0; i < 7; ++i) A.qb[i] = ctx->tree_qb[i];
  const dim3 block(kTreeThreads, kTreeLeaves);
  auto launch = [&](auto kernel, int first, int n) -> cudaError_t {
    if (n == 0) return cudaSuccess;
    A.sched = ctx->tree_sched + first;
    A.nleaf = n;
    const dim3 grid((unsigned)((n + kTreeLeaves - 1) / kTreeLeaves), (unsigned)ctx->nchunk);
    kernel<<<grid, block, 0, ctx->stream>>>(A);
    return cudaGetLastError();
  };
  const int nreg = ctx->tree_nreg, nall = (int)ctx->ncell;
  const cudaError_t e = (ctx->dim == 2) ? launch(tree_sweep32_kernel<2, true>, 0, nreg)
                                        : launch(tree_sweep32_kernel<3, true>, 0, nreg);
  if (e != cudaSuccess) return e;
  return (ctx->dim == 2) ? launch(tree_sweep32_kernel<2, false>, nreg, nall - nreg)
                         : launch(tree_sweep32_kernel<3, false>, nreg, nall - nreg);
}

} // namespace ibdvm

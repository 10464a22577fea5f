// Persistent 2-D time stepping (sm_103a): a shot's rows are split into bands,
// one CTA per band, and every launch runs many time steps.
//
// Algorithm 1 lines 1 and 5 (operators f and f^T) for a batch of 2-D shots.
// A 2-D shot is small (801 x 301 points: 1 MB per level), so its state stays
// in shared memory and is stepped without a kernel launch per step:
//   * CTA k of a shot owns a band of rpc grid rows.  Its shared memory holds
//     the band of the current and the previous level (ping-pong: the new level
//     overwrites the previous one point by point), rows of 4 + nx + 4 floats
//     with zero columns for the x stencil, and c2 where it fits;
//   * a thread marches along one float4 column of a chunk of N rows, the z
//     neighbours in a register queue.  N is a template parameter and the band a
//     whole number of chunks, so that no row and no column is guarded (rows past
//     the grid and columns past nx have c2 = 0 and stay zero): with a guarded
//     loop a step took 237 warp instructions per 128 points, now 145, of which
//     the stencil needs 66;
//   * the first and the last chunk march away from the neighbouring bands, so
//     the rows that a neighbour needs are formed first;
//   * entries that inject are added in index order at every node
//     (deterministic): a unit whose entries are one row with one entry per point
//     at most (a source, surface receivers), those of the rows next to a
//     neighbour and all of a cluster's by the thread that marches the unit, the
//     others after the march, a thread per node;
//   * the levels that the caller needs go to their ring slots in global memory
//     (the window GEMM reads them, the next launch starts from them).
// Two exchanges of the band edges (the R rows next to a neighbour):
//   * cluster: the bands of a shot are one thread-block cluster (at most 16
//     CTAs); edges are read from the neighbour's shared memory, one cluster
//     barrier per step (470 cycles);
//   * bands (BAND): the bands of all shots of the batch are one cooperative
//     grid over the whole GPU.  A thread stores the edge values it forms also
//     as 8-byte words (value, step tag) in global memory; the neighbour's
//     thread of the same column, the only one that needs them, loads the words
//     when its march ends and reads again as the next one begins until they
//     carry the step's tag: no fence and no flag (1640-2480 cycles from the store
//     to the reader; 3100 for a flag behind a fence), and most of that passes
//     while the rest of the band is marched.  The wait is bounded: on a timeout
//     the CTA sets bit 0 of *err and steps on without waiting; the launch then
//     ends with NaN in its last level and samples.
// Why both: clusters of this size leave SMs idle (8 shots of 12 CTAs: 96 of
// 152 SMs; 7 clusters of 16 at once), bands use all of them, but an exchange
// through L2 costs more than a cluster barrier, which decides on small grids and
// on wide, shallow ones (clusters of four rows a march); c2_step_cost has the
// measurements.
// Measured per step on GB300 (forward calls of 1500 and 300 levels, their
// difference), before (clusters only, one CTA of 16 warps with guarded rows) and
// now: 601 x 201, 16 shots, order 8: levels 6.1 -> 3.7 us, compensated 13.2 ->
// 7.9 us; 801 x 301, 8 shots: 6.4 -> 3.7, 19.7 -> 8.2 us; 101 x 101, one shot,
// order 4: 1.7 -> 1.2 us; an absorbing layer (601 x 201, 4 shots, then two
// launches per step) 31 -> 4.2 us.  Bound by the shared memory
// pipe (32 wavefronts per 128 points of the levels form: the row and its
// neighbours, c2, the previous and the new level, the ring) and by issue.
//
// Levels form: the arithmetic of the per-step 2-D sweep, operation for
// operation (bit-identical results, but for entries that share a node, whose
// products the per-step path adds unrounded), with or without the absorbing layer.
// Compensated form (forward only): the wavefield is a double-float u + e (e
// stored as bf16) stepped with an error-free transformation, so that the
// rounding of the stored levels, which the Laplacian of the probed field
// amplifies, is carried instead of lost; the Laplacian of u is taken in the
// per-neighbour difference form, exact for neighbours within a factor of two of
// the centre.
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "tp_internal.h"
#include "tp_quotient.h"

namespace tp {

namespace {

constexpr int C2_THREADS = 512;
constexpr int C2_MAXCOL = C2_THREADS;  // float4 columns of a band (nx <= 2048)
constexpr int C2_MAXLIST = 1024; // injection or sampling entries of one shot
constexpr int C2_MAXC = 16;      // cluster size limit (non-portable above 8)
constexpr int C2_MAXBANDS = 152; // CTAs of a cooperative launch
constexpr size_t C2_SMEM = 227 * 1024;

enum C2Mode { C2_LEVELS = 0, C2_COMP = 1, C2_DAMP = 2 };  // (index the tables of c2_step_cost)
struct C2Args {
  Layout L;
  Weights W;
  int nshots, C, rpc, sx, nx4;
  int capi, caps;  // capacities of a band's injection and sampling lists (entries)
  int dir, lev0, nsteps, fresh, store_all;
  float* ring; int nslots; long long ring_ss;  // level l of shot s: ring + s*ring_ss + (l % nslots)*L.field
  __nv_bfloat16* eslots; long long e_ss;       // comp: e of level l: eslots + s*e_ss + (l % 2)*L.field
  const float* c2;
  const long long* inj_off; const float* inj_coef; int ninj;
  const float* inj_val; long long inj_val_ss; int inj_shift;   // row of the values: new level + inj_shift
  const long long* samp_off; int nsamp;
  float* samp_out; long long samp_out_ss; int samp_shift;      // row of the output: new level + samp_shift
  unsigned char* edge;  // BAND: tagged edge words, [plane][cta][side][parity][row][column] of 16 bytes
  uint32_t tag0;        // tag of level lev0 in the first round of shots
  long long spin;       // limit of a wait for an edge word (cycles)
  int* err;
};

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// bf16 <-> fp32 for four values
__device__ __forceinline__ float4 bf4(uint2 r) {
  return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                     __uint_as_float(r.y & 0xffff0000u));
}
__device__ __forceinline__ uint2 to_bf4(float4 v) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}

// s = a + b exactly as s + err (Knuth's TwoSum, 6 operations)
__device__ __forceinline__ float two_sum(float a, float b, float* err) {
  const float s = a + b;
  const float bb = s - a;
  *err = (a - (s - bb)) + (b - bb);
  return s;
}

__device__ __forceinline__ uint32_t sa(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ float4 lds4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ uint2 lds2(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ int ldsi(uint32_t a) {
  int v;
  asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ int4 ldsi4(uint32_t a) {
  int4 v;
  asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts4(uint32_t a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void sts2(uint32_t a, uint2 v) {
  asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(v.x), "r"(v.y) : "memory");
}
// the same from any CTA of the cluster (shared::cluster address)
__device__ __forceinline__ float4 ldc4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ uint2 ldc2(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t mapa(uint32_t a, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// Two edge words of 8 bytes, each a 32-bit value and the tag of its step; a
// word is written and read as one access, so a fresh tag brings its value.
__device__ __forceinline__ uint4 ld_words(const unsigned char* p) {
  unsigned long long a, b;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p));
  return make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
}
__device__ __forceinline__ void st_words(unsigned char* p, uint32_t v0, uint32_t v1, uint32_t tag) {
  const unsigned long long a = ((unsigned long long)tag << 32) | v0, b = ((unsigned long long)tag << 32) | v1;
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}

__device__ __forceinline__ float comp4(const float4& v, int p) {
  return p == 0 ? v.x : (p == 1 ? v.y : (p == 2 ? v.z : v.w));
}

// The operators of one row, 4 points: u[i] the rows i - R of the column (u[R]
// the row itself), low(k) the low parts of row k of the column (COMP; 0: the row
// itself), cq = c2; in shared memory the row (ua, for the neighbours in x) and
// the previous level (na), low parts at eoff and neff + address / 2.  o: the new level,
// en: its low part; c1, s2: the previous level and the sums of S(u) (for the
// absorbing layer).
template <int R, int MODE, class Low>
__device__ __forceinline__ void row4(const Weights& W, const float4* u, Low low, float4 cq, uint32_t ua, uint32_t na,
                                     uint32_t eoff, uint32_t neff, float (&o)[4], float (&en)[4], float4& c1,
                                     float2 (&s2)[2]) {
  constexpr bool COMP = MODE == C2_COMP;
  const float2 m4 = f2(-4.f, -4.f), m1 = f2(-1.f, -1.f), two = f2(2.f, 2.f);
  const float4 xc = u[R];
  if (!COMP) {
    const float4 xl = lds4(ua - 16u), xr = lds4(ua + 16u);
    const float v[12] = {xl.x, xl.y, xl.z, xl.w, xc.x, xc.y, xc.z, xc.w, xr.x, xr.y, xr.z, xr.w};
    c1 = lds4(na);
    // centred form, the per-step 2-D sweep's operations in its order (two
    // points per packed instruction; the x pairs at odd distances are not
    // register pairs, so those sums are scalar)
#pragma unroll
    for (int k = 1; k <= R; ++k) {
      const float4 zp = u[R + k], zm = u[R - k];
      const float2 wk = f2(W.w[k], W.w[k]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int pp = 2 * h;
        const float2 xs = (k & 1) ? f2(__fadd_rn(v[4 + pp + k], v[4 + pp - k]), __fadd_rn(v[5 + pp + k], v[5 + pp - k]))
                                  : __fadd2_rn(f2(v[4 + pp + k], v[5 + pp + k]), f2(v[4 + pp - k], v[5 + pp - k]));
        const float2 zs = __fadd2_rn(h ? f2(zp.z, zp.w) : f2(zp.x, zp.y), h ? f2(zm.z, zm.w) : f2(zm.x, zm.y));
        const float2 t = __ffma2_rn(m4, f2(v[4 + pp], v[5 + pp]), __fadd2_rn(xs, zs));
        s2[h] = k == 1 ? __fmul2_rn(wk, t) : __ffma2_rn(wk, t, s2[h]);
      }
    }
    // new = c2 S + (2u - u_prev); 2u is exact, so the FMA rounds 2u - u_prev once, as a subtraction
#pragma unroll
    for (int p = 0; p < 4; ++p)
      o[p] = fmaf(comp4(cq, p), p & 1 ? s2[p / 2].y : s2[p / 2].x, fmaf(2.f, v[4 + p], -comp4(c1, p)));
    return;
  }
  // double-float levels: U = u + e.  S(e) in the centred form (e is a few ulp of
  // u: its rounding is negligible), S(u) in the difference form for k = 1, 2 and
  // the centred form for the small weights k = 3, 4 (their rounding is a few
  // hundredths of an ulp of u)
  const uint32_t ea = eoff + ua / 2u;
  const float4 fl = bf4(lds2(ea - 8u)), fr = bf4(lds2(ea + 8u)), fc = bf4(low(0));
  const float ve[12] = {fl.x, fl.y, fl.z, fl.w, fc.x, fc.y, fc.z, fc.w, fr.x, fr.y, fr.z, fr.w};
  float2 su[2], se[2];
#pragma unroll
  for (int k = 1; k <= R; ++k) {
    const float4 ezp = bf4(low(k)), ezm = bf4(low(-k));
    const float2 wk = f2(W.w[k], W.w[k]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int pp = 2 * h;
      const float2 xe = (k & 1) ? f2(__fadd_rn(ve[4 + pp + k], ve[4 + pp - k]), __fadd_rn(ve[5 + pp + k], ve[5 + pp - k]))
                                : __fadd2_rn(f2(ve[4 + pp + k], ve[5 + pp + k]), f2(ve[4 + pp - k], ve[5 + pp - k]));
      const float2 ze = __fadd2_rn(h ? f2(ezp.z, ezp.w) : f2(ezp.x, ezp.y), h ? f2(ezm.z, ezm.w) : f2(ezm.x, ezm.y));
      const float2 te = __ffma2_rn(m4, f2(ve[4 + pp], ve[5 + pp]), __fadd2_rn(xe, ze));
      se[h] = k == 1 ? __fmul2_rn(wk, te) : __ffma2_rn(wk, te, se[h]);
    }
  }
  const float4 xl = lds4(ua - 16u), xr = lds4(ua + 16u);
  const float v[12] = {xl.x, xl.y, xl.z, xl.w, xc.x, xc.y, xc.z, xc.w, xr.x, xr.y, xr.z, xr.w};
#pragma unroll
  for (int k = 1; k <= R; ++k) {
    const float4 zp = u[R + k], zm = u[R - k];
    const float2 wk = f2(W.w[k], W.w[k]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int pp = 2 * h;
      const float2 cv = f2(v[4 + pp], v[5 + pp]);
      const float2 zpp = h ? f2(zp.z, zp.w) : f2(zp.x, zp.y), zmm = h ? f2(zm.z, zm.w) : f2(zm.x, zm.y);
      float2 t;
      if (k <= 2) {
        // the two heavy weights: per-neighbour differences, exact for
        // neighbours within a factor two of the centre
        float2 dxp, dxm;
        if (k & 1) {
          dxp = f2(__fadd_rn(v[4 + pp + k], -cv.x), __fadd_rn(v[5 + pp + k], -cv.y));
          dxm = f2(__fadd_rn(v[4 + pp - k], -cv.x), __fadd_rn(v[5 + pp - k], -cv.y));
        } else {
          dxp = __ffma2_rn(m1, cv, f2(v[4 + pp + k], v[5 + pp + k]));
          dxm = __ffma2_rn(m1, cv, f2(v[4 + pp - k], v[5 + pp - k]));
        }
        const float2 dzp = __ffma2_rn(m1, cv, zpp), dzm = __ffma2_rn(m1, cv, zmm);
        t = __fadd2_rn(__fadd2_rn(dxp, dxm), __fadd2_rn(dzp, dzm));
      } else {
        const float2 xs = (k & 1) ? f2(__fadd_rn(v[4 + pp + k], v[4 + pp - k]), __fadd_rn(v[5 + pp + k], v[5 + pp - k]))
                                  : __fadd2_rn(f2(v[4 + pp + k], v[5 + pp + k]), f2(v[4 + pp - k], v[5 + pp - k]));
        t = __ffma2_rn(m4, cv, __fadd2_rn(xs, __fadd2_rn(zpp, zmm)));
      }
      su[h] = k == 1 ? __fmul2_rn(wk, t) : __ffma2_rn(wk, t, su[h]);
    }
  }
  c1 = lds4(na);
  const float4 f1 = bf4(lds2(neff + na / 2u));
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int pp = 2 * h;
    const float2 uu = f2(v[4 + pp], v[5 + pp]), ee = f2(ve[4 + pp], ve[5 + pp]);
    const float2 cp = f2(comp4(c1, pp), comp4(c1, pp + 1)), ep = f2(comp4(f1, pp), comp4(f1, pp + 1));
    const float2 cc2 = f2(comp4(cq, pp), comp4(cq, pp + 1));
    // 2u - u_prev exactly (TwoSum), then the small terms, then TwoSum again
    // (x - y as fma(-1, y, x): the product is exact)
    const float2 u2 = __fmul2_rn(two, uu);
    const float2 av = __ffma2_rn(m1, cp, u2);
    const float2 bb = __ffma2_rn(m1, u2, av);
    const float2 ea = __ffma2_rn(m1, __fadd2_rn(cp, bb), __ffma2_rn(m1, __ffma2_rn(m1, bb, av), u2));
    const float2 b = __ffma2_rn(cc2, __fadd2_rn(su[h], se[h]), __ffma2_rn(m1, ep, __fmul2_rn(two, ee)));
    const float2 bt = __fadd2_rn(b, ea);
    const float2 sm = __fadd2_rn(av, bt);
    const float2 b2 = __ffma2_rn(m1, av, sm);
    const float2 er2 = __fadd2_rn(__ffma2_rn(m1, __ffma2_rn(m1, b2, sm), av), __ffma2_rn(m1, b2, bt));
    o[pp] = sm.x;
    o[pp + 1] = sm.y;
    en[pp] = er2.x;
    en[pp + 1] = er2.y;
  }
}

// A unit of work: one float4 column of a chunk of N rows of the band, marched
// by one thread with the z neighbours in a register queue (blocks of BL rows
// unrolled, so that the queue moves once per block).  The band's rpc rows are a
// multiple of N; rows past the grid and columns past nx have c2 = 0 and stay
// zero, so that no row and no column is guarded.
// LEAN (clusters without c2 in shared memory, for wide grids): the levels alone
// fill the shared memory.  c2 comes from global memory, nothing is kept per
// unit, all entries are added after the march, and the last chunk of a band
// has as many rows as are left.  Compensated step, order 8: 1800 x 100 8.4 us,
// 2001 x 101 x 8 shots 10.6 us (8.3 and 17.1 us when a cluster kept c2 in global
// memory and guarded every row).
template <int R, int MODE, bool BAND, int N, bool C2S>
__global__ void __launch_bounds__(C2_THREADS, 1) sweep2d_shots(C2Args a) {
  constexpr bool COMP = MODE == C2_COMP, DAMP = MODE == C2_DAMP, LEAN = !BAND && !C2S;
  static_assert(!LEAN || (!DAMP && N <= 4), "a lean march is one block of rows without a layer");
  constexpr int PER = C2_MAXLIST / C2_THREADS;  // list entries per thread
  const int tid = threadIdx.x;
  const int C = a.C, rank = blockIdx.x % C, cid = blockIdx.x / C, ncl = gridDim.x / C;
  const int sx = a.sx, sx4 = a.sx / 4, rpc = a.rpc, nx4 = a.nx4;
  const int nz = a.L.nz, nx = a.L.nx, px = a.L.px;
  const int z0 = rank * rpc;
  const int nrow = min(rpc, nz - z0);  // rows of the grid that this CTA owns (>= 1)
  const int nch = LEAN ? (rpc + N - 1) / N : rpc / N, units = nch * nx4;
  const int ntab = LEAN ? 0 : units;  // units with entries in the tables below

  // shared memory: both levels of the band, a zero row (clusters), the low
  // parts of both levels (COMP), c2, the band's injection and sampling
  // entries, the damping by distance (DAMP)
  extern __shared__ __align__(16) unsigned char smem[];
  float* const U0 = reinterpret_cast<float*>(smem);
  float* const U1 = U0 + (size_t)rpc * sx;
  float* const Z = U1 + (size_t)rpc * sx;  // zeros (as fp32 and as bf16)
  float* pf = Z + (BAND ? 0 : sx);
  // bands: the low parts have R rows before and after the band (behind a
  // march's first row), one region between the buffers for both of them
  const int er = BAND ? R : 0;
  __nv_bfloat16* const E0 = reinterpret_cast<__nv_bfloat16*>(pf) + (size_t)er * sx;
  __nv_bfloat16* const E1 = E0 + (size_t)(rpc + er) * sx;
  if (COMP) pf = reinterpret_cast<float*>(E1 + (size_t)(rpc + er) * sx);
  float* const c2b = pf;
  if (C2S) pf += (size_t)rpc * 4 * nx4;
  uint32_t* const il = reinterpret_cast<uint32_t*>(pf);  // injection, by node: node (band index) << 16 | LEAD | MANY | k
  uint32_t* const sl = il + a.capi;                      // sampling: the same
  const int vstep = a.capi + 4;                               // floats from one step's values to the next step's
  float* const ival = reinterpret_cast<float*>(sl + a.caps);  // [2][vstep]: values of this step and the next, [capi]: 0
  // entries by unit: in the common case (one row of the unit, one entry per
  // point at most) the row's place in the march and the entry of each of its 4
  // points; else (a chain) entries by node.  Those in edge rows (WALK: all) are
  // walked along nxt when the unit is marched; the others are added after the
  // march, where an entry with LEAD stands for the nxt entries of its node from
  // it on.  (WALK: so does one with MANY, and the last of them leads on.)  Step at
  // 401 x 401 with 1024 receivers at a node 9.7 us, in a patch of 32 x 32 5.6 us,
  // along a borehole 4.4 us, in a row 3.5 us (14 ms, 43, 7.5 and 4.0 us when the
  // unit's thread walked the chain once for every entry).
  // Per unit, read where it is used (kept in registers, it spilled):
  //   ua[u]: byte offset of its first row in a level buffer, offset in a field,
  //          byte offset in c2, flags | its first row << 8
  //   ub[u]: words of its first row and of the nearest row behind it (byte
  //          offsets for parity 0), chain's first entry | march row of the line
  //          << 16, column
  int4* const ua_ = reinterpret_cast<int4*>(ival + 2 * vstep);
  int4* const ub_ = ua_ + ntab;
  ushort4* const uline = reinterpret_cast<ushort4*>(ub_ + ntab);
  uint16_t* const tl = reinterpret_cast<uint16_t*>(uline + ntab);  // last entry of a unit (set-up)
  uint16_t* const nxt = tl + (ntab + 1) / 2 * 2;                // next entry of the same unit; LEAD, MANY: entries of its node
  int* const cnt = reinterpret_cast<int*>(nxt + (ntab + 1) / 2 % 2 * 2 + a.capi);  // [0] injection, [1] sampling entries, [3] LEAD used, [4 ..] per-warp counts
  volatile int* const aborted = cnt + 2;
  uint32_t* const tab = reinterpret_cast<uint32_t*>(cnt + 4 + C2_THREADS / 32);  // clusters: edge rows of the levels, low parts
  float2* const dmp = reinterpret_cast<float2*>(tab + (BAND ? 0 : 8 * R));
  // all chains walked: beside the marches of clusters, of the layer and of c2 in
  // global memory the code after the march cost a step 3 to 11 %
  constexpr bool WALK = !LEAN && (!BAND || DAMP || !C2S);
  constexpr uint32_t NONE = 0xffff, LEAD = 0x8000, MANY = 0x4000, KMASK = 0x3fff;
  static_assert(C2_MAXLIST <= (int)KMASK, "an entry's index and two flags in 16 bits");
  constexpr int F_ON = 1, F_UP = 2, F_FULL = 4, F_NB = 8, F_OUT = 16, F_PUB = 32, F_LATE = 64;  // flags of a unit

  if (!BAND) {
    // tab[b * 2R + i] (and 4R + ...: low parts): edge row i of buffer b, rows
    // -R .. -1 of the band, then rpc .. rpc + R - 1
    for (int i = tid; i < 4 * R; i += C2_THREADS) {
      const int b = i / (2 * R), e = i % (2 * R), zz = z0 + (e < R ? e - R : rpc + e - R);
      uint32_t u = mapa(sa(Z), rank), lo = u;
      if (zz >= 0 && zz < nz) {
        const int rk = zz / rpc, lr = zz - rk * rpc;
        u = mapa(sa((b ? U1 : U0) + (size_t)lr * sx), rk);
        if (COMP) lo = mapa(sa((b ? E1 : E0) + (size_t)lr * sx), rk);
      }
      tab[i] = u;
      tab[4 * R + i] = lo;
    }
    for (int i = tid; i < sx; i += C2_THREADS) Z[i] = 0.f;
  }
  if (DAMP)  // a = samax ((sw - d) / sw)^2 by distance (sponge_a's operations) and 1 / (1 + a); [sw]: outside the layer
    for (int d = tid; d <= a.W.sw; d += C2_THREADS) {
      const float t = (float)(a.W.sw - d) / (float)a.W.sw, ad = a.W.samax * t * t;
      dmp[d] = make_float2(ad, 1.0f / (1.0f + ad));
    }
  if (tid == 0) *aborted = 0;
  if (C2S)
    for (int i = tid; i < rpc * nx4; i += C2_THREADS)
      reinterpret_cast<float4*>(c2b)[i] =
          i / nx4 < nrow ? __ldg(reinterpret_cast<const float4*>(a.c2 + (long long)(z0 + i / nx4 + H) * px + HX) + i % nx4)
                         : make_float4(0.f, 0.f, 0.f, 0.f);

  const uint32_t sU0 = sa(U0), sE0 = sa(E0), sC2 = sa(c2b), lbytes = (uint32_t)(rpc * sx) * 4u;
  const uint32_t ebytes = (uint32_t)((rpc + er) * sx) * 2u;  // from one buffer of low parts to the other
  // chunk -> first row and direction of its march: the last chunk up, the
  // others down, so that the rows next to a neighbour come first
  auto march = [&](int ch, int& start, int& d) {
    const bool up = ch > 0 && ch == nch - 1;
    d = up ? -1 : 1;
    start = up ? ch * N + N - 1 : ch * N;
  };
  // BAND: edge words, offset of (cta, side 0 first / 1 last rows, parity, row, column), planes apart
  const uint32_t erow = (uint32_t)nx4 * 16u, epar = erow * R, eplane = gridDim.x * 4u * epar;
  const uint32_t mine = blockIdx.x * 4u * epar;  // this CTA's words; the band above's precede them, below's follow
  auto publish = [&](uint32_t o, float4 v, uint2 e, uint32_t tag) {
    unsigned char* w = a.edge + o;
    st_words(w, __float_as_uint(v.x), __float_as_uint(v.y), tag);
    st_words(w + eplane, __float_as_uint(v.z), __float_as_uint(v.w), tag);
    if (COMP) st_words(w + 2 * eplane, e.x, e.y, tag);
  };

  uint32_t tagb = a.tag0;
  for (int shot = cid; shot < a.nshots; shot += ncl, tagb += (uint32_t)a.nsteps) {
    // ---------------------------------------------------------- per-shot set-up
    // this band's injection and sampling entries, compacted in index order
    for (int list = 0; list < 2; ++list) {
      const int num = list == 0 ? a.ninj : a.nsamp;
      const long long* off = list == 0 ? a.inj_off + (long long)shot * a.ninj
                                       : (num > 0 ? a.samp_off + (long long)shot * a.nsamp : nullptr);
      uint32_t* out = list == 0 ? il : sl;
      if (tid == 0) cnt[list] = 0;
      __syncthreads();
      for (int base = 0; base < num; base += C2_THREADS) {
        const int k = base + tid;
        int l = -1;
        if (k < num) {
          const long long o = off[k];
          if (o >= 0) {
            const int zz = (int)(o / px) - H, xx = (int)(o % px) - HX;
            if (zz >= z0 && zz < z0 + nrow) l = (zz - z0) * sx + 4 + xx;
          }
        }
        const unsigned m = __ballot_sync(0xffffffffu, l >= 0);
        if ((tid & 31) == 0) cnt[4 + (tid >> 5)] = __popc(m);
        __syncthreads();
        int before = 0;
        for (int w = 0; w < (tid >> 5); ++w) before += cnt[4 + w];
        if (l >= 0) out[cnt[list] + before + __popc(m & ((1u << (tid & 31)) - 1u))] = (uint32_t)l << 16 | (uint32_t)k;
        __syncthreads();
        if (tid == 0) {
          int tot = 0;
          for (int w = 0; w < C2_THREADS / 32; ++w) tot += cnt[4 + w];
          cnt[list] += tot;
        }
        __syncthreads();
      }
    }
    const int ni = cnt[0], ns = cnt[1];
    // the injection entries by node, and in index order at a node: the entries
    // of a node are neighbours in the list
    bool moved = false;
    for (int i = tid; i + 1 < ni; i += C2_THREADS) moved = moved || il[i] > il[i + 1];
    if (__syncthreads_or(moved)) {
      uint32_t key[PER];
      int to[PER];
      for (int i = ni + tid; i < a.capi; i += C2_THREADS) il[i] = 0xffffffffu;
      __syncthreads();
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        key[q] = tid + q * C2_THREADS < ni ? il[tid + q * C2_THREADS] : 0u;
        to[q] = 0;
      }
      for (int i = 0; i < ni; i += 4) {
        const uint4 e = *reinterpret_cast<const uint4*>(il + i);
#pragma unroll
        for (int q = 0; q < PER; ++q) to[q] += (e.x < key[q]) + (e.y < key[q]) + (e.z < key[q]) + (e.w < key[q]);
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < PER; ++q)
        if (tid + q * C2_THREADS < ni) il[to[q]] = key[q];
      __syncthreads();
    }
    // a chain of entries per unit, in this order
    for (int u = tid; u < ntab; u += C2_THREADS) {
      ub_[u].z = (int)(NONE << 16 | NONE);
      tl[u] = (uint16_t)NONE;
    }
    if (tid == 0) cnt[3] = 0;
    __syncthreads();
    if (LEAN) {
      for (int i = tid; i < ni; i += C2_THREADS) {
        const uint32_t l = il[i] >> 16;
        if (i > 0 && il[i - 1] >> 16 == l) continue;
        int n = 1;
        while (i + n < ni && il[i + n] >> 16 == l) ++n;
        il[i] |= LEAD;
        nxt[i] = (uint16_t)n;
        cnt[3] = 1;
      }
    } else if (tid < 32) {
      for (int b = 0; b < ni; b += 32) {
        const int i = b + tid;
        const bool on = i < ni;
        int u = -1 - tid;
        if (on) {
          const int l = (int)(il[i] >> 16), rr = l / sx;
          u = rr / N * nx4 + (l - rr * sx - 4) / 4;
          nxt[i] = (uint16_t)NONE;
        }
        const unsigned m = __match_any_sync(0xffffffffu, u);
        __syncwarp();
        if (on) {
          const unsigned below = m & ((1u << tid) - 1u);
          if (below) nxt[b + 31 - __clz(below)] = (uint16_t)i;
          else if (tl[u] != NONE) nxt[tl[u]] = (uint16_t)i;
          else ub_[u].z = (int)(NONE << 16 | (uint32_t)i);
        }
        __syncwarp();
        if (on && !(m >> tid >> 1)) tl[u] = (uint16_t)i;
        __syncwarp();
      }
    }
    __syncthreads();
    for (int u = tid; u < ntab; u += C2_THREADS) {
      const int ch = u / nx4, cu = u - ch * nx4;
      int start, d, row = -1, at[4] = {a.capi, a.capi, a.capi, a.capi};
      march(ch, start, d);
      const bool top = start == 0 && d > 0, bottom = start == rpc - 1 && d < 0;
      const bool nb = (top && rank > 0) || (bottom && rank < C - 1);  // a neighbour's rows behind
      uint32_t ent = (uint32_t)ub_[u].z;
      bool line = true, edge = false;  // edge: entries among the R rows that a neighbour needs
      for (uint32_t i = ent & NONE; i != NONE; i = nxt[i]) {
        const int l = (int)(il[i] >> 16), r = l / sx, p = (l - r * sx) & 3;
        line = line && (row < 0 || row == r);
        row = r;
        edge = edge || (BAND && nb && (r - start) * d < R);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q == p) {
            line = line && at[q] == a.capi;
            at[q] = (int)i;
          }
      }
      if (row >= 0 && line && !edge) {
        ent = (uint32_t)((row - start) * d) << 16 | NONE;
      } else {
        uint32_t head = NONE, last = NONE;  // of the entries in edge rows
        for (uint32_t i = ent & NONE; i != NONE;) {
          const uint32_t lead = i, l = il[i] >> 16;
          uint32_t tail = i;
          int n = 0;
          for (; i != NONE && il[i] >> 16 == l; i = nxt[i], ++n) tail = i;
          if (WALK || (edge && ((int)(l / (uint32_t)sx) - start) * d < R)) {
            if (head == NONE) head = lead;
            last = tail;
            if (WALK && n > 1) {
              il[lead] |= MANY;
              nxt[lead] = (uint16_t)n;
            }
          } else {
            il[lead] |= LEAD;
            nxt[lead] = (uint16_t)n;
            cnt[3] = 1;
          }
        }
        if (last != NONE) nxt[last] = (uint16_t)NONE;
        ent = NONE << 16 | head;
      }
      uline[u] = make_ushort4((unsigned short)at[0], (unsigned short)at[1], (unsigned short)at[2], (unsigned short)at[3]);
      int f = ch * N < nrow ? F_ON : 0;
      if (d < 0) f |= F_UP;
      if (start < nrow && start + d * (N - 1) < nrow) f |= F_FULL;
      if (BAND && nb) f |= F_NB | (edge ? F_LATE : F_PUB);
      if (BAND && (top || bottom) && !nb) f |= F_OUT;
      ua_[u] = make_int4((start * sx + 4 + 4 * cu) * 4, (z0 + H + start) * px + HX + 4 * cu, (start * nx4 + cu) * 16, f | start << 8);
      ub_[u] = make_int4((int)((top ? mine : mine + 2u * epar + (R - 1) * erow) + (uint32_t)cu * 16u),
                         (int)((top ? mine - 2u * epar + (R - 1) * erow : mine + 4u * epar) + (uint32_t)cu * 16u), (int)ent, cu);
    }

    // state of the shot: the current and previous levels (and their low parts)
    float* const ring = a.ring + (long long)shot * a.ring_ss;
    __nv_bfloat16* const eb = COMP ? a.eslots + (long long)shot * a.e_ss : nullptr;
    auto slot = [&](int l) { return (long long)(((l % a.nslots) + a.nslots) % a.nslots) * a.L.field; };
    const int lc0 = a.lev0, lp0 = a.lev0 - a.dir;
    {
      const float* gc = ring + slot(lc0);
      const float* gp = ring + slot(lp0);
      for (int i = tid; i < rpc * sx4; i += C2_THREADS) {
        const int r = i / sx4, c = i % sx4;
        const long long g = (long long)(z0 + r + H) * px + HX - 4 + 4 * c;
        const bool in = !a.fresh && r < nrow;
        float4 vc = make_float4(0.f, 0.f, 0.f, 0.f), vp = vc;
        if (in) {
          vc = *reinterpret_cast<const float4*>(gc + g);
          vp = *reinterpret_cast<const float4*>(gp + g);
        }
        reinterpret_cast<float4*>(U0 + (size_t)r * sx)[c] = vc;
        reinterpret_cast<float4*>(U1 + (size_t)r * sx)[c] = vp;
        if (COMP) {
          uint2 ec = make_uint2(0u, 0u), ep = ec;
          if (in) {
            ec = *reinterpret_cast<const uint2*>(eb + (long long)(lc0 & 1) * a.L.field + g);
            ep = *reinterpret_cast<const uint2*>(eb + (long long)(lp0 & 1) * a.L.field + g);
          }
          *reinterpret_cast<uint2*>(E0 + (size_t)r * sx + 4 * c) = ec;
          *reinterpret_cast<uint2*>(E1 + (size_t)r * sx + 4 * c) = ep;
        }
      }
    }
    // value that entry i adds to level lev
    auto entry = [&](int i, int lev) {
      const int k = (int)(il[i] & KMASK);
      return __ldg(a.inj_coef + (long long)shot * a.ninj + k) *
             __ldg(a.inj_val + (long long)shot * a.inj_val_ss + (long long)(lev + a.inj_shift) * a.ninj + k);
    };
    for (int i = tid; i < ni; i += C2_THREADS) ival[i] = entry(i, a.lev0 + a.dir);
    if (tid < 2) ival[tid * vstep + a.capi] = 0.f;
    // receivers of a complete level
    auto sample = [&](int lev, const float* Ub) {
      const int orow = lev + a.samp_shift;
      if (orow < 0 || !a.samp_out) return;
      float* out = a.samp_out + (long long)shot * a.samp_out_ss + (long long)orow * a.nsamp;
      for (int i = tid; i < ns; i += C2_THREADS) out[sl[i] & 0xffffu] = Ub[sl[i] >> 16];
    };
    __syncthreads();
    if (BAND) {
      for (int i = tid; i < 2 * R * nx4; i += C2_THREADS) {
        const int row = i / nx4, c = i - row * nx4, side = row >= R, t = row - side * R;
        if (side ? rank == C - 1 : rank == 0) continue;
        const uint32_t o = (uint32_t)((side ? rpc - R + t : t) * sx + 4 + 4 * c);
        publish(mine + side * 2u * epar + (tagb & 1u) * epar + (uint32_t)t * erow + (uint32_t)c * 16u, lds4(sU0 + o * 4u),
                COMP ? lds2(sE0 + o * 2u) : make_uint2(0u, 0u), tagb);
      }
    } else {
      cluster_arrive();  // every band of the cluster is loaded
    }

    __syncthreads();
    const int rs = sx * 4;
    const uint32_t sA = sa(ua_), sB = sa(ub_);
    // the words of the R rows behind (k = 0: the nearest), loaded when a march
    // ends for the next one (COMP: as it begins, there are no registers to spare)
    constexpr bool AHEAD = BAND && !COMP;
    uint4 wa[BAND ? R : 1], wb[BAND ? R : 1], wc[BAND && COMP ? R : 1];
    auto ask = [&](int k, uint32_t o) {
      const unsigned char* p = a.edge + o;
      wa[BAND ? k : 0] = ld_words(p);
      wb[BAND ? k : 0] = ld_words(p + eplane);
      if (COMP) wc[BAND && COMP ? k : 0] = ld_words(p + 2 * eplane);
    };
    // bounded wait for words at offset o
    auto settle = [&](uint32_t o, uint4& x, uint4& y, uint4& z, uint32_t tag) {
      auto came = [&] { return x.y == tag && x.w == tag && y.y == tag && y.w == tag && (!COMP || (z.y == tag && z.w == tag)); };
      if (came()) return;
      const unsigned char* p = a.edge + o;
      const long long t0 = clock64();
      while (!came()) {
        if (*aborted) break;
        if (clock64() - t0 > a.spin) {
          *aborted = 1;
          atomicOr(a.err, 1);
          break;
        }
        x = ld_words(p);
        y = ld_words(p + eplane);
        if (COMP) z = ld_words(p + 2 * eplane);
      }
    };
    const bool ahead = AHEAD && units <= C2_THREADS;
    auto ask_ahead = [&](uint32_t tag) {  // the words of this thread's rows behind
      if (!ahead || tid >= units) return;
      const int f = ldsi(sA + (uint32_t)tid * 16u + 12u);
      if ((f & (F_ON | F_NB)) != (F_ON | F_NB)) return;
      const uint32_t o = (uint32_t)ldsi(sB + (uint32_t)tid * 16u + 4u) + (tag & 1u) * epar, st = f & F_UP ? erow : 0u - erow;
#pragma unroll
      for (int k = 0; k < R; ++k) ask(k, o + (uint32_t)k * st);
    };
    ask_ahead(tagb);
    const uint32_t sLead = sa(cnt + 3);
    int slot_new = ((a.lev0 + a.dir) % a.nslots + a.nslots) % a.nslots;
    float* glev = ring + (long long)slot_new * a.L.field;  // the new level's field
    const int kfrom = a.store_all ? 0 : a.nsteps - 2;      // levels from this step on go to their ring slots
    for (int step = 0, cur = 0; step < a.nsteps; ++step, cur ^= 1) {
      const int lcur = a.lev0 + step * a.dir;
      const uint32_t tag = tagb + (uint32_t)step;
      // values that the next step injects (loaded now, put in place when this step ends)
      float pv[PER];
      if (ni > 0 && step + 1 < a.nsteps) {
#pragma unroll
        for (int q = 0; q < PER; ++q) pv[q] = tid + q * C2_THREADS < ni ? entry(tid + q * C2_THREADS, lcur + 2 * a.dir) : 0.f;
      }
      // the current level is complete: its receivers (the first level of a
      // launch was sampled by the launch before)
      if (ns > 0 && step > 0) sample(lcur, cur ? U1 : U0);
      if (!BAND) {
        __syncwarp();
        cluster_wait();  // the level's edge rows are complete in every band
      }
      const bool keep = step >= kfrom;
      const uint32_t nd = cur ? 0u - lbytes : lbytes;  // from the current level to the new one
      // low parts of the value at shared address x: at eoff + x / 2 in the current level, at neff + x / 2 in the new one
      const uint32_t eoff = cur ? sE0 + ebytes - (sU0 + lbytes) / 2u : sE0 - sU0 / 2u;
      const uint32_t neff = cur ? sE0 - sU0 / 2u : sE0 + ebytes - (sU0 + lbytes) / 2u;
      for (int un = tid; un < units; un += C2_THREADS) {
        // the unit's entries (bands read them after the march: a register more spills)
        uint32_t ent = LEAN || BAND ? NONE << 16 | NONE : (uint32_t)ldsi(sB + (uint32_t)un * 16u + 8u);
        {
          int4 A;
          int cul = 0;  // LEAN: the column
          if (LEAN) {
            const int ch = un / nx4, first = ch * N;
            cul = un - ch * nx4;
            A = make_int4((first * sx + 4 + 4 * cul) * 4, (z0 + H + first) * px + HX + 4 * cul, 0,
                          (first < nrow ? F_ON : 0) | (first + N <= nrow ? F_FULL : 0) | first << 8);
          } else {
            A = ldsi4(sA + (uint32_t)un * 16u);
          }
          const int f = A.w;
          if (!(f & F_ON)) continue;
          const int ds = f & F_UP ? -rs : rs, gd = f & F_UP ? -px : px, cd = (f & F_UP ? -nx4 : nx4) * 16;
          uint32_t ua = sU0 + (cur ? lbytes : 0u) + (uint32_t)A.x;
          // c2 of the unit's rows, in shared or in global memory (zero past the grid: padding)
          uint32_t c2a = sC2 + (uint32_t)A.z;
          int go = A.y;  // the row's place in a field
          auto ld_c2 = [&](int x) { return C2S ? lds4(c2a) : __ldg(reinterpret_cast<const float4*>(a.c2 + x)); };
          // clusters: row r, in the band or an edge row (zero outside the grid)
          auto ld_any = [&](int r, uint32_t x, float4& u, uint2& e) {
            if (r >= 0 && r < rpc) {
              u = lds4(x);
              if (COMP) e = lds2(eoff + x / 2u);
            } else {
              const int i = cur * 2 * R + (r < 0 ? r + R : r - rpc + R);
              const uint32_t co = (uint32_t)(4 + 4 * (LEAN ? cul : ldsi(sB + (uint32_t)un * 16u + 12u)));
              u = ldc4(tab[i] + co * 4u);
              if (COMP) e = ldc2(tab[4 * R + i] + co * 2u);
            }
          };
          const int start = f >> 8, d = f & F_UP ? -1 : 1;
          constexpr int BL = N % 4 == 0 ? 4 : N;  // rows of an unrolled block
          float4 u[BL + 2 * R], cqn = ld_c2(go);
          constexpr bool EQ = COMP && !BAND;  // low parts queued too (bands: read for every row, a second queue spilled)
          uint2 e[EQ ? BL + 2 * R : 1];
          uint32_t ha = ua - (uint32_t)(R * ds);  // a row's address as it enters the queue
#pragma unroll
          for (int i = 0; i < 2 * R; ++i) {
            if (!BAND) {
              ld_any(start + d * (i - R), ha, u[i], e[EQ ? i : 0]);
            } else if (i >= R || !(f & (F_NB | F_OUT))) {  // N >= R: the rows of the march, or those of the chunk behind
              u[i] = lds4(ha);
            }
            ha += (uint32_t)ds;
          }
          if (BAND && f & F_NB) {
            const uint32_t o = (uint32_t)ldsi(sB + (uint32_t)un * 16u + 4u) + (tag & 1u) * epar, st = f & F_UP ? erow : 0u - erow;
            constexpr int G = COMP ? 2 : R;  // rows asked for at once
#pragma unroll
            for (int k0 = 0; k0 < R; k0 += G) {
              if (!ahead) {
#pragma unroll
                for (int k = k0; k < k0 + G; ++k) ask(k, o + (uint32_t)k * st);
              }
#pragma unroll
              for (int k = k0; k < k0 + G; ++k) {
                uint4& x = wa[BAND ? k : 0];
                uint4& y = wb[BAND ? k : 0];
                uint4& z = wc[BAND && COMP ? k : 0];
                settle(o + (uint32_t)k * st, x, y, z, tag);
                u[R - 1 - k] = make_float4(__uint_as_float(x.x), __uint_as_float(x.z), __uint_as_float(y.x), __uint_as_float(y.z));
                if (COMP) sts2(eoff + ua / 2u - (uint32_t)((k + 1) * (ds / 2)), make_uint2(z.x, z.z));
              }
            }
          } else if (BAND && f & F_OUT) {
#pragma unroll
            for (int k = 0; k < R; ++k) {
              u[R - 1 - k] = make_float4(0.f, 0.f, 0.f, 0.f);
              if (COMP) sts2(eoff + ua / 2u - (uint32_t)((k + 1) * (ds / 2)), make_uint2(0u, 0u));
            }
          }
          const bool pub = BAND && f & F_PUB && step + 1 < a.nsteps;
          uint32_t w = pub ? (uint32_t)ldsi(sB + (uint32_t)un * 16u) + epar - (tag & 1u) * epar : 0u;
          const uint32_t wd = f & F_UP ? 0u - erow : erow;
#pragma unroll 1
          for (int b = 0; b < N / BL; ++b) {
#pragma unroll
            for (int jj = 0; jj < BL; ++jj) {
              if (LEAN && start + jj >= rpc) break;  // the last chunk's rows
              // the row R beyond this one completes the queue (bands: a row of the next chunk at most)
              if (BAND) {
                u[jj + 2 * R] = lds4(ha);
              } else {
                ld_any(start + d * (b * BL + jj + R), ha, u[jj + 2 * R], e[EQ ? jj + 2 * R : 0]);
              }
              ha += (uint32_t)ds;
              const float4 cq = cqn;
              c2a += (uint32_t)cd;
              if (jj + 1 < BL || b + 1 < N / BL) cqn = ld_c2(go + gd);
              const uint32_t na = ua + nd;
              float o[4], en[4] = {0.f, 0.f, 0.f, 0.f};
              float4 c1;
              float2 s2[2];
              auto low = [&](int k) {
                if constexpr (EQ) return e[jj + R + k];
                else return lds2(eoff + ua / 2u + (uint32_t)(k * ds / 2));
              };
              row4<R, MODE>(a.W, u + jj, low, cq, ua, na, eoff, neff, o, en, c1, s2);
              if (DAMP) {
                const int dz = nz - 1 - (z0 + start + d * (b * BL + jj)), cu = ldsi(sB + (uint32_t)un * 16u + 12u);
                if (min(min(4 * cu, nx - 4 - 4 * cu), dz) < a.W.sw) {
#pragma unroll
                  for (int p = 0; p < 4; ++p) {
                    const int dd = min(min(4 * cu + p, nx - 1 - (4 * cu + p)), dz);
                    const float2 ai = dmp[dd >= 0 && dd < a.W.sw ? dd : a.W.sw];
                    // tp_stencil.cu's epilogue; a = 0 (outside the layer) gives the undamped value
                    o[p] = quotient(fmaf(comp4(cq, p), p & 1 ? s2[p / 2].y : s2[p / 2].x,
                                         fmaf(-(1.0f - ai.x), comp4(c1, p), 2.0f * comp4(u[jj + R], p))),
                                    1.0f + ai.x, ai.y);
                  }
                }
              }
              // the new value over the previous level (own points: no other thread reads them in this step)
              const float4 ov = make_float4(o[0], o[1], o[2], o[3]);
              const uint2 ev = COMP ? to_bf4(make_float4(en[0], en[1], en[2], en[3])) : make_uint2(0u, 0u);
              sts4(na, ov);
              if (COMP) sts2(neff + na / 2u, ev);
              if (keep && (f & F_FULL || start + d * (b * BL + jj) < nrow)) *reinterpret_cast<float4*>(glev + go) = ov;
              go += gd;
              ua += (uint32_t)ds;
              if (BAND && jj < R && b == 0 && pub) {
                publish(w, ov, ev, tag + 1);
                w += wd;
              }
            }
            if (N > BL) {
#pragma unroll
              for (int i = 0; i < 2 * R; ++i) {
                u[i] = u[i + BL];
                if (EQ) e[EQ ? i : 0] = e[EQ ? i + BL : 0];
              }
            }
          }
        }
        // entries at this unit's points, added to the values just stored
        if (BAND) ent = (uint32_t)ldsi(sB + (uint32_t)un * 16u + 8u);
        if (ent != (NONE << 16 | NONE)) {
          const int f = ldsi(sA + (uint32_t)un * 16u + 12u), start = f >> 8, d = f & F_UP ? -1 : 1;
          const int cu = ldsi(sB + (uint32_t)un * 16u + 12u);
          const float* v = ival + (step & 1) * vstep;
          float* const Un = cur ? U0 : U1;
          __nv_bfloat16* const En = cur ? E0 : E1;
          if (ent >> 16 != NONE) {  // a line: one row, one entry per point at most
            const int r = start + d * (int)(ent >> 16), l = r * sx + 4 + 4 * cu;
            const ushort4 k = uline[un];
            const float val[4] = {v[k.x], v[k.y], v[k.z], v[k.w]};
            float4 x = *reinterpret_cast<const float4*>(Un + l);
            float o[4] = {x.x, x.y, x.z, x.w};
            if (COMP) {
              const float4 ee = bf4(*reinterpret_cast<const uint2*>(En + l));
              float eo[4] = {ee.x, ee.y, ee.z, ee.w};
#pragma unroll
              for (int p = 0; p < 4; ++p) {
                float err;
                o[p] = two_sum(o[p], val[p], &err);
                eo[p] += err;
              }
              *reinterpret_cast<uint2*>(En + l) = to_bf4(make_float4(eo[0], eo[1], eo[2], eo[3]));
            } else {
#pragma unroll
              for (int p = 0; p < 4; ++p) o[p] = o[p] + val[p];
            }
            x = make_float4(o[0], o[1], o[2], o[3]);
            *reinterpret_cast<float4*>(Un + l) = x;
            if (keep) *reinterpret_cast<float4*>(glev + (long long)(z0 + H + r) * px + HX + 4 * cu) = x;
          }
          // a chain: by node, a node's entries in index order
          for (uint32_t i = LEAN ? NONE : ent & NONE; i != NONE;) {
            const uint32_t l = il[i] >> 16;
            float x = Un[l], xe = COMP ? __bfloat162float(En[l]) : 0.f;
            auto add = [&](float val) {
              if (COMP) {
                float err;
                x = two_sum(x, val, &err);
                xe += err;
              } else {
                x = x + val;
              }
            };
            if (WALK) {
              const int n = il[i] & MANY ? nxt[i] : 1;
#pragma unroll 4
              for (int k = 0; k < n; ++k) add(v[i + k]);
              i = nxt[i + n - 1];
            } else {  // (as above it spills)
              for (; i != NONE && il[i] >> 16 == l; i = nxt[i]) add(v[i]);
            }
            Un[l] = x;
            if (COMP) En[l] = __float2bfloat16(xe);
            const int r = (int)l / sx;
            if (keep) glev[(long long)(z0 + H + r) * px + HX + ((int)l - r * sx - 4)] = x;
          }
        }
        if (BAND && ent != (NONE << 16 | NONE) && step + 1 < a.nsteps) {
          const int4 A = ldsi4(sA + (uint32_t)un * 16u);
          if (A.w & F_LATE) {
            const uint32_t w = (uint32_t)ldsi(sB + (uint32_t)un * 16u) + epar - (tag & 1u) * epar;
            for (int j = 0; j < R; ++j) {
              const uint32_t x = sU0 + (cur ? 0u : lbytes) + (uint32_t)(A.x + j * (A.w & F_UP ? -rs : rs));
              publish(w + (uint32_t)(j * (A.w & F_UP ? -(int)erow : (int)erow)), lds4(x),
                      COMP ? lds2(neff + x / 2u) : make_uint2(0u, 0u), tag + 1);
            }
          }
        }
      }
      if (!WALK && ldsi(sLead)) {  // the other units' entries: a thread adds all of a node's, in order
        __syncthreads();
        const float* v = ival + (step & 1) * vstep;
        float* const Un = cur ? U0 : U1;
        __nv_bfloat16* const En = cur ? E0 : E1;
        for (int i = tid; i < ni; i += C2_THREADS) {
          const uint32_t e = il[i], l = e >> 16;
          if (!(e & LEAD)) continue;
          const int n = nxt[i];
          float x = Un[l], xe = COMP ? __bfloat162float(En[l]) : 0.f;
#pragma unroll 4
          for (int k = 0; k < n; ++k) {
            if (COMP) {
              float err;
              x = two_sum(x, v[i + k], &err);
              xe += err;
            } else {
              x = x + v[i + k];
            }
          }
          Un[l] = x;
          if (COMP) En[l] = __float2bfloat16(xe);
          const int r = (int)l / sx;
          if (keep) glev[(long long)(z0 + H + r) * px + HX + ((int)l - r * sx - 4)] = x;
        }
      }
      if (ni > 0 && step + 1 < a.nsteps) {
#pragma unroll
        for (int q = 0; q < PER; ++q)
          if (tid + q * C2_THREADS < ni) ival[((step + 1) & 1) * vstep + tid + q * C2_THREADS] = pv[q];
      }
      // the words of the next level's edge rows, on their way while the CTA gathers
      if (step + 1 < a.nsteps) ask_ahead(tag + 1);
      slot_new += a.dir;
      glev += a.dir * a.L.field;
      if (slot_new == a.nslots || slot_new < 0) {
        glev -= a.dir * (long long)a.nslots * a.L.field;
        slot_new = slot_new < 0 ? a.nslots - 1 : 0;
      }
      __syncthreads();  // the new level is complete in this band
      if (!BAND) cluster_arrive();
    }
    // the last level's receivers, and the low parts of the last two levels
    // (the next launch starts from them)
    const int lfin = a.lev0 + a.nsteps * a.dir;
    if (ns > 0) sample(lfin, a.nsteps & 1 ? U1 : U0);
    if (COMP)
      for (int i = tid; i < nrow * nx4; i += C2_THREADS) {
        const int r = i / nx4, c = i - r * nx4;
        const long long go = (long long)(z0 + r + H) * px + HX + 4 * c;
        const size_t so = (size_t)r * sx + 4 + 4 * c;
        *reinterpret_cast<uint2*>(eb + (long long)(lfin & 1) * a.L.field + go) =
            *reinterpret_cast<const uint2*>((a.nsteps & 1 ? E1 : E0) + so);
        *reinterpret_cast<uint2*>(eb + (long long)((lfin - a.dir) & 1) * a.L.field + go) =
            *reinterpret_cast<const uint2*>((a.nsteps & 1 ? E0 : E1) + so);
      }
    // after a wait that gave up (here or in a neighbour, before its rows came
    // here): the last level's samples and a node of it are NaN, so that no result
    // formed from invalid rows passes for a valid one
    if (BAND && (*aborted || (*static_cast<volatile int*>(a.err) & 1))) {
      const float nan = __int_as_float(0x7fffffff);
      if (ns > 0 && a.samp_out && lfin + a.samp_shift >= 0) {
        float* out = a.samp_out + (long long)shot * a.samp_out_ss + (long long)(lfin + a.samp_shift) * a.nsamp;
        for (int i = tid; i < ns; i += C2_THREADS) out[sl[i] & 0xffffu] = nan;
      }
      if (tid == 0) ring[slot(lfin) + (long long)(z0 + H) * px + HX] = nan;
    }
    if (!BAND) cluster_wait();  // no CTA leaves (or starts the next shot) while a neighbour reads its band
    __syncthreads();            // this shot's lists and levels are no longer read
  }
}

// list capacity for n entries (a band may hold all of a shot's entries)
int c2_cap(int n) { return (std::max(n, 1) + 3) / 4 * 4; }

// shared memory of a band of rpc rows (chunks of N)
size_t c2_bytes(int rpc, int N, int sx, int nx4, int R, int mode, bool band, bool c2s, int sw, int capi, int caps) {
  const size_t units = band || c2s ? (size_t)(rpc / N) * nx4 : 0;  // with entries in the tables (lean: none)
  size_t b = (size_t)(2 * rpc + (band ? 0 : 1)) * sx * 4;   // both levels, zero row
  if (mode == C2_COMP) b += (size_t)(2 * rpc + (band ? 3 * R : 0)) * sx * 2;  // low parts of both levels (bf16)
  if (c2s) b += (size_t)rpc * nx4 * 16;                     // c2
  b += (size_t)capi * (4 + 8 + 2) + 32 + (size_t)caps * 4;  // injection and sampling entries
  b += units * 40 + (units + 1) / 2 * 4 + 8;                // per unit
  b += (size_t)(4 + C2_THREADS / 32) * 4;                   // counts
  if (!band) b += (size_t)8 * R * 4;                        // edge row table
  if (mode == C2_DAMP) b += (size_t)(sw + 1) * 8 + 8;
  return (b + 15) / 16 * 16;
}

// Whether a shot of this grid fits one cluster of C CTAs, for the acceptance
// of the compensated form: an upper bound of what a lean cluster of these CTAs
// needs (c2_bytes without c2: at least 32 rpc + 32 R + 2 cap - 40 bytes less), so
// that every grid accepted has a plan.
bool c2_accepts(const Layout& L, int R, int C, int cap) {
  const int nx4 = (L.nx + 3) / 4, sx = 4 * nx4 + 8;
  const int rpc = (L.nz + C - 1) / C;
  if (nx4 > C2_MAXCOL) return false;
  size_t b = (size_t)(2 * rpc + 1) * sx * 4 + (size_t)2 * rpc * sx * 2;
  b += (size_t)2 * 2 * (rpc + 2 * R) * sizeof(void*) + (size_t)cap * 20 + (size_t)(4 + C2_THREADS / 32) * 4;
  return (b + 15) / 16 * 16 <= C2_SMEM;
}

struct C2Plan {
  int C = 0, rpc = 0, N = 0, groups = 0, c2s = 0;  // CTAs per shot, rows per CTA and unit, shots at once
  bool band = false;
  size_t smem = 0;
  double est = 0, rank = 0;  // c2_step_cost and c2_rank, all rounds
};

// rows that the marches of a column read from neighbouring CTAs
int c2_remote(int rpc, int N, int R) {
  int n = 0;
  for (int a = 0; a < rpc; a += N) n += std::max(0, R - a) + std::max(0, std::min(a + N, rpc) + R - rpc);
  return n;
}

// Estimated us of a step in which every CTA has rpc rows, marched N at a time
// (rows of nx4 columns, units of 32 per warp): a sum of the rows marched, the
// 2R queue rows that every march fills, the passes of the CTA's threads, their
// latency (by rows of a march) and, in clusters, the rows read from a neighbour's
// shared memory.  The coefficients are a least-squares fit (relative,
// non-negative) to 19036 measured splits of 480 random grids (8 to 2048 x 16 to
// 420, 1 to 128 shots, both orders, all modes); mean error 4 to 9 %.
double c2_step_cost(int rpc, int N, int nx4, int R, int mode, bool band, int c2s) {
  const int units = (rpc + N - 1) / N * nx4, passes = (units + C2_THREADS - 1) / C2_THREADS;
  const double u = units / 32.0, order8 = R == 4;
  if (band) {
    // [mode]: constant, order 8, warps, latency by N, columns, passes, rows (N = 8), rows (c2 in global memory), rows (order 8)
    static const double K[3][9] = {{1.011, 1.058, 0.0056, 0.0115, 0.318, 0.669, 0.0062, 0.0054, 0.0006},
                                   {0., 0.808, 0.0481, 0.166, 0.264, 1.318, 0.0106, 0.0054, 0.0146},
                                   {0., 0.833, 0.0454, 0.442, 0.082, 1.023, 0.0064, 0.0069, 0.0070}};
    const double* k = K[mode];
    return k[0] + k[1] * order8 + k[2] * u + k[3] * N + k[4] * nx4 / 100 + k[5] * passes +
           u * N * (k[6] * (N == 8) + k[7] * !c2s + k[8] * order8);
  }
  if (!c2s) {  // lean: constant, order 8, rows filled, passes
    static const double K[2][4] = {{1.392, 0.169, 0.0051, 0.953}, {1.086, 0.662, 0.0142, 1.594}};
    const double* k = K[mode];
    return k[0] + k[1] * order8 + k[2] * u * 2 * R + k[3] * passes;
  }
  // clusters, [mode]: constant, order 8, rows marched, rows filled, remote rows, latency by N, passes, latency by N of a pass
  static const double K[3][8] = {{1.075, 0.229, 0.0053, 0.0030, 0.125, 0., 0.168, 0.155},
                                 {1.108, 0.374, 0.0155, 0.0057, 0.192, 0., 0.085, 0.267},
                                 {1.271, 0.149, 0.0108, 0.0021, 0.087, 0.0595, 0.145, 0.322}};
  const double* k = K[mode];
  return k[0] + k[1] * order8 + k[2] * u * N + k[3] * u * 2 * R + k[4] * c2_remote(rpc, N, R) * nx4 / 1000 + k[5] * N +
         passes * (k[6] + k[7] * N);
}

// Rank of a split into bands, or into clusters of one or two rows a march: a
// step's time from measurements of medium grids, with the floor that the
// exchange of bands sets.  Near the floor the phases of the exchange decide, by
// up to 25 % and not smoothly, where the fit above is no better (by the fit alone:
// 601 x 201 x 16 shots 4.2 us instead of 3.9, 397 x 401 x 4 3.8 instead of 3.1); it
// knows no remote rows (c2_choose).
double c2_rank(int rpc, int N, int nx4, int R, int mode, bool band) {
  const int units = rpc / N * nx4, passes = (units + C2_THREADS - 1) / C2_THREADS;
  const double w = std::min(16, (units + 31) / 32);
  if (band) {
    const double row = mode == C2_COMP ? (N == 8 ? 0.066 : 0.05) : (mode == C2_DAMP ? 0.026 : 0.0185);
    const double floor = R == 4 ? 3.6 : (N == 8 ? 1.9 : 1.5) * (mode == C2_COMP ? 1.45 : 1.0);
    return std::max(floor, (mode == C2_COMP ? 1.9 : 1.6) + passes * N * row * w) + 0.03 * passes * w;
  }
  const double row = mode == C2_COMP ? 0.05 : (mode == C2_DAMP ? 0.024 : 0.02), fill = mode == C2_COMP ? 0.004 : 0.0025;
  return (N == 1 ? 1.25 : 1.4) + passes * w * (N * row + 2 * R * fill);
}

// c2s 0: c2 in global memory (bands; lean clusters)
C2Plan c2_try(const Layout& L, int R, int mode, int sw, int nshots, int C, int N, int groups, bool band, int c2s, int capi,
              int caps) {
  C2Plan p;
  const int nx4 = (L.nx + 3) / 4, sx = 4 * nx4 + 8;
  if (nx4 > C2_MAXCOL || groups < 1) return p;
  const int rows = (L.nz + C - 1) / C;
  // bands: at least two chunks, so that the rows beyond a chunk are in the band
  const int rpc = !band && !c2s ? rows : std::max((rows + N - 1) / N, band ? 2 : 1) * N;
  if ((L.nz + rpc - 1) / rpc != C) return p;  // no empty bands
  if ((size_t)rpc * sx > 65535) return p;  // the lists keep band indices in 16 bits
  const size_t sm = c2_bytes(rpc, N, sx, nx4, R, mode, band, c2s, sw, capi, caps);
  if (sm > C2_SMEM) return p;
  p.C = C; p.rpc = rpc; p.N = N; p.groups = std::min(groups, nshots); p.c2s = c2s; p.band = band; p.smem = sm;
  const double rounds = (nshots + p.groups - 1) / p.groups;
  p.est = rounds * c2_step_cost(rpc, N, nx4, R, mode, band, c2s);
  p.rank = rounds * c2_rank(rpc, N, nx4, R, mode, band);
  return p;
}

int c2_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return C2_MAXBANDS;
  }
  return std::min(sms, C2_MAXBANDS);
}

// The best split into bands of one cooperative grid (C = 0: none fits), by rank;
// fit (may be null): with a fifth of the estimate, which tells the splits at the
// floor apart (601 x 201: 26 bands of 8 rows 3.4 us, 13 of 16 4.1).  With a layer,
// whose marches are longer, both by the estimate (order 4, 601 x 201 x 16: 5.3 us,
// by rank 5.9).
C2Plan c2_bands(const Layout& L, int R, int mode, int sw, int nshots, int capi, int caps, C2Plan* fit) {
  C2Plan best, other;
  auto rank = [&](const C2Plan& p) { return mode == C2_DAMP ? p.est : p.rank; };
  const int sms = c2_sms(), most = std::min(sms, (L.nz + 7) / 8);  // (bands have 8 rows at least)
  for (int C = 1; C <= most; ++C)
    for (int N : {8, 4}) {
      C2Plan p = c2_try(L, R, mode, sw, nshots, C, N, sms / C, true, 1, capi, caps);
      if (!p.C) p = c2_try(L, R, mode, sw, nshots, C, N, sms / C, true, 0, capi, caps);
      if (!p.C) continue;
      if (!best.C || rank(p) < rank(best)) best = p;
      if (!other.C || rank(p) + 0.2 * p.est < rank(other) + 0.2 * other.est) other = p;
    }
  if (fit) *fit = other;
  return best;
}

// clusters of C CTAs with `smem` bytes each that fit on the current device at
// once (cached); without a device, what a GB300 reports
template <int R, int MODE, int N, bool C2S>
int c2_max_clusters(int C, size_t smem) {
  static std::mutex m;
  static std::vector<std::pair<long long, int>> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    static const int gb300[C2_MAXC] = {152, 76, 46, 36, 28, 23, 15, 15, 15, 13, 8, 8, 7, 7, 7, 7};
    return gb300[C - 1];
  }
  const long long key = ((long long)dev << 40) | ((long long)C << 32) | (long long)smem;
  {
    std::lock_guard<std::mutex> lk(m);
    for (auto& e : cache)
      if (e.first == key) return e.second;
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)C);
  cfg.blockDim = dim3(C2_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (smem_limit_once<sweep2d_shots<R, MODE, false, N, C2S>>((int)C2_SMEM, true) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, sweep2d_shots<R, MODE, false, N, C2S>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  std::lock_guard<std::mutex> lk(m);
  cache.emplace_back(key, n);
  return n;
}

// The split of the least rank among bands and clusters of one and two rows a
// march; another one (clusters of four rows and lean ones included) where the
// fitted estimate gives it 10 % less.  Over the 480 grids no split chosen so is
// more than 3 % slower than the one by rank alone and 52 are faster by more (1500 x
// 60 2.7 us a step instead of 5.0, 601 x 201 3.4 instead of 4.3, 2000 x 64 x 2 3.3
// instead of 4.4); by the estimate alone 13 and 104.  The chosen split takes on
// average 3.0 % longer than the best measured one (by rank 5.0 %).
template <int R, int MODE>
C2Plan c2_choose(const Layout& L, int sw, int nshots, int capi, int caps) {
  C2Plan best, base = c2_bands(L, R, MODE, sw, nshots, capi, caps, &best);
  auto cluster = [&](int C, int N, int c2s, auto at_once) {
    C2Plan p = c2_try(L, R, MODE, sw, nshots, C, N, nshots, false, c2s, capi, caps);
    if (!p.C) return;
    p = c2_try(L, R, MODE, sw, nshots, C, N, at_once(C, p.smem), false, c2s, capi, caps);
    if (p.C && (!best.C || p.est < best.est)) best = p;
    if (p.C && N <= 2 && (!base.C || p.rank < base.rank)) base = p;
  };
  for (int C = 1; C <= C2_MAXC; ++C) {
    cluster(C, 4, 1, c2_max_clusters<R, MODE, 4, true>);
    cluster(C, 2, 1, c2_max_clusters<R, MODE, 2, true>);
    cluster(C, 1, 1, c2_max_clusters<R, MODE, 1, true>);
    if constexpr (MODE != C2_DAMP) cluster(C, 4, 0, c2_max_clusters<R, MODE, 4, false>);
  }
  return !base.C || best.est < 0.9 * base.est ? best : base;
}

template <int R, int MODE, bool BAND, int N, bool C2S>
cudaError_t c2_run(const C2Args& a, const C2Plan& pl, cudaStream_t s) {
  const cudaError_t e = smem_limit_once<sweep2d_shots<R, MODE, BAND, N, C2S>>((int)C2_SMEM, !BAND);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  if (BAND) {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  } else {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)pl.C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
  }
  cfg.gridDim = dim3((unsigned)(pl.C * pl.groups));
  cfg.blockDim = dim3(C2_THREADS);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t l = cudaLaunchKernelEx(&cfg, sweep2d_shots<R, MODE, BAND, N, C2S>, a);
  return l != cudaSuccess ? l : cudaGetLastError();
}

C2Plan c2_plan(const Layout& L, const Weights& W, int mode, int nshots, int ninj, int nsamp) {
  const int capi = c2_cap(ninj), caps = c2_cap(nsamp);
#define TP_C2(RR) (mode == C2_COMP ? c2_choose<RR, C2_COMP>(L, W.sw, nshots, capi, caps)                       \
                                   : (mode == C2_DAMP ? c2_choose<RR, C2_DAMP>(L, W.sw, nshots, capi, caps)    \
                                                      : c2_choose<RR, C2_LEVELS>(L, W.sw, nshots, capi, caps)))
  return W.R == 4 ? TP_C2(4) : TP_C2(2);
#undef TP_C2
}

template <int R, int MODE>
cudaError_t c2_launch(const C2Args& a0, cudaStream_t s) {
  C2Args a = a0;
  a.capi = c2_cap(a.ninj);
  a.caps = c2_cap(a.nsamp);
  const C2Plan pl = c2_choose<R, MODE>(a.L, a.W.sw, a.nshots, a.capi, a.caps);
  if (!pl.C || (pl.band && !a.edge)) return cudaErrorInvalidConfiguration;
  a.C = pl.C;
  a.rpc = pl.rpc;
  a.nx4 = (a.L.nx + 3) / 4;
  a.sx = 4 * a.nx4 + 8;
  if (pl.band) {
    if (pl.N == 4) return pl.c2s ? c2_run<R, MODE, true, 4, true>(a, pl, s) : c2_run<R, MODE, true, 4, false>(a, pl, s);
    return pl.c2s ? c2_run<R, MODE, true, 8, true>(a, pl, s) : c2_run<R, MODE, true, 8, false>(a, pl, s);
  }
  if constexpr (MODE != C2_DAMP)
    if (!pl.c2s) return c2_run<R, MODE, false, 4, false>(a, pl, s);
  return pl.N == 4   ? c2_run<R, MODE, false, 4, true>(a, pl, s)
         : pl.N == 2 ? c2_run<R, MODE, false, 2, true>(a, pl, s)
                     : c2_run<R, MODE, false, 1, true>(a, pl, s);
}

}  // namespace

bool compensated2d_fits(const Layout& L, const Weights& W, int nsrc, int nrec) {
  if (L.ndim != 2 || W.sw > 0) return false;
  if (nsrc > C2_MAXLIST || nrec > C2_MAXLIST) return false;
  // the larger of the two sets in both lists covers the forward and the adjoint launches
  const int cap = c2_cap(std::max(nsrc, nrec));
  for (int C = 1; C <= C2_MAXC; ++C)
    if (c2_accepts(L, W.R, C, cap)) return true;
  return false;
}

bool persist2d_fits(const Layout& L, const Weights& W, int nshots, int nsrc, int nrec) {
  if (L.ndim != 2 || nsrc > C2_MAXLIST || nrec > C2_MAXLIST) return false;
  const int cap = c2_cap(std::max(nsrc, nrec));
  return c2_bands(L, W.R, W.sw > 0 ? C2_DAMP : C2_LEVELS, W.sw, nshots, cap, cap, nullptr).C > 0;
}

void plan2d(const Layout& L, const Weights& W, bool comp, int nshots, int ninj, int nsamp, int plan[6]) {
  const C2Plan p = c2_plan(L, W, comp ? C2_COMP : (W.sw > 0 ? C2_DAMP : C2_LEVELS), nshots, ninj, nsamp);
  const int v[6] = {p.C ? (p.band ? 1 : 2) : 0, p.C, p.rpc, p.N, p.groups, p.c2s};
  std::copy(v, v + 6, plan);
}

size_t edge2d_bytes(const Layout& L, const Weights& W, int nshots, bool comp) {
  const long long ctas = std::min<long long>(C2_MAXBANDS, (long long)nshots * ((L.nz + 7) / 8));  // bands have 8 rows at least
  return (size_t)ctas * 4 * W.R * ((L.nx + 3) / 4) * 16 * (comp ? 3 : 2);
}

cudaError_t launch_cluster2d(const Cluster2dArgs& c, cudaStream_t s) {
  C2Args a{};
  a.L = c.L;
  a.W = c.W;
  a.nshots = c.nshots;
  a.dir = c.dir;
  a.lev0 = c.lev0;
  a.nsteps = c.nsteps;
  a.fresh = c.fresh;
  a.store_all = c.store_all;
  a.ring = c.ring; a.nslots = c.nslots; a.ring_ss = c.ring_ss;
  a.eslots = reinterpret_cast<__nv_bfloat16*>(c.eslots); a.e_ss = c.e_ss;
  a.c2 = c.c2;
  a.inj_off = c.inj_off; a.inj_coef = c.inj_coef; a.ninj = c.ninj;
  a.inj_val = c.inj_val; a.inj_val_ss = c.inj_val_ss; a.inj_shift = c.inj_shift;
  a.samp_off = c.samp_off; a.nsamp = c.nsamp;
  a.samp_out = c.samp_out; a.samp_out_ss = c.samp_out_ss; a.samp_shift = c.samp_shift;
  a.edge = static_cast<unsigned char*>(c.edge);
  a.tag0 = c.tag0;
  a.spin = wait_limit_cycles();
  a.err = c.err;
  prof_before(0, s);  // TP_KERNEL_STENCIL
  cudaError_t e;
  const int mode = c.comp ? C2_COMP : (c.W.sw > 0 ? C2_DAMP : C2_LEVELS);
#define TP_C2(RR) (mode == C2_COMP ? c2_launch<RR, C2_COMP>(a, s)                         \
                                   : (mode == C2_DAMP ? c2_launch<RR, C2_DAMP>(a, s) : c2_launch<RR, C2_LEVELS>(a, s)))
  e = c.W.R == 4 ? TP_C2(4) : TP_C2(2);
#undef TP_C2
  prof_after(0, s);
  return e;
}

}  // namespace tp

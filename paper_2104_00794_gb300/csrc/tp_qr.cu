// Range-finding probes (Eq. 6): Q_s = qr(D_s D_s^T Z_s) for every shot s,
// D_s the observed record as an nt x nrec matrix and Z_s random probes.
//
//   W = D^T Z   (nrec x r)   one thread per receiver and part of the time axis
//   Y = D W     (nt x r)     tiles of 32 time levels, 2 x 2 sums per thread
//   Q = orth(Y)              classical Gram-Schmidt applied twice per column
//                            (stable for a numerically full-rank Y), one
//                            cluster per shot; diag(R) > 0
// All sums are fp64, at 1.6 operations per clock and SM the bound of every
// kernel here: a record of 2500 x 801 samples, 8 shots, r = 16 needs 2 x 256 M
// multiply-adds (1.05 ms at the measured rate).  So the work is spread over all
// SMs (the time axis of W in parts, added in order; 8 CTAs per shot in
// Gram-Schmidt), operands are converted once, and no sum goes through a wide
// shuffle tree.  Before, a thread per receiver walked the whole time axis
// (6.6 ms on 56 CTAs), a warp per level summed by shuffles (1.2 ms) and one CTA
// per shot orthogonalised (1.5 ms): 9.46 ms for that record, now 1.56 ms.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdio>

#include "tp_internal.h"
#include "tprobe.h"

namespace tp {

namespace {

namespace cg = cooperative_groups;

constexpr int QR_RMAX = 32;
constexpr int QR_THREADS = 256;
constexpr int QR_CLUSTER = 8;  // CTAs per shot in Gram-Schmidt
constexpr int QR_TB = 32;      // time levels staged at once (W), per tile (Y)
constexpr int QR_JB = 64;      // receivers per tile of Y

// part p of W: sum over the levels [p chunk, (p + 1) chunk)
template <int RP>
__global__ void __launch_bounds__(128) qr_dtz_kernel(const float* __restrict__ D, const float* __restrict__ Z, int nt,
                                                     int nrec, int r, int chunk, double* __restrict__ part) {
  __shared__ __align__(16) double zs[QR_TB * RP];
  const int s = blockIdx.z, p = blockIdx.y, j = blockIdx.x * 128 + threadIdx.x;
  const int t0 = p * chunk, t1 = min(nt, t0 + chunk);
  const float* Ds = D + (long long)s * nt * nrec + min(j, nrec - 1);
  const float* Zs = Z + (long long)s * nt * r;
  double acc[RP];
#pragma unroll
  for (int i = 0; i < RP; ++i) acc[i] = 0.0;
  for (int b = t0; b < t1; b += QR_TB) {
    __syncthreads();
    for (int e = threadIdx.x; e < QR_TB * RP; e += 128) {
      const int t = b + e / RP, i = e % RP;
      zs[e] = (t < t1 && i < r) ? (double)Zs[(long long)t * r + i] : 0.0;
    }
    __syncthreads();
    const int m = min(QR_TB, t1 - b);
#pragma unroll 4
    for (int t = 0; t < m; ++t) {
      const double d = Ds[(long long)(b + t) * nrec];
#pragma unroll
      for (int i = 0; i < RP; ++i) acc[i] += d * zs[t * RP + i];
    }
  }
  if (j >= nrec) return;
  double* o = part + (((long long)p * gridDim.z + s) * nrec + j) * r;
#pragma unroll
  for (int i = 0; i < RP; ++i)
    if (i < r) o[i] = acc[i];
}

// W = its parts, added in order
__global__ void __launch_bounds__(256) qr_parts_kernel(const double* __restrict__ part, int nparts, long long n,
                                                       double* __restrict__ W) {
  for (long long e = blockIdx.x * 256LL + threadIdx.x; e < n; e += gridDim.x * 256LL) {
    double v = part[e];
    for (int p = 1; p < nparts; ++p) v += part[p * n + e];
    W[e] = v;
  }
}

// a tile of QR_TB levels of Y: thread (row pair, column pair), RP / 2 column pairs
template <int RP>
__global__ void __launch_bounds__(QR_TB / 2 * RP / 2) qr_dw_kernel(const float* __restrict__ D, const double* __restrict__ W,
                                                                   int nt, int nrec, int r, double* __restrict__ Y) {
  constexpr int NT = QR_TB / 2 * RP / 2;
  __shared__ __align__(16) double ds[QR_JB][QR_TB + 2];  // [receiver][level]
  __shared__ __align__(16) double ws[QR_JB][RP];
  const int s = blockIdx.y, t0 = blockIdx.x * QR_TB, tid = threadIdx.x;
  const int c = tid % (RP / 2), q = tid / (RP / 2);
  const float* Dt = D + ((long long)s * nt + t0) * nrec;
  const double* Ws = W + (long long)s * nrec * r;
  double a00 = 0.0, a01 = 0.0, a10 = 0.0, a11 = 0.0;
  for (int j0 = 0; j0 < nrec; j0 += QR_JB) {
    __syncthreads();
    for (int e = tid; e < QR_JB * QR_TB; e += NT) {
      const int j = e % QR_JB, t = e / QR_JB;
      ds[j][t] = (j0 + j < nrec && t0 + t < nt) ? (double)Dt[(long long)t * nrec + j0 + j] : 0.0;
    }
    for (int e = tid; e < QR_JB * RP; e += NT) {
      const int j = e / RP, i = e % RP;
      ws[j][i] = (j0 + j < nrec && i < r) ? Ws[(long long)(j0 + j) * r + i] : 0.0;
    }
    __syncthreads();
    const int m = min(QR_JB, nrec - j0);
#pragma unroll 4
    for (int j = 0; j < m; ++j) {
      const double2 d = *reinterpret_cast<const double2*>(&ds[j][2 * q]), w = *reinterpret_cast<const double2*>(&ws[j][2 * c]);
      a00 += d.x * w.x;
      a01 += d.x * w.y;
      a10 += d.y * w.x;
      a11 += d.y * w.y;
    }
  }
  const int t = t0 + 2 * q, i = 2 * c;
  double* y = Y + ((long long)s * nt + t) * r + i;
  if (t < nt && i < r) y[0] = a00;
  if (t < nt && i + 1 < r) y[1] = a01;
  if (t + 1 < nt && i < r) y[r] = a10;
  if (t + 1 < nt && i + 1 < r) y[r + 1] = a11;
}

// Y is overwritten by the orthonormal Q (fp64); Qf receives it in fp32.  A
// cluster per shot, its CTAs share the levels; every sum over the levels is
// formed per thread, CTA and cluster in a fixed order.
__global__ void __cluster_dims__(QR_CLUSTER, 1, 1) __launch_bounds__(QR_THREADS)
qr_cgs2_kernel(double* __restrict__ Y, int nt, int r, float* __restrict__ Qf, int* err) {
  __shared__ double seg[QR_THREADS];                 // a thread's share of a dot product
  __shared__ double sums[2][QR_RMAX];                // this CTA's share (two buffers: the next dot products may start early)
  __shared__ double h[QR_RMAX];
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), s = blockIdx.x / QR_CLUSTER, tid = threadIdx.x;
  const int per = (nt + QR_CLUSTER - 1) / QR_CLUSTER, t0 = min(nt, rank * per), t1 = min(nt, t0 + per);
  double* Ys = Y + (long long)s * nt * r;
  const int rp = r <= 8 ? 8 : (r <= 16 ? 16 : 32);   // threads per level in a dot product
  const int i = tid % rp, g = tid / rp, ng = QR_THREADS / rp;
  int buf = 0;
  // h[i] = column i . column k over the cluster, i < n (h[0] = |column k|^2 for n = 0)
  auto dots = [&](int n, int k) {
    const int m = n ? n : 1;
    double acc = 0.0;
    if (i < m)
      for (int t = t0 + g; t < t1; t += ng) {
        const double v = Ys[(long long)t * r + k];
        acc += v * (n ? Ys[(long long)t * r + i] : v);
      }
    seg[tid] = acc;
    __syncthreads();
    if (tid < m) {
      double v = 0.0;
      for (int q = 0; q < ng; ++q) v += seg[q * rp + tid];
      sums[buf][tid] = v;
    }
    cluster.sync();
    if (tid < m) {
      double v = 0.0;
      for (int c = 0; c < QR_CLUSTER; ++c) v += *cluster.map_shared_rank(&sums[buf][tid], c);
      h[tid] = v;
    }
    buf ^= 1;
    __syncthreads();
  };
  for (int k = 0; k < r; ++k) {
    dots(0, k);
    const double n0 = h[0];
    __syncthreads();
    for (int pass = 0; pass < 2 && k > 0; ++pass) {  // twice is enough
      dots(k, k);
      for (int t = t0 + tid; t < t1; t += QR_THREADS) {
        double v = Ys[(long long)t * r + k];
        for (int c = 0; c < k; ++c) v -= Ys[(long long)t * r + c] * h[c];
        Ys[(long long)t * r + k] = v;
      }
      __syncthreads();
    }
    dots(0, k);
    const double nn = h[0];
    // a column that vanished relative to its own size: numerically rank deficient
    const bool dep = !(nn > 1e-24 * n0) || nn <= 0.0;
    if (dep && tid == 0 && rank == 0) atomicOr(err, 4);
    const double inv = dep ? 0.0 : 1.0 / sqrt(nn);
    for (int t = t0 + tid; t < t1; t += QR_THREADS) {
      const double v = Ys[(long long)t * r + k] * inv;
      Ys[(long long)t * r + k] = v;
      Qf[((long long)s * nt + t) * r + k] = (float)v;
    }
    __syncthreads();
  }
  cluster.sync();  // no CTA leaves while another reads its sums
}

long long up256(long long b) { return (b + 255) / 256 * 256; }

struct QrLayout {
  size_t o_err, o_Z, o_W, o_Y, o_part, bytes;
  int nparts, chunk;  // parts of the time axis in W = D^T Z
};

QrLayout qr_layout(int nt, int nrec, int nshots, int r) {
  QrLayout L{};
  size_t cur = 0;
  L.o_err = cur; cur += 256;
  L.o_Z = cur; cur += up256((long long)nshots * nt * r * sizeof(float));
  L.o_W = cur; cur += up256((long long)nshots * nrec * r * sizeof(double));
  L.o_Y = cur; cur += up256((long long)nshots * nt * r * sizeof(double));
  // enough CTAs of 128 receivers to fill the GPU a few times over
  const long long ctas = (long long)((nrec + 127) / 128) * nshots;
  L.nparts = (int)std::max<long long>(1, std::min<long long>(1024 / ctas, (nt + QR_TB - 1) / QR_TB));
  L.chunk = ((nt + L.nparts - 1) / L.nparts + QR_TB - 1) / QR_TB * QR_TB;
  L.nparts = (nt + L.chunk - 1) / L.chunk;
  L.o_part = cur; cur += L.nparts > 1 ? up256((long long)L.nparts * nshots * nrec * r * sizeof(double)) : 0;
  L.bytes = cur;
  return L;
}

}  // namespace
}  // namespace tp

extern "C" {

size_t tp_qr_workspace_bytes(int nt, int nrec, int nshots, int r) {
  if (nt < 1 || nrec < 1 || nshots < 1 || r < 1 || r > tp::QR_RMAX) return 0;
  return tp::qr_layout(nt, nrec, nshots, r).bytes;
}

tp_status tp_qr_probes(const tp_probe* probe, int nt, int nrec, int nshots, const float* d_obs, float* Q, void* ws,
                       size_t ws_bytes, void* stream) {
  using namespace tp;
  char buf[160];
  auto bad = [&](tp_status st, const char* m) {
    snprintf(buf, sizeof(buf), "tp_qr_probes: %s", m);
    set_last_error(buf);
    return st;
  };
  if (!probe || !d_obs || !Q || !ws) return bad(TP_ERR_ARG, "NULL argument");
  if (probe->kind != TP_PROBE_RADEMACHER && probe->kind != TP_PROBE_GAUSSIAN)
    return bad(TP_ERR_ARG, "the random probes Z must be Rademacher or Gaussian");
  if (probe->r < 1 || probe->r > QR_RMAX) return bad(TP_ERR_ARG, "r must be in 1..32");
  if (nt < probe->r) return bad(TP_ERR_ARG, "nt must be >= r");
  if (nrec < 1 || nshots < 1) return bad(TP_ERR_ARG, "nrec and nshots must be >= 1");
  if (reinterpret_cast<uintptr_t>(ws) % 256) return bad(TP_ERR_ARG, "workspace must be 256-byte aligned");
  const QrLayout L = qr_layout(nt, nrec, nshots, probe->r);
  if (ws_bytes < L.bytes) return bad(TP_ERR_NOMEM, "workspace too small");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(ws);
  const int r = probe->r;
  cudaError_t e = cudaMemsetAsync(w + L.o_err, 0, 256, st);
  if (e == cudaSuccess) e = launch_probes(probe->kind, nt, r, probe->seed, 0, nshots, nullptr,
                                          reinterpret_cast<float*>(w + L.o_Z), st);
  if (e == cudaSuccess) {
    prof_before(5, st);
    const float* Z = reinterpret_cast<const float*>(w + L.o_Z);
    double* W = reinterpret_cast<double*>(w + L.o_W);
    double* Y = reinterpret_cast<double*>(w + L.o_Y);
    double* part = L.nparts > 1 ? reinterpret_cast<double*>(w + L.o_part) : W;
    const dim3 gw((nrec + 127) / 128, L.nparts, nshots), gy((nt + QR_TB - 1) / QR_TB, nshots);
#define TP_QR(RP)                                                                          \
  do {                                                                                     \
    qr_dtz_kernel<RP><<<gw, 128, 0, st>>>(d_obs, Z, nt, nrec, r, L.chunk, part);           \
    if (L.nparts > 1) {                                                                    \
      const long long n = (long long)nshots * nrec * r;                                    \
      qr_parts_kernel<<<(unsigned)std::min<long long>((n + 255) / 256, 2048), 256, 0, st>>>(part, L.nparts, n, W); \
    }                                                                                      \
    qr_dw_kernel<RP><<<gy, QR_TB / 2 * RP / 2, 0, st>>>(d_obs, W, nt, nrec, r, Y);         \
  } while (0)
    if (r <= 4) TP_QR(4);
    else if (r <= 8) TP_QR(8);
    else if (r <= 16) TP_QR(16);
    else TP_QR(32);
#undef TP_QR
    qr_cgs2_kernel<<<nshots * QR_CLUSTER, QR_THREADS, 0, st>>>(Y, nt, r, Q, reinterpret_cast<int*>(w + L.o_err));
    prof_after(5, st);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    snprintf(buf, sizeof(buf), "tp_qr_probes: %s", cudaGetErrorString(e));
    set_last_error(buf);
    return TP_ERR_CUDA;
  }
  return TP_OK;
}

}  // extern "C"

// Wall shear stress at the Lagrangian points (Sec. 2.6): WSS = |t - (t.n) n|,
// t = 2 mu eps(u) n, with the velocity derivatives from second-order DC-PSE
// operators (the meshless method Sec. 2.6 cites) over the finest-level nodes
// around each wall point on the fluid side, FP64.
#include <algorithm>
#include <cmath>

#include "device.cuh"
#include "ibmove.hpp"
#include "wss.hpp"

namespace ibg {

IBG_KCOUNT_DEFINE
unsigned long long wss_kcount() {
  unsigned long long v = 0;
  cudaMemcpyFromSymbol(&v, g_kcount, sizeof(v));
  return v;
}

namespace {

// The candidates of a point are the finest-level nodes of a box around it
// (about 1200), of which the kernel keeps the ~90 within the cutoff on the fluid
// side.  The FP64 rate (two lanes a clock and SM) bounds the work, so a warp
// takes a point and spends FP64 on full warps of kept nodes only: the
// lanes test the box in FP32 with a margin, what passes is queued, and every 32
// queued nodes are tested exactly and summed together.  The moment matrix
// of the nine monomials holds only the 31 distinct moments of degrees 2 to 4;
// the derivatives are linear in the 27 moments of the velocity, so one pass over
// the nodes suffices.  Each set is summed over the lanes in one butterfly; the
// 9 x 9 Cholesky solves of 32 points share one warp, a point a lane.  ib_wss on
// the 32,000 points of the refined 64x64x256 tube, host copies included: 7.91 ms
// with a thread per point and two passes, 1.78 ms here (FP64 pipe 66 % busy).
constexpr int WSS_PTS = 32;       // points of a CTA
constexpr int WSS_WARPS = 8;

// a kept node's index in the box, flattened
struct Box {
  int32_t lo[3], n[3];
  __device__ __forceinline__ void node(int i, int32_t (&q)[3]) const {
    const int zy = i / n[0], z = zy / n[1];
    q[0] = lo[0] + (i - zy * n[0]);
    q[1] = lo[1] + (zy - z * n[1]);
    q[2] = lo[2] + z;
  }
};

// Exact selection of node q for the point at X with normal np_.  Distances and
// projections are rounded term by term (no fused multiply-add) so that the
// selection is exactly that of a plain evaluation.
__device__ __forceinline__ bool selected(const MoveGrid& G, const double* X, const double* np_, double rc2,
                                         const int32_t (&q)[3], double (&d)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) d[a] = __dsub_rn(__dadd_rn(G.origin[a], __dmul_rn(double(q[a]), G.hf[a])), X[a]);
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
  if (!(r2 <= rc2)) return false;
  const double dn = __dadd_rn(__dadd_rn(__dmul_rn(d[0], np_[0]), __dmul_rn(d[1], np_[1])), __dmul_rn(d[2], np_[2]));
  return dn < 0.0;
}

// Calls body(valid, slot, d) for the kept nodes of a point, 32 at a time over the
// lanes of the warp (every lane takes part, valid or not); returns their number.
// queue: 64 entries of the warp.
template <typename Body>
__device__ __forceinline__ int for_nodes(const MoveGrid& G, const double* X, const double* np_, double rc2,
                                         const float (&h)[3], const int32_t (&rad)[3], int2* queue, Body&& body) {
  const int lane = threadIdx.x & 31;
  Box box;
  float f[3], nf[3];
  int32_t c[3];
  double nmax = fmax(fabs(np_[0]), fmax(fabs(np_[1]), fabs(np_[2])));
  // the FP32 test is in units of the largest spacing (h: the spacings in them), so
  // that no length of a problem leaves the FP32 range; normals that FP32
  // cannot scale are left to the exact test
  const bool plain = nmax >= 1e-300 && isfinite(np_[0]) && isfinite(np_[1]) && isfinite(np_[2]);
  const double rn = 1.0 / nmax;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double x = (X[a] - G.origin[a]) / G.hf[a];
    c[a] = int32_t(floor(x));
    box.lo[a] = max(c[a] - rad[a], 0);
    box.n[a] = max(0, min(c[a] + 1 + rad[a], int32_t(G.nf[a])) - box.lo[a] + 1);
    f[a] = float(x - double(c[a])) * h[a];
    nf[a] = plain ? float(np_[a] * rn) : 0.f;
  }
  constexpr float r2max = float(WSS_RADIUS * WSS_RADIUS * 1.001), dmax = float(1e-3 * WSS_RADIUS);
  const int n = box.n[0] * box.n[1] * box.n[2];
  int kept = 0, in = 0;   // nodes of the queue (uniform over the warp)
  auto flush = [&](int m) {
    __syncwarp();
    const bool on = lane < m;
    const int2 e = queue[on ? lane : 0];
    int32_t q[3];
    double d[3];
    box.node(e.x, q);
    const bool ok = on && selected(G, X, np_, rc2, q, d);
    kept += __popc(__ballot_sync(0xffffffffu, ok));
    body(ok, e.y, d);
    __syncwarp();
  };
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane;
    bool pass = false;
    int32_t slot = 0;
    if (i < n) {
      int32_t q[3];
      box.node(i, q);
      const float dx = float(q[0] - c[0]) * h[0] - f[0], dy = float(q[1] - c[1]) * h[1] - f[1],
                  dz = float(q[2] - c[2]) * h[2] - f[2];
      if (dx * dx + dy * dy + dz * dz <= r2max && (!plain || dx * nf[0] + dy * nf[1] + dz * nf[2] <= dmax)) {
        const int32_t b = G.bmap[(int64_t(q[2] / DBS) * G.nb[1] + q[1] / DBS) * G.nb[0] + q[0] / DBS];
        if (b >= 0) {
          slot = b * DBV + ((q[2] % DBS) * DBS + (q[1] % DBS)) * DBS + (q[0] % DBS);
          pass = (G.meta[slot] & D_VALID) != 0;
        }
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, pass);
    if (pass) queue[in + __popc(m & ((1u << lane) - 1u))] = make_int2(i, slot);
    in += __popc(m);
    if (in >= 32) {
      flush(32);
      in -= 32;
      if (lane < in) queue[lane] = queue[32 + lane];
      __syncwarp();
    }
  }
  if (in > 0) flush(in);
  return kept;
}

// index of moment x^a y^b z^c (2 <= a + b + c <= 4) in the order the sums are made
__host__ __device__ constexpr int moment(int a, int b, int c) {
  const int d = a + b + c, off = d == 2 ? 0 : d == 3 ? 6 : 16;
  int k = 0;
  for (int x = d; x >= 0; --x)
    for (int y = d - x; y >= 0; --y, ++k)
      if (x == a && y == b) return off + k;
  return -1;
}
// the nine monomials z^alpha, 1 <= |alpha| <= 2, first-degree ones first
__host__ __device__ constexpr int alpha(int r, int a) {
  constexpr int t[9][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {2, 0, 0}, {1, 1, 0}, {1, 0, 1}, {0, 2, 0}, {0, 1, 1}, {0, 0, 2}};
  return t[r][a];
}
__host__ __device__ constexpr int moment_of(int r, int c) {
  return moment(alpha(r, 0) + alpha(c, 0), alpha(r, 1) + alpha(c, 1), alpha(r, 2) + alpha(c, 2));
}

// Sum over the lanes of 32 values, value k in lane k.
__device__ __forceinline__ double transpose_sum(double (&a)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int b = 0; b < 5; ++b) {
    const int off = 16 >> b;
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int j = 0; j < off; ++j) {
      const double send = up ? a[j] : a[j + off], keep = up ? a[j + off] : a[j];
      a[j] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  return a[0];
}

__global__ void __launch_bounds__(32 * WSS_WARPS)
    k_wss(MoveGrid G, int64_t M, const double* __restrict__ X, const double* __restrict__ UB,
          const double* __restrict__ nrm, const double* __restrict__ u, int64_t ns, double eps, double rc2,
          float hx, float hy, float hz, int32_t rx, int32_t ry, int32_t rz, double mu2, double* __restrict__ wss,
          double* __restrict__ grad, int32_t* __restrict__ err) {
  KCOUNT();
  __shared__ double mom[WSS_PTS][33];       // sum_q w_q z_q^gamma of every point
  __shared__ double rhs[WSS_PTS][33];       // sum_q w_q P_r(z_q) (u_i(q) - U_B,i), at 9 i + r
  __shared__ int cnt[WSS_PTS];
  __shared__ int2 queue[WSS_WARPS][64];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t p0 = int64_t(blockIdx.x) * WSS_PTS;
  const int np = int(min(int64_t(WSS_PTS), M - p0));
  const int32_t rad[3] = {rx, ry, rz};
  const float h[3] = {hx, hy, hz};
  const double inv = 1.0 / eps;
  for (int k = w; k < np; k += WSS_WARPS) {
    const double* ub = UB + 3 * (p0 + k);
    double m[32], b[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) m[j] = b[j] = 0.0;
    const int n = for_nodes(G, X + 3 * (p0 + k), nrm + 3 * (p0 + k), rc2, h, rad, queue[w],
                            [&](bool ok, int32_t s, const double (&d)[3]) {
      if (!ok) return;
      const double x = d[0] * inv, y = d[1] * inv, z = d[2] * inv;
      const double wt = exp(-(x * x + y * y + z * z));
      // every moment from one of a degree less; x leads, then y, then z
      const double g1[3] = {wt * x, wt * y, wt * z};
      double g2[6], g3[10];
      g2[0] = g1[0] * x; g2[1] = g1[0] * y; g2[2] = g1[0] * z;
      g2[3] = g1[1] * y; g2[4] = g1[1] * z; g2[5] = g1[2] * z;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const double du = u[(int64_t)i * ns + s] - ub[i];
#pragma unroll
        for (int r = 0; r < 9; ++r) b[9 * i + r] = fma(du, r < 3 ? g1[r < 3 ? r : 0] : g2[r < 3 ? 0 : r - 3], b[9 * i + r]);
      }
#pragma unroll
      for (int j = 0; j < 6; ++j) g3[j] = g2[j] * x;
      g3[6] = g2[3] * y; g3[7] = g2[4] * y; g3[8] = g2[5] * y; g3[9] = g2[5] * z;
#pragma unroll
      for (int j = 0; j < 6; ++j) m[j] += g2[j];
#pragma unroll
      for (int j = 0; j < 10; ++j) m[6 + j] += g3[j];
#pragma unroll
      for (int j = 0; j < 10; ++j) m[16 + j] = fma(g3[j], x, m[16 + j]);
#pragma unroll
      for (int j = 6; j < 10; ++j) m[20 + j] = fma(g3[j], y, m[20 + j]);
      m[30] = fma(g3[9], z, m[30]);
    });
    mom[k][lane] = transpose_sum(m);
    rhs[k][lane] = transpose_sum(b);
    if (lane == 0) cnt[k] = n;
  }
  __syncthreads();
  // the rest with a point a lane
  if (w != 0 || lane >= np) return;
  const int64_t p = p0 + lane;
  const double* np_ = nrm + 3 * p;
  // Cholesky A = L L^T of the moment matrix A = sum_q w_q P_q P_q^T
  double A[45], rd[9];
#pragma unroll
  for (int r = 0; r < 9; ++r)
#pragma unroll
    for (int c = 0; c <= r; ++c) A[r * (r + 1) / 2 + c] = mom[lane][moment_of(r, c)];
  bool ok = cnt[lane] >= 9;
#pragma unroll
  for (int r = 0; r < 9; ++r) {
#pragma unroll
    for (int c = 0; c <= r; ++c) {
      double v = A[r * (r + 1) / 2 + c];
#pragma unroll
      for (int k = 0; k < c; ++k) v -= A[r * (r + 1) / 2 + k] * A[c * (c + 1) / 2 + k];
      if (c == r) {
        ok = ok && v > 0.0;
        A[r * (r + 1) / 2 + r] = sqrt(v);
        rd[r] = 1.0 / A[r * (r + 1) / 2 + r];
      } else {
        A[r * (r + 1) / 2 + c] = v * rd[c];
      }
    }
  }
  if (!ok) {
    atomicMax(err, 1);
    wss[p] = 0.0;
    return;
  }
  // d u_i / d x_j = (1/eps) sum_q (u_i(q) - U_B,i) eta_j(z_q) = (1/eps) (A^-1 e_j) . rhs_i
  double g[3][3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    double y[9];
#pragma unroll
    for (int r = 0; r < 9; ++r) {   // L y = e_j
      double v = r == j ? 1.0 : 0.0;
#pragma unroll
      for (int k = j; k < r; ++k) v -= A[r * (r + 1) / 2 + k] * y[k];
      y[r] = r < j ? 0.0 : v * rd[r];
    }
#pragma unroll
    for (int r = 8; r >= 0; --r) {   // L^T x = y
      double v = y[r];
#pragma unroll
      for (int k = r + 1; k < 9; ++k) v -= A[k * (k + 1) / 2 + r] * y[k];
      y[r] = v * rd[r];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      double v = 0.0;
#pragma unroll
      for (int r = 0; r < 9; ++r) v = fma(y[r], rhs[lane][9 * i + r], v);
      g[i][j] = v / eps;
    }
  }
  // t = 2 mu eps(u) n with eps(u) = (g + g^T) / 2
  double t[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    double v = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j) v += 0.5 * (g[i][j] + g[j][i]) * np_[j];
    t[i] = mu2 * v;
  }
  const double tn = t[0] * np_[0] + t[1] * np_[1] + t[2] * np_[2];
  double s2 = 0.0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double v = t[i] - tn * np_[i];
    s2 += v * v;
  }
  wss[p] = sqrt(s2);
  if (grad)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) grad[9 * p + 3 * i + j] = g[i][j];
}

}  // namespace

void wss_compute(const MoveGrid& G, const double hf[3], int64_t M, const double* X, const double* UB,
                 const double* nrm, const double* u, int64_t ns, double nu_rho, double* wss, double* grad,
                 int32_t* err, cudaStream_t st) {
  if (M == 0) return;
  const double e = std::max(hf[0], std::max(hf[1], hf[2]));
  const double rc = WSS_RADIUS * e;
  int32_t r[3];
  for (int a = 0; a < 3; ++a) r[a] = int32_t(std::ceil(rc / hf[a])) + 1;
  IBG_LAUNCH(k_wss, unsigned((M + WSS_PTS - 1) / WSS_PTS), 32 * WSS_WARPS, 0, st, G, M, X, UB, nrm, u, ns, e, rc * rc,
             float(hf[0] / e), float(hf[1] / e), float(hf[2] / e), r[0], r[1], r[2], 2.0 * nu_rho, wss,
             grad, err);
}

}  // namespace ibg

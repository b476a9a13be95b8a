// Force solve of one problem by one thread-block cluster.
//
// The PCG on S (Eq. 21-22, three right-hand sides) is a chain of several
// hundred to a thousand short dependent steps when the wall points are as
// dense as the grid (Sec. 2.5), each over a few thousand rows: as kernel
// launches an iteration is two launches and two grid reductions, all latency
// (15-25 us whatever the size).  Here a cluster of up to 16 CTAs (co-scheduled
// by the hardware, so its barriers end) runs the whole loop of one problem: rows
// in equal contiguous ranges, p of the rows around a CTA's own formed in every CTA
// that needs it from the owners' residuals (distributed shared memory), S
// kept in shared memory as far as it fits (16-bit columns into that window), partial
// sums stored straight into every CTA, two hardware barriers an iteration
// (about 500 cycles each; a third one where some CTA has no window).  It takes the
// problems for which it is the faster side (af_plan.hpp): dense systems beyond
// the shared memories and points in an order that needs p from everywhere go to the loop.
// A problem's arithmetic depends on its own rows only, so it keeps its bits
// alone and in any batch; problems of a batch run side by side.
// Bound: latency of the barriers and scalars at a few hundred rows (3.9 us an
// iteration); at some thousand dense rows barriers and shared-memory latency, the
// shared-memory pipe at 57 % (8160 rows of 41 entries: 10 us); in FP64 the FP64 pipe of
// 16 SMs, 57 % busy between barriers (2000 rows of 40: 11 us).
// A step: 8x8x16 tube 19.1 -> 5.25 ms, 16x16x64 tube in FP64 30.9 -> 13.9 ms, dense
// 32x32x128 tube 22.5 -> 11.1 ms (of which the reductions alone gave a third).
#pragma once

#include "af_plan.hpp"

namespace ibg {

__device__ __forceinline__ uint32_t cluster_addr(uint32_t smem, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem), "r"(rank));
  return a;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_load3(uint32_t a, float (&v)[3]) {
  asm volatile("{\n\t.reg .f32 pad;\n\tld.shared::cluster.v4.f32 {%0, %1, %2, pad}, [%3];\n\t}"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2])
               : "r"(a));
}
__device__ __forceinline__ void cluster_load3(uint32_t a, double (&v)[3]) {
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[2]) : "r"(a + 16));
}
__device__ __forceinline__ void cluster_load4(uint32_t a, float (&v)[4]) {
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
               : "r"(a));
}
__device__ __forceinline__ void cluster_load4(uint32_t a, double (&v)[4]) {
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a));
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v[2]), "=d"(v[3]) : "r"(a + 16));
}
__device__ __forceinline__ void window_load3(const float* a, float (&v)[3]) {
  const float4 x = *reinterpret_cast<const float4*>(a);
  v[0] = x.x, v[1] = x.y, v[2] = x.z;
}
__device__ __forceinline__ void window_load3(const double* a, double (&v)[3]) {
  const double2 x = *reinterpret_cast<const double2*>(a);
  v[0] = x.x, v[1] = x.y, v[2] = a[2];
}
__device__ __forceinline__ void cluster_store(uint32_t a, int v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// products that round on their own
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// sum over the first `width` lanes (a power of two), valid in lane 0
__device__ __forceinline__ double lanes_sum(double x, int width) {
  for (int o = width >> 1; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  return x;
}

using three = std::integral_constant<int, 3>;
using six = std::integral_constant<int, 6>;

template <typename T>
__global__ void __launch_bounds__(AFC_THREADS, 1)
    k_af_cluster(IBDev ib, const T* __restrict__ val, const T* __restrict__ dinv, T* __restrict__ x,
                 const T* __restrict__ r0, KState* __restrict__ ks) {
  KCOUNT();
  extern __shared__ __align__(16) unsigned char afc_sm[];
  __shared__ double part[2][AFC_MAX][6];   // sums of every CTA: p.q, then r.z and r.r
  __shared__ T red[6][AFC_THREADS / 32 * AFC_RPT];
  __shared__ T sal[3], sbe[3];
  __shared__ KState sk[3];
  __shared__ int win, goff[AFC_MAX];       // goff: where every CTA's own rows start in its window, -1: no window
  uint32_t rank, cl;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(cl));
  const int inst = blockIdx.x / cl;
  const int64_t R0 = int64_t(ib.seg_t[inst]) * 256;
  const int n = (ib.seg_t[inst + 1] - ib.seg_t[inst]) * 256;   // whole blocks of 256 rows
  // uniform over the cluster: nothing to do, or a problem of the loop's
  if (!(ib.af_route[inst] & (sizeof(T) == 4 ? AF_CLUSTER32 : AF_CLUSTER64)) || (ks[3 * inst].done && ks[3 * inst + 1].done && ks[3 * inst + 2].done)) return;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const AfcShape sh = afc_shape<T>(n, int(cl));
  const bool units = sh.units;
  const int rper = sh.rper, ubytes = sh.ubytes;
  const int rpc = max(0, min(n - int(rank) * rper, rper));   // rows of this CTA
  const int64_t row0 = R0 + int64_t(rank) * rper;
  const int e0 = rpc ? ib.rowptr[row0] : 0, ne = rpc ? ib.rowptr[row0 + rpc] - e0 : 0;
  // threads per row of the product: four with two chains each in FP32; two in
  // FP64, whose rate pays for every idle lane of a row's last round
  constexpr int lpr = sizeof(T) == 8 ? 2 : AFL / 2;
  // no more warps than the rows need: the others leave (the barriers count
  // the threads that are left)
  const int nt = min(AFC_THREADS, max(256, AFL * rper));
  if (t >= nt) return;
  // The rows whose p the CTA's columns need from the others: points listed along
  // the wall need a short run before and after its own.  That window of p
  // is copied once an iteration; where it does not fit (points in another
  // order) every column is read from its owner.
  if (t == 0) win = 0;
  __syncthreads();
  {
    int need = 0;
    for (int e = t; e < ne; e += nt) {
      const int k = int(ib.col[e0 + e] - row0);
      need = max(need, max(-k, k - rpc + 1));
    }
    if (need > 0) atomicMax(&win, need);
  }
  __syncthreads();
  const int own0 = min(int(rank) * rper, n);   // the problem's row of the CTA's first one
  const bool fast = win <= sh.window;
  const int G = fast ? win : 0;
  const int w0 = max(0, own0 - G), wn = min(n, own0 + rpc + G) - w0;   // window: rows [w0, w0 + wn) of the problem
  // in place of part: the sums of every 32 rows of the problem, [2][6][n / 32]
  T* unit = reinterpret_cast<T*>(afc_sm);
  T* r = reinterpret_cast<T*>(afc_sm + ubytes);   // [rper][4]: r and 1/diag, at the same place in every CTA
  T* pw = r + 4 * rper;                    // [wn][4]: p
  T* p = pw + 4 * (own0 - w0);
  T* q = pw + 4 * wn;                      // [rpc][3]
  T* cv = q + 3 * rpc;                     // cached values of S ...
  const int cap = fast ? min(ne, afc_cached<T>(sh, wn - rpc)) : 0;
  const int capr = (cap + 1) / 2 * 2;      // (an even number of 16-bit places)
  uint16_t* cc = reinterpret_cast<uint16_t*>(cv + capr);   // ... and their columns' places in the window
  int* rp = reinterpret_cast<int*>(cc + capr);             // [rpc + 1] entries relative to e0
  cluster_barrier();                       // every CTA runs
  if (t < int(cl)) cluster_store(cluster_addr(smem_u32(&goff[rank]), uint32_t(t)), fast ? own0 - w0 : -1);
  const uint32_t rbase = smem_u32(r), pbase = smem_u32(pw);
  // cluster address of r at row k of the problem
  auto owner = [&](int k) -> uint32_t {
    const int o = k / rper;
    return cluster_addr(rbase + uint32_t(k - o * rper) * uint32_t(4 * sizeof(T)), uint32_t(o));
  };
  for (int e = t; e < cap; e += nt) {
    cv[e] = val[e0 + e];
    cc[e] = uint16_t(ib.col[e0 + e] - R0 - w0);
  }
  if (rpc)
    for (int i = t; i <= rpc; i += nt) rp[i] = ib.rowptr[row0 + i] - e0;
  for (int i = t; i < rpc; i += nt) {
    r[4 * i + 3] = dinv[row0 + i];
#pragma unroll
    for (int c = 0; c < 3; ++c) r[4 * i + c] = r0[3 * (row0 + i) + c];
  }
  for (int i = t; i < 4 * wn; i += nt) pw[i] = T(0);
  if (t < 3) {
    sk[t] = ks[3 * inst + t];
    sk[t].tt = sk[t].tol2 * sk[t].bb;      // the square norm to reach
    sbe[t] = T(0);
  }
  __syncwarp();
  cluster_barrier();
  // small problems in FP32: a thread for each of the loop's eight lanes of a row
  const bool wide = sizeof(T) == 4 && nt >= AFL * rper && fast && cap == ne;
  bool all_fast = true;
  for (int o = 0; o < int(cl); ++o) all_fast = all_fast && goff[o] >= 0;
  // p at row k of the problem, from its owner
  auto column3 = [&](int k, T (&v)[3]) {
    const int o = k / rper, at = max(goff[o], 0) + k - o * rper;
    cluster_load3(cluster_addr(pbase + uint32_t(at) * uint32_t(4 * sizeof(T)), uint32_t(o)), v);
  };
  auto wrow = [&](int i) { return i < own0 - w0 ? i : i + rpc; };   // window row of the i-th row of others
  const uint32_t ghost0 = t < wn - rpc ? owner(w0 + wrow(t)) : 0u;
  // The sums over rows carry the bits of the loop's kernels in FP32 within the blocks
  // of rows that those kernels sum, in their order (p.q: 32 rows, four to a
  // warp, then eight warps; r.z and r.r: 256 rows, 32 to a warp, then eight
  // warps): an ill-conditioned S makes the number of passes, and whether FP64
  // takes over, hang on them.  Beyond the blocks both add in FP64, in another order
  // (p.q from 1025 rows on, r.z and r.r from 4097), and both round FP64 quotients
  // to FP32, so that the scalars differ only where the last bit of FP64 decides.
  auto unit_sums = [&](auto& v, auto nv, int u, int buf) {   // a warp's 32 rows, in one butterfly (warp_sums)
    constexpr int NV = decltype(nv)::value, P = NV == 3 ? 4 : 8, PB = NV == 3 ? 2 : 3;
    constexpr int off[5] = {NV == 3 ? 2 : 16, NV == 3 ? 1 : 8, NV == 3 ? 16 : 4, NV == 3 ? 8 : 2, NV == 3 ? 4 : 1};
    T a[P];
    int k = 0;
#pragma unroll
    for (int j = 0; j < P; ++j) a[j] = j < NV ? v[j < NV ? j : 0] : T(0);
#pragma unroll
    for (int b = 0; b < PB; ++b) {
      const int h = P >> (b + 1);
      const bool up = (lane & off[b]) != 0;
      if (up) k += h;
#pragma unroll
      for (int j = 0; j < h; ++j) {
        const T send = up ? a[j] : a[j + h], keep = up ? a[j + h] : a[j];
        a[j] = keep + __shfl_xor_sync(0xffffffffu, send, off[b]);
      }
    }
#pragma unroll
    for (int b = PB; b < 5; ++b) a[0] += __shfl_xor_sync(0xffffffffu, a[0], off[b]);
    // value k is in every lane with k's bits: lane o of those stores it to CTA o, ...
    int place = 0;   // the lane's number among the holders of its value
#pragma unroll
    for (int b = PB; b < 5; ++b) place = 2 * place + ((lane & off[b]) != 0);
    if (k < NV) {
      if (units) {
        for (int o = place; o < int(cl); o += 32 / P)
          cluster_store(cluster_addr(smem_u32(&unit[(6 * buf + k) * (n / 32) + own0 / 32 + u]), uint32_t(o)), a[0]);
      } else if (place == 0) {
        red[k][u] = a[0];
      }
    }
  };
  // eight warps' sums of a block of 256 rows
  auto block256 = [](const T* u) {
    return ((u[0] + u[4]) + (u[2] + u[6])) + ((u[1] + u[5]) + (u[3] + u[7]));
  };
  const int nu = rpc / 32;                 // units of this CTA
  // the CTA's sums to every CTA of the cluster (units: each warp has sent its own)
  auto exchange = [&](auto nv, int buf) {
    constexpr int NV = decltype(nv)::value;
    if (!units) {
      __syncthreads();
      if (w < NV) {
        double s = 0.0;
        if constexpr (NV == 3 || sizeof(T) == 8) {
          for (int u = lane; u < nu; u += 32) s += double(red[w][u]);
          s = lanes_sum(s, nu > 16 ? 32 : 16);
        } else {
          for (int u = lane; u < nu / 8; u += 32) s += double(block256(&red[w][8 * u]));
          s = lanes_sum(s, 8);
        }
        s = __shfl_sync(0xffffffffu, s, 0);
        if (lane < int(cl)) cluster_store(cluster_addr(smem_u32(&part[buf][rank][w]), uint32_t(lane)), s);
      }
    }
    __syncwarp();
    cluster_barrier();
  };
  // a value summed over the cluster by a warp: p.q with all lanes (valid in lane
  // 0), r.z and r.r with half of them each (k by lane; valid in lanes 0 and 16)
  auto total = [&](auto nv, int buf, int k) -> double {
    constexpr int NV = decltype(nv)::value;
    double s = 0.0;
    if constexpr (NV == 3) {
      if (units) {
        for (int u = lane; u < n / 32; u += 32) s += double(unit[(6 * buf + k) * (n / 32) + u]);
        return lanes_sum(s, n > 512 ? 32 : 16);
      }
      s = lane < int(cl) ? part[buf][lane][k] : 0.0;
      return lanes_sum(s, int(cl));
    } else {
      const int l = lane & 15;
      if (units) {
        if (l < n / 256) s = double(block256(&unit[(6 * buf + k) * (n / 32) + 8 * l]));
      } else if (l < int(cl)) {
        s = part[buf][l][k];
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o, 16);
      return s;
    }
  };
  T xr[AFC_RPT][3];                        // this thread's rows of x
#pragma unroll
  for (int j = 0; j < AFC_RPT; ++j)
#pragma unroll
    for (int c = 0; c < 3; ++c) xr[j][c] = t + j * nt < rpc ? x[3 * (row0 + t + j * nt) + c] : T(0);
  // r of the first of this thread's rows of others; fetched while the scalars are formed
  T gh[4] = {T(0), T(0), T(0), T(0)};
  const bool ghosts = t < wn - rpc;
  if (ghosts) cluster_load4(ghost0, gh);
  bool live = true;
  while (live) {
    // p = z + beta p, z = D^-1 r.  Every CTA forms p of its whole window, the
    // others' rows from their r: the same values as their owners', without a
    // barrier in between.
    {
      const T b[3] = {sbe[0], sbe[1], sbe[2]};
      auto direct = [&](int j, const T (&v)[4]) {
#pragma unroll
        for (int c = 0; c < 3; ++c) pw[4 * j + c] = fma(b[c], pw[4 * j + c], mul_rn(v[c], v[3]));
      };
      for (int i = t; i < rpc; i += nt) {
        T v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = r[4 * i + c];
        direct(own0 - w0 + i, v);
      }
      for (int i = t; i < wn - rpc; i += nt) {
        const int j = wrow(i);
        if (i != t) cluster_load4(owner(w0 + j), gh);
        direct(j, gh);
      }
    }
    if (all_fast) {
      __syncthreads();
    } else {
      __syncwarp();
      cluster_barrier();
    }
    // q = S p
    if (wide) {
      const int i = t / AFL, l = t & (AFL - 1);
      if (i < rpc) {                       // whole warps
        T acc[3] = {T(0), T(0), T(0)};
        const int f1 = rp[i + 1];
#pragma unroll 4
        for (int f = rp[i] + l; f < f1; f += AFL) {
          T v[3];
          window_load3(pw + 4 * cc[f], v);
          const T a = cv[f];
#pragma unroll
          for (int c = 0; c < 3; ++c) acc[c] = fma(a, v[c], acc[c]);
        }
        const bool up = (l & 4) != 0;
        T s0 = (up ? acc[1] : acc[0]) + __shfl_xor_sync(0xffffffffu, up ? acc[0] : acc[1], 4);
        T s1 = acc[2] + __shfl_xor_sync(0xffffffffu, acc[2], 4);
#pragma unroll
        for (int o = 2; o > 0; o >>= 1) {
          s0 += __shfl_xor_sync(0xffffffffu, s0, o);
          s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        }
        if (l == 0) {
          q[3 * i] = s0;
          q[3 * i + 2] = s1;
        } else if (l == 4) {
          q[3 * i + 1] = s0;
        }
      }
    }
    const int lr = t & (lpr - 1);
    for (int i = wide ? rpc : t / lpr; i < rpc; i += nt / lpr) {
      T acc[2][3] = {{T(0), T(0), T(0)}, {T(0), T(0), T(0)}};
      auto add = [&](T (&s)[3], T a, const T (&v)[3]) {
#pragma unroll
        for (int c = 0; c < 3; ++c) s[c] = fma(a, v[c], s[c]);
      };
      const int f1 = rp[i + 1], fc = min(f1, cap);
      int f = rp[i] + lr, h = 0;
      if constexpr (sizeof(T) == 8) {
#pragma unroll 4
        for (; f < fc; f += lpr) {
          T v[3];
          window_load3(pw + 4 * cc[f], v);
          add(acc[0], cv[f], v);
        }
      } else {
        // a thread takes the entries of lanes lr and lr + 4 of the loop's eight
#pragma unroll 2
        for (; f + 4 < fc; f += AFL) {
          T v[3], u[3];
          window_load3(pw + 4 * cc[f], v);
          window_load3(pw + 4 * cc[f + 4], u);
          add(acc[0], cv[f], v);
          add(acc[1], cv[f + 4], u);
        }
      }
      for (; f < f1; f += lpr, h ^= 1) {   // the last one, and entries that did not fit
        T v[3], a;
        if (f < fc) {
          a = cv[f];
          window_load3(pw + 4 * cc[f], v);
        } else {
          const int k = int(ib.col[e0 + f] - R0);
          a = val[e0 + f];
          if (unsigned(k - w0) < unsigned(wn)) window_load3(pw + 4 * (k - w0), v);
          else column3(k, v);
        }
        if (h && sizeof(T) == 4) add(acc[1], a, v);
        else add(acc[0], a, v);
      }
      // the three sums over the row's lanes (whole warps get here together: a CTA's
      // rows are a multiple of 32), two of them in one butterfly step
      constexpr int hb = lpr / 2;
      const bool up = (lr & hb) != 0;
      T s0, s1;
      {
        const T a0 = sizeof(T) == 8 ? acc[0][0] : acc[0][0] + acc[1][0],
                a1 = sizeof(T) == 8 ? acc[0][1] : acc[0][1] + acc[1][1],
                a2 = sizeof(T) == 8 ? acc[0][2] : acc[0][2] + acc[1][2];
        s0 = (up ? a1 : a0) + __shfl_xor_sync(0xffffffffu, up ? a0 : a1, hb);
        s1 = a2 + __shfl_xor_sync(0xffffffffu, a2, hb);
        if constexpr (lpr == 4) {
          s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
          s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
        }
      }
      if (lr == 0) {
        q[3 * i] = s0;
        q[3 * i + 2] = s1;
      } else if (lr == hb) {
        q[3 * i + 1] = s0;
      }
    }
    __syncthreads();
    for (int i = t; i < rpc; i += nt) {
      T v[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) v[c] = mul_rn(p[4 * i + c], q[3 * i + c]);
      unit_sums(v, three{}, i / 32, 0);
    }
    exchange(three{}, 0);
    if (w < 3) {
      const double pq = total(three{}, 0, w);
      if (lane == 0) {
        KState& k = sk[w];
        if (!k.done) {
          k.pq = pq;
          T al = T(0);
          if (!(pq > 0.0) || !isfinite(pq)) {
            k.done = 1;
            k.status = 5;
          } else {
            al = T(k.rz / pq);
          }
          sal[w] = al;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < AFC_RPT; ++j) {
      const int i = t + j * nt;
      if (i >= rpc) break;                 // whole warps: a CTA's rows are a multiple of 32
      const T d = r[4 * i + 3];
      T v[6];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        v[2 * c] = v[2 * c + 1] = T(0);
        if (sk[c].done) continue;
        const T a = sal[c];
        xr[j][c] = fma(a, p[4 * i + c], xr[j][c]);
        const T rv = fma(-a, q[3 * i + c], r[4 * i + c]);
        r[4 * i + c] = rv;
        v[2 * c] = mul_rn(rv, mul_rn(rv, d));
        v[2 * c + 1] = mul_rn(rv, rv);
      }
      unit_sums(v, six{}, i / 32, 1);
    }
    exchange(six{}, 1);
    if (ghosts) cluster_load4(ghost0, gh);
    if (w < 3) {
      // r.z in the lower lanes, r.r in the upper ones
      const double sum = total(six{}, 1, 2 * w + (lane >> 4));
      const double rzn = sum, rr = __shfl_sync(0xffffffffu, sum, 16);
      KState& k = sk[w];
      if (lane == 0) {
        T be = T(0);
        if (!k.done) {
          k.iter++;
          k.rr = rr;
          if (!isfinite(rr)) { k.done = 1; k.status = 5; }
          else if (rr <= k.tt) k.done = 1;
          else if (k.iter >= k.max_iter) { k.done = 1; k.status = 4; }
          else {
            be = T(rzn / k.rz);
            k.rz = rzn;
          }
        }
        sbe[w] = be;
      }
    }
    __syncthreads();
    live = !(sk[0].done && sk[1].done && sk[2].done);
  }
  // no CTA leaves while another still reads its rows: the last fetch has arrived
  // (its values are used) before this CTA's arrival
  if (ghosts) pw[4 * wrow(t) + 3] = gh[0] + gh[1] + gh[2] + gh[3];
  __syncwarp();
  cluster_barrier();
#pragma unroll
  for (int j = 0; j < AFC_RPT; ++j)
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (t + j * nt < rpc) x[3 * (row0 + t + j * nt) + c] = xr[j][c];
  if (rank == 0 && t < 3) ks[3 * inst + t] = sk[t];
}

}  // namespace ibg

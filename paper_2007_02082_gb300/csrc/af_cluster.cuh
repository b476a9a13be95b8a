// Force solve of one problem by one thread-block cluster.
//
// The PCG on S (Eq. 21-22, three right-hand sides) is a chain of several
// hundred to a thousand short dependent steps when the wall points are as
// dense as the grid (Sec. 2.5), each over a few thousand rows: as kernel
// launches an iteration is two launches and two grid reductions, all latency
// (20-25 us whatever the size).  Here a cluster of up to 16 CTAs (co-scheduled
// by the hardware, so its barriers end) runs the whole loop of one problem: rows
// in equal contiguous ranges, the direction p in shared memory and gathered from
// the other CTAs' (distributed shared memory; the columns are kept as ready
// cluster addresses), as much of S as fits beside it, partial sums exchanged in
// shared memory, three hardware barriers an iteration, no host or launch in
// between.  A problem's arithmetic depends on its own rows only, so it
// keeps its bits alone and in any batch; problems of a batch run side by side.
// Bound: barrier and shared-memory latency (FP64: the FP64 rate of 16 SMs).
#pragma once

namespace ibg {

constexpr int AFC_THREADS = 1024;
constexpr int AFC_MAX = 16;                 // CTAs per cluster at most
constexpr int AFC_SMEM = 222 * 1024;        // dynamic shared memory asked for (with the static part below 227 KB)

__device__ __forceinline__ uint32_t cluster_addr(uint32_t smem, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem), "r"(rank));
  return a;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_load3(uint32_t a, float (&v)[3]) {
  float pad;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(pad) : "r"(a));
}
__device__ __forceinline__ void cluster_load3(uint32_t a, double (&v)[3]) {
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[2]) : "r"(a + 16));
}
__device__ __forceinline__ void cluster_store(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// bytes of shared memory per row: p (four values, 16-byte pieces), q, r, 1/diag
// and the row's first entry
template <typename T>
__host__ __device__ constexpr int afc_row_bytes() { return 11 * int(sizeof(T)) + 4; }
// rows of a CTA at most
template <typename T>
__host__ __device__ constexpr int afc_max_rows() { return (AFC_SMEM - 64) / afc_row_bytes<T>() / 16 * 16; }
// whether a problem of n (padded) rows runs in clusters of cl CTAs
template <typename T>
__host__ __device__ constexpr bool afc_fits(int64_t n, int cl) { return cl > 0 && n <= int64_t(cl) * afc_max_rows<T>(); }

template <typename T>
__global__ void __launch_bounds__(AFC_THREADS, 1)
    k_af_cluster(IBDev ib, const T* __restrict__ val, const T* __restrict__ dinv, T* __restrict__ x,
                 const T* __restrict__ r0, KState* __restrict__ ks) {
  KCOUNT();
  extern __shared__ __align__(16) unsigned char afc_sm[];
  __shared__ double part[2][AFC_MAX][6];   // partial sums of every CTA: p.q, then r.z and r.r
  __shared__ T red[32 * 6];
  __shared__ double tot[6];
  __shared__ T sal[3], sbe[3];
  __shared__ KState sk[3];
  uint32_t rank, cl;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(cl));
  const int inst = blockIdx.x / cl;
  const int64_t R0 = int64_t(ib.seg_t[inst]) * 256;
  const int n = (ib.seg_t[inst + 1] - ib.seg_t[inst]) * 256;   // whole blocks of 256 rows
  // uniform over the cluster: nothing to do, or too large for a cluster
  if (n == 0 || !afc_fits<T>(n, cl) || (ks[3 * inst].done && ks[3 * inst + 1].done && ks[3 * inst + 2].done)) return;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int rpc = n / int(cl);             // rows of this CTA
  const int64_t row0 = R0 + int64_t(rank) * rpc;
  T* p = reinterpret_cast<T*>(afc_sm);     // [rpc][4]
  T* q = p + 4 * rpc;                      // [rpc][3]
  T* r = q + 3 * rpc;                      // [rpc][3]
  T* di = r + 3 * rpc;                     // [rpc]
  T* cv = di + rpc;                        // cached values of S, then their columns' addresses
  const int e0 = ib.rowptr[row0], ne = ib.rowptr[row0 + rpc] - e0;
  const int cap = min(ne, int((AFC_SMEM - 64 - rpc * afc_row_bytes<T>()) / int(sizeof(T) + 4)));
  uint32_t* ca = reinterpret_cast<uint32_t*>(cv + cap);
  int* rp = reinterpret_cast<int*>(ca + cap);   // [rpc + 1] entries relative to e0
  const uint32_t pbase = smem_u32(p);
  auto column = [&](int e) -> uint32_t {   // cluster address of p at entry e's column
    const int k = int(ib.col[e] - R0), o = k / rpc;
    return cluster_addr(pbase + uint32_t(k - o * rpc) * uint32_t(4 * sizeof(T)), uint32_t(o));
  };
  for (int e = t; e < cap; e += AFC_THREADS) {
    cv[e] = val[e0 + e];
    ca[e] = column(e0 + e);
  }
  for (int i = t; i <= rpc; i += AFC_THREADS) rp[i] = ib.rowptr[row0 + i] - e0;
  for (int i = t; i < rpc; i += AFC_THREADS) {
    di[i] = dinv[row0 + i];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      r[3 * i + c] = r0[3 * (row0 + i) + c];
      p[4 * i + c] = T(0);
    }
    p[4 * i + 3] = T(0);
  }
  if (t < 3) {
    sk[t] = ks[3 * inst + t];
    sbe[t] = T(0);
  }
  __syncthreads();
  // warps that hold rows in the row-per-thread passes; lanes per row of the product
  const int nact = min(32, (rpc + 31) / 32);
  const int lpr = rpc <= 32 ? 32 : 8;
  // CTA totals of NV values (each thread's v) to every CTA of the cluster
  auto exchange = [&](auto& v, auto nv, int buf) {
    constexpr int NV = decltype(nv)::value;
    if (w < nact) warp_sums<T, NV>(v, red, w);
    __syncthreads();
    if (w < NV) {
      const T s = lane_sum(lane < nact ? red[w * 32 + lane] : T(0));
      if (lane == 0) tot[w] = double(s);
    }
    __syncthreads();
    if (t < int(cl) * NV) cluster_store(cluster_addr(smem_u32(&part[buf][rank][t % NV]), uint32_t(t / NV)), tot[t % NV]);
    __syncwarp();
    cluster_barrier();
  };
  bool live = true;
  while (live) {
    // p = z + beta p, z = D^-1 r
    {
      const T b[3] = {sbe[0], sbe[1], sbe[2]};
      for (int i = t; i < rpc; i += AFC_THREADS)
#pragma unroll
        for (int c = 0; c < 3; ++c) p[4 * i + c] = r[3 * i + c] * di[i] + b[c] * p[4 * i + c];
    }
    cluster_barrier();
    // q = S p
    const int lr = t & (lpr - 1);
    for (int i = t / lpr; i < rpc; i += AFC_THREADS / lpr) {
      T acc[3] = {T(0), T(0), T(0)};
      const int f1 = rp[i + 1];
#pragma unroll 2
      for (int f = rp[i] + lr; f < f1; f += lpr) {
        const T a = f < cap ? cv[f] : val[e0 + f];
        T v[3];
        cluster_load3(f < cap ? ca[f] : column(e0 + f), v);
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[c] += a * v[c];
      }
      // the three sums over the row's lanes (whole warps get here together: a CTA's
      // rows are a multiple of 16), two of them in one butterfly step
      const int h = lpr >> 1;
      const bool up = (lr & h) != 0;
      T s0 = (up ? acc[1] : acc[0]) + __shfl_xor_sync(0xffffffffu, up ? acc[0] : acc[1], h);
      T s1 = acc[2] + __shfl_xor_sync(0xffffffffu, acc[2], h);
      for (int o = h >> 1; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      }
      if (lr == 0) {
        q[3 * i] = s0;
        q[3 * i + 2] = s1;
      } else if (lr == h) {
        q[3 * i + 1] = s0;
      }
    }
    __syncthreads();
    {
      T v[3] = {T(0), T(0), T(0)};
      for (int i = t; i < rpc; i += AFC_THREADS)
#pragma unroll
        for (int c = 0; c < 3; ++c) v[c] += p[4 * i + c] * q[3 * i + c];
      exchange(v, std::integral_constant<int, 3>{}, 0);
    }
    if (w < 3) {
      const double pq = lane_sum(lane < int(cl) ? part[0][lane][w] : 0.0);
      if (lane == 0) {
        KState& k = sk[w];
        if (!k.done) {
          k.pq = pq;
          if (!(pq > 0.0) || !isfinite(pq)) {
            k.done = 1;
            k.status = 5;
            k.alpha = 0.0;
          } else {
            k.alpha = k.rz / pq;
          }
          k.af = float(k.alpha);
        }
        sal[w] = k_alpha<T>(k);
      }
    }
    __syncthreads();
    {
      T v[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
      for (int i = t; i < rpc; i += AFC_THREADS) {
        T* xi = x + 3 * (row0 + i);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          if (sk[c].done) continue;
          const T a = sal[c];
          xi[c] += a * p[4 * i + c];
          const T rv = r[3 * i + c] - a * q[3 * i + c];
          r[3 * i + c] = rv;
          v[2 * c] += rv * (rv * di[i]);
          v[2 * c + 1] += rv * rv;
        }
      }
      exchange(v, std::integral_constant<int, 6>{}, 1);
    }
    if (w < 3) {
      const double rzn = lane_sum(lane < int(cl) ? part[1][lane][2 * w] : 0.0);
      const double rr = lane_sum(lane < int(cl) ? part[1][lane][2 * w + 1] : 0.0);
      KState& k = sk[w];
      if (lane == 0 && !k.done) {
        k.iter++;
        k.rr = rr;
        if (!isfinite(rr)) { k.done = 1; k.status = 5; }
        else if (rr <= k.tol2 * k.bb) k.done = 1;
        else if (k.iter >= k.max_iter) { k.done = 1; k.status = 4; }
        else {
          k.beta = rzn / k.rz;
          k.bf = float(k.beta);
          k.rz = rzn;
        }
        sbe[w] = k.done ? T(0) : k_beta<T>(k);
      }
    }
    __syncthreads();
    live = !(sk[0].done && sk[1].done && sk[2].done);
  }
  if (rank == 0 && t < 3) ks[3 * inst + t] = sk[t];
}

}  // namespace ibg

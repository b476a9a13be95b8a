// Force solve of one problem by one thread-block cluster.
//
// The PCG on S (Eq. 21-22, three right-hand sides) is a chain of several
// hundred to a thousand short dependent steps when the wall points are as
// dense as the grid (Sec. 2.5), each over a few thousand rows: as kernel
// launches an iteration is two launches and two grid reductions, all latency
// (15-25 us whatever the size).  Here a cluster of up to 16 CTAs (co-scheduled
// by the hardware, so its barriers end) runs the whole loop of one problem: rows
// in equal contiguous ranges, p of the rows around a CTA's own copied once an
// iteration through distributed shared memory, S kept in shared memory as far
// as it fits (16-bit columns into that window), partial sums stored straight
// into every CTA, three hardware barriers an iteration (about 500 cycles each).
// A problem's arithmetic depends on its own rows only, so it keeps its bits
// alone and in any batch; problems of a batch run side by side.
// Bound: latency of the barriers and FP64 scalars at a few hundred rows (5 us an
// iteration), shared-memory wavefronts of the product at some thousand dense rows
// (8160 rows of 41 entries: 11 us), in FP64 the FP64 rate of 16 SMs (2000 rows: 13 us).
// A step: 8x8x16 tube 22.0 -> 6.5 ms, 16x16x64 tube in FP64 22.6 -> 15.3 ms, dense
// 32x32x128 tube 22.8 -> 12.0 ms (of which the reductions alone gave a third).
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
__device__ __forceinline__ void cluster_store(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// bytes of shared memory per row: p with 1/diag (four values), q, r and the row's first entry
template <typename T>
__host__ __device__ constexpr int afc_row_bytes() { return 10 * int(sizeof(T)) + 4; }
// Padded rows of a problem that runs in clusters of cl CTAs.  FP32: while its
// rows take half of the shared memory (at 32,000 rows of 10 entries 14 us an
// iteration, as the loop; the rest of the range still saves the launches).
// FP64: while the FP64 rate of 16 SMs costs less than the loop's launches
// (2000 rows of 40 entries 13 us against 25; 32,000 rows of 10 measured 80 against 50).
template <typename T>
__host__ __device__ constexpr int64_t afc_max_rows(int cl) { return int64_t(cl) * (sizeof(T) == 4 ? 2560 : 384); }
template <typename T>
__host__ __device__ constexpr bool afc_fits(int64_t n, int cl) { return cl > 0 && n <= afc_max_rows<T>(cl); }

template <typename T>
__global__ void __launch_bounds__(AFC_THREADS, 1)
    k_af_cluster(IBDev ib, const T* __restrict__ val, const T* __restrict__ dinv, T* __restrict__ x,
                 const T* __restrict__ r0, KState* __restrict__ ks) {
  KCOUNT();
  extern __shared__ __align__(16) unsigned char afc_sm[];
  __shared__ double part[2][AFC_MAX][6];   // partial sums of every CTA: p.q, then r.z and r.r
  __shared__ T red[32 * 6];
  __shared__ T sal[3], sbe[3];
  __shared__ KState sk[3];
  __shared__ int win, goff[AFC_MAX];
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
  const int e0 = ib.rowptr[row0], ne = ib.rowptr[row0 + rpc] - e0;
  // lanes per row of the product: four where rows are short (all of the
  // problem decides, so that its CTAs agree), eight otherwise
  const int lpr = ib.rowptr[R0 + n] - ib.rowptr[R0] < 20 * n || sizeof(T) == 8 ? 4 : 8;
  // no more warps than the rows need: the others leave (the barriers count
  // the threads that are left)
  const int nt = min(AFC_THREADS, max(256, lpr * rpc));
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
  const int own0 = int(rank) * rpc;        // the problem's row of the CTA's first one
  const int room = AFC_SMEM - 64 - rpc * afc_row_bytes<T>();
  const bool fast = win <= room / int(16 * sizeof(T));   // the window takes half the room at most
  const int G = fast ? win : 0;
  const int w0 = max(0, own0 - G), wn = min(n, own0 + rpc + G) - w0;   // window: rows [w0, w0 + wn) of the problem
  T* pw = reinterpret_cast<T*>(afc_sm);    // [wn][4]: p; the own rows' fourth value is 1/diag
  T* p = pw + 4 * (own0 - w0);
  T* q = pw + 4 * wn;                      // [rpc][3]
  T* r = q + 3 * rpc;                      // [rpc][3]
  T* cv = r + 3 * rpc;                     // cached values of S ...
  const int cap = fast ? min(ne, (room - (wn - rpc) * int(4 * sizeof(T))) / int(sizeof(T) + 2)) / 2 * 2 : 0;
  uint16_t* cc = reinterpret_cast<uint16_t*>(cv + cap);   // ... and their columns' places in the window
  int* rp = reinterpret_cast<int*>(cc + cap);             // [rpc + 1] entries relative to e0
  // where every CTA's own rows start in its window (once every CTA runs)
  cluster_barrier();
  if (t < int(cl)) cluster_store(cluster_addr(smem_u32(&goff[rank]), uint32_t(t)), own0 - w0);
  const uint32_t pbase = smem_u32(pw);
  auto owner = [&](int k) -> uint32_t {    // cluster address of p at row k of the problem
    const int o = k / rpc;
    return cluster_addr(pbase + uint32_t(goff[o] + k - o * rpc) * uint32_t(4 * sizeof(T)), uint32_t(o));
  };
  for (int e = t; e < cap; e += nt) {
    cv[e] = val[e0 + e];
    cc[e] = uint16_t(ib.col[e0 + e] - R0 - w0);
  }
  for (int i = t; i <= rpc; i += nt) rp[i] = ib.rowptr[row0 + i] - e0;
  for (int i = t; i < rpc; i += nt) {
    p[4 * i + 3] = dinv[row0 + i];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      r[3 * i + c] = r0[3 * (row0 + i) + c];
      p[4 * i + c] = T(0);
    }
  }
  if (t < 3) {
    sk[t] = ks[3 * inst + t];
    sbe[t] = T(0);
  }
  __syncwarp();
  cluster_barrier();
  const int nact = min(nt / 32, (rpc + 31) / 32);   // warps that hold rows in the row-per-thread passes
  auto wrow = [&](int i) { return i < own0 - w0 ? i : i + rpc; };   // window row of the i-th row of others
  const uint32_t ghost0 = t < wn - rpc ? owner(w0 + wrow(t)) : 0u;
  // CTA totals of NV values (each thread's v) to every CTA of the cluster
  auto exchange = [&](auto& v, auto nv, int buf) {
    constexpr int NV = decltype(nv)::value;
    if (w < nact) warp_sums<T, NV>(v, red, w);
    __syncthreads();
    if (w < NV) {
      const double s = double(__shfl_sync(0xffffffffu, lane_sum(lane < nact ? red[w * 32 + lane] : T(0)), 0));
      if (lane < int(cl)) cluster_store(cluster_addr(smem_u32(&part[buf][rank][w]), uint32_t(lane)), s);
      __syncwarp();
    }
    cluster_barrier();
  };
  bool live = true;
  while (live) {
    // p = z + beta p, z = D^-1 r
    {
      const T b[3] = {sbe[0], sbe[1], sbe[2]};
      for (int i = t; i < rpc; i += nt) {
        const T d = p[4 * i + 3];
#pragma unroll
        for (int c = 0; c < 3; ++c) p[4 * i + c] = r[3 * i + c] * d + b[c] * p[4 * i + c];
      }
    }
    __syncwarp();
    cluster_barrier();
    // the others' rows of the window
    for (int i = t; i < wn - rpc; i += nt) {
      const int j = wrow(i);
      T v[3];
      cluster_load3(i == t ? ghost0 : owner(w0 + j), v);
#pragma unroll
      for (int c = 0; c < 3; ++c) pw[4 * j + c] = v[c];
    }
    __syncthreads();
    // q = S p
    const int lr = t & (lpr - 1);
    for (int i = t / lpr; i < rpc; i += nt / lpr) {
      T acc[3] = {T(0), T(0), T(0)};
      auto add = [&](T a, const T (&v)[3]) {
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[c] += a * v[c];
      };
      const int f1 = rp[i + 1], fc = min(f1, cap);
      int f = rp[i] + lr;
#pragma unroll 4
      for (; f < fc; f += lpr) {
        T v[3];
        window_load3(pw + 4 * cc[f], v);
        add(cv[f], v);
      }
      for (; f < f1; f += lpr) {   // entries that did not fit
        const int k = int(ib.col[e0 + f] - R0);
        T v[3];
        if (fast) window_load3(pw + 4 * (k - w0), v);
        else cluster_load3(owner(k), v);
        add(val[e0 + f], v);
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
      for (int i = t; i < rpc; i += nt)
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
      for (int i = t; i < rpc; i += nt) {
        T* xi = x + 3 * (row0 + i);
        const T d = p[4 * i + 3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          if (sk[c].done) continue;
          const T a = sal[c];
          atomicAdd(xi + c, a * p[4 * i + c]);   // this thread's own element: no load to wait for
          const T rv = r[3 * i + c] - a * q[3 * i + c];
          r[3 * i + c] = rv;
          v[2 * c] += rv * (rv * d);
          v[2 * c + 1] += rv * rv;
        }
      }
      exchange(v, std::integral_constant<int, 6>{}, 1);
    }
    if (w < 3) {
      const double rzn = lane_sum(lane < int(cl) ? part[1][lane][2 * w] : 0.0);
      const double rr = lane_sum(lane < int(cl) ? part[1][lane][2 * w + 1] : 0.0);
      KState& k = sk[w];
      if (lane == 0) {
        if (!k.done) {
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

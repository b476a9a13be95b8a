// Test driver for the force solve (csrc/ib.cu) on systems given in a file: the
// library's own routines, linked from libibgpu.so, with the cluster solve or the
// loop of launches chosen from outside, which no entry point of the library offers.
//
//   force_probe IN OUT
//
// IN: int64 ninst, mixed, cluster (CTAs; 0: the loop for every problem, -1: the library's choice),
// max_iter, max_outer, reps; double rtol, rtol_inner; int64 rows of every problem
// (padded, multiples of 256); int32 rowptr, col (global rows); double val, dinv,
// b, g (3 a row, g the start).  OUT: per problem int32 iterations[3], status,
// outer; then g as double; then the seconds of each repetition.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "ib.hpp"
#include "krylov.hpp"

using namespace ibg;

#define CK(x)                                                                     \
  do {                                                                            \
    cudaError_t e_ = (x);                                                         \
    if (e_ != cudaSuccess) {                                                      \
      std::fprintf(stderr, "%s: %s\n", #x, cudaGetErrorString(e_));               \
      return 1;                                                                   \
    }                                                                             \
  } while (0)

template <typename T>
static std::vector<T> take(FILE* f, size_t n) {
  std::vector<T> v(n);
  if (std::fread(v.data(), sizeof(T), n, f) != n) {
    std::fprintf(stderr, "short input\n");
    std::exit(2);
  }
  return v;
}

template <typename T>
static T* put(const std::vector<T>& v) {
  T* p = nullptr;
  if (cudaMalloc(&p, std::max<size_t>(v.size(), 1) * sizeof(T)) != cudaSuccess ||
      cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess) {
    std::fprintf(stderr, "upload failed\n");
    std::exit(2);
  }
  return p;
}

int main(int argc, char** argv) {
  FILE* f = argc == 3 ? std::fopen(argv[1], "rb") : nullptr;
  if (!f) return 2;
  const auto head = take<int64_t>(f, 6);
  const auto tol = take<double>(f, 2);
  const int n = int(head[0]), max_iter = int(head[3]), max_outer = int(head[4]), reps = int(head[5]);
  const bool mixed = head[1] != 0;
  const auto rows = take<int64_t>(f, n);
  int64_t M = 0;
  std::vector<int32_t> st(1, 0), sg(1, 0), pinst;
  for (int i = 0; i < n; ++i) {
    M += rows[i];
    st.push_back(int32_t(M / 256));
    sg.push_back(int32_t(M / 32));
    pinst.resize(M, i);
  }
  const auto rowptr = take<int32_t>(f, M + 1);
  const auto col = take<int32_t>(f, rowptr[M]);
  const auto val = take<double>(f, rowptr[M]);
  const auto dinv = take<double>(f, M);
  const auto b = take<double>(f, 3 * M);
  auto g = take<double>(f, 3 * M);
  std::fclose(f);

  IBDev ib{};
  ib.M = M;
  ib.ninst = n;
  ib.pinst = put(pinst);
  ib.seg_t = put(st);
  ib.seg_g = put(sg);
  ib.rowptr = put(rowptr);
  ib.col = put(col);
  ib.val = put(val);
  ib.dinv = put(dinv);
  ib.val32 = put(std::vector<float>(val.begin(), val.end()));
  ib.dinv32 = put(std::vector<float>(dinv.begin(), dinv.end()));
  std::vector<uint8_t> route(n);
  ib_choose_solver(ib, st.data(), rowptr.data(), col.data(), mixed, route.data());
  if (head[2] >= 0) {
    ib.af_cl32 = ib.af_cl64 = int32_t(head[2]);
    ib.af_big32 = ib.af_big64 = head[2] == 0;
    ib.af_small32 = ib.af_small64 = head[2] != 0;
    for (uint8_t& v : route) v = head[2] ? AF_CLUSTER32 | AF_CLUSTER64 : 0;
  }
  ib.af_route = put(route);
  RedBuf rb;
  rb.partials = put(std::vector<double>(2 * (M / 32 + 1) * 16 + n * 16 + 64));
  rb.counter = put(std::vector<unsigned>(M / 32 + 2));
  KState* ks = put(std::vector<KState>(3 * n));
  OState* os = put(std::vector<OState>(n));
  SolveRec* rec = put(std::vector<SolveRec>(4 * n));
  double *db = put(b), *dg = put(g), *y64 = put(std::vector<double>(3 * M)), *work = put(std::vector<double>(15 * M));
  float* w32 = put(std::vector<float>(21 * M));
  KState* ksh;
  OState* osh;
  CK(cudaMallocHost(&ksh, 3 * n * sizeof(KState)));
  CK(cudaMallocHost(&osh, n * sizeof(OState)));
  cudaStream_t s;
  CK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  CaptureCtx cc;
  for (int k = 0; k < 4; ++k) {
    cudaStream_t side;
    CK(cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking));
    cc.side.push_back(side);
  }
  // the step's form: captured once, launched as a graph
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  cc.capturing = true;
  const cudaError_t e =
      mixed ? ib_solve_mixed(ib, db, dg, y64, w32, ks, ksh, os, osh, rb, tol[0], tol[1], max_iter, max_outer, rec, s, &cc)
            : ib_solve(ib, db, dg, work, ks, ksh, rb, tol[0], max_iter, rec, s, &cc);
  CK(cudaStreamEndCapture(s, &graph));
  CK(e);
  CK(cudaGraphInstantiate(&exec, graph, 0));
  cudaEvent_t t0, t1;
  CK(cudaEventCreate(&t0));
  CK(cudaEventCreate(&t1));
  std::vector<double> sec;
  for (int k = 0; k < reps; ++k) {
    CK(cudaMemcpyAsync(dg, g.data(), 3 * M * sizeof(double), cudaMemcpyHostToDevice, s));
    CK(cudaMemsetAsync(rec, 0, 4 * n * sizeof(SolveRec), s));
    CK(cudaEventRecord(t0, s));
    CK(cudaGraphLaunch(exec, s));
    CK(cudaEventRecord(t1, s));
    CK(cudaStreamSynchronize(s));
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, t0, t1));
    sec.push_back(1e-3 * ms);
  }
  CK(cudaGetLastError());
  std::vector<SolveRec> r(4 * n);
  CK(cudaMemcpy(r.data(), rec, r.size() * sizeof(SolveRec), cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(g.data(), dg, 3 * M * sizeof(double), cudaMemcpyDeviceToHost));
  f = std::fopen(argv[2], "wb");
  if (!f) return 2;
  for (int i = 0; i < n; ++i) {
    const int32_t v[5] = {r[4 * i].iters[0], r[4 * i].iters[1], r[4 * i].iters[2], r[4 * i].status, r[4 * i].outer};
    std::fwrite(v, sizeof(v), 1, f);
  }
  std::fwrite(g.data(), sizeof(double), g.size(), f);
  std::fwrite(sec.data(), sizeof(double), sec.size(), f);
  return std::fclose(f) == 0 ? 0 : 2;
}

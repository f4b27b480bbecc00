// Runs the values' own row program (k2_fine_row) on the host, and sincos2 over
// a list of angles.  Input (stdin): n P rows groups terms gates threads, gates
// and terms and parameters as run.cpp reads them; or, with n = 0, a count and
// that many angles.  Shared memory is followed by a guard.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <thread>

#include "cuda_runtime.h"
namespace tdq {
alignas(16) unsigned char raw[16], smem_raw[(227 << 10) + 4096];
}
#include "k2_body.cuh"
#include "lin_program.cu"

using namespace tdq;

template <class T>
static T get() {
  double v;
  if (scanf("%lf", &v) != 1) exit(2);
  return (T)v;
}

int main() {
  const int n = get<int>();
  if (n == 0) {
    for (int i = get<int>(); i > 0; i--) {
      const SinCos r = sincos2(get<float>());
      printf("%.17g %.17g\n", (double)r.s + r.sl, (double)r.c + r.cl);
    }
    return 0;
  }
  const int P = get<int>(), rows = get<int>(), ng = get<int>(), nt = get<int>(), G = get<int>(), threads = get<int>();
  std::vector<SweepOp> ops(G);
  for (SweepOp& o : ops) {
    o.kind = get<int8_t>(); o.p0 = get<int8_t>(); o.p1 = get<int8_t>(); o.nang = get<int8_t>();
    for (int j = 0; j < 3; j++) o.src[j] = get<int>();
    for (int j = 0; j < 3; j++) o.slot[j] = -1, o.fixed[j] = 0.f;
  }
  std::vector<TermDev> terms(nt);
  std::vector<int> gptr(ng + 1, 0);
  for (TermDev& t : terms) {
    t.pmask_lo = get<uint32_t>(); t.pmask_hi = 0; t.coeff = get<float>(); t.group = get<int>();
    for (int g = t.group + 1; g <= ng; g++) gptr[g]++;
  }
  std::vector<float> params((size_t)rows * P);
  for (float& p : params) p = get<float>();
  const LinProgram prog = lin_program(ops, n, n, 0, 2, 2, false, false);
  for (TermDev& t : terms) {
    uint32_t m = 0;
    for (int q = 0; q < n; q++)
      if ((t.pmask_lo >> q) & 1u) m ^= prog.map.row[q];
    if (parity32(t.pmask_lo & prog.map.b)) t.coeff = -t.coeff;
    t.pmask_lo = m;
  }
  std::vector<FineOp> fine;
  for (const LinOp& g : prog.ops)
    fine.push_back({g.kind, g.m, g.f, g.f2, g.b | (g.b2 << 1), g.op >= 0 ? ops[g.op].src[g.ang] : 0, 0.f, 0});
  const size_t dim = (size_t)1 << n;
  std::vector<float> odiag((size_t)ng * dim);
  for (int g = 0; g < ng; g++)
    for (size_t y = 0; y < dim; y++)
      odiag[g * dim + y] = diag_weight(terms.data(), gptr[g], gptr[g + 1], (uint32_t)y);
  std::vector<double> values((size_t)rows * ng, -7.0);
  int status = 0;
  SweepArgs a{};
  a.n = n; a.params = params.data(); a.pstride = P; a.n_groups = ng; a.odiag = odiag.data(); a.values = values.data();
  a.status = &status; a.ps_copies = 1; a.fine = fine.data(); a.nfine = (int)fine.size(); a.fine_rows = rows;
  const size_t bytes = k2_fine_bytes(n);
  for (int b = 0; b < rows; b++) {
    memset(smem_raw, 0xff, bytes);
    memset(smem_raw + bytes, 0x5a, 4096);
    Cta c(threads);
    std::vector<std::thread> pool;
    for (int t = 0; t < threads; t++)
      pool.emplace_back([&, t] {
        cta = &c;
        threadIdx.x = t;
        blockIdx.x = b;
        blockDim.x = threads;
        k2_fine_row(a, b);
      });
    for (auto& t : pool) t.join();
    for (int i = 0; i < 4096; i++)
      if (smem_raw[bytes + i] != 0x5a) { fprintf(stderr, "write past shared memory (byte %d)\n", i); return 1; }
  }
  printf("status %d\n", status);
  for (double v : values) printf("%.17g ", v);
  printf("\n");
  return 0;
}

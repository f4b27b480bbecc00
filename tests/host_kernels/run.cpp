// Runs a generated sweep program (GENERATED: the text of tdq_sweep_source) on
// the host, as the library launches it, and writes its values and gradients
// (or final state) to stdout.  Input (stdin, whitespace separated):
//   n tile(0: whole state) fwd_bits rev_bits adjoint P rows groups terms gates
//   gates x (kind p0 p1 nang src0 src1 src2 slot0 slot1 slot2)
//   terms x (mask coeff group), sorted by group;  rows x P parameters
// Shared memory is followed by a guard that must stay untouched.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <thread>

#include "cuda_runtime.h"
namespace tdq {
alignas(16) unsigned char raw[(227 << 10) + 4096], smem_raw[(227 << 10) + 4096];
}
#include GENERATED
#include "lin_program.cu"

using namespace tdq;

template <class K>
static void launch(unsigned grid, unsigned threads, unsigned char* smem, size_t bytes, K kernel) {
  if (bytes > (227u << 10)) { fprintf(stderr, "shared memory %zu\n", bytes); exit(1); }
  for (unsigned b = 0; b < grid; b++) {
    memset(smem, 0xff, bytes);  // (NaNs)
    memset(smem + bytes, 0x5a, 4096);
    Cta c(threads);
    std::vector<std::thread> pool;
    for (unsigned t = 0; t < threads; t++)
      pool.emplace_back([&, t] {
        cta = &c;
        threadIdx.x = t;
        blockIdx.x = b;
        blockDim.x = threads;
        gridDim.x = grid;
        kernel();
      });
    for (auto& t : pool) t.join();
    for (int i = 0; i < 4096; i++)
      if (smem[bytes + i] != 0x5a) { fprintf(stderr, "write past shared memory (byte %d)\n", i); exit(1); }
  }
}

template <class T>
static T get() {
  double v;
  if (scanf("%lf", &v) != 1) exit(2);
  return (T)v;
}

#define CAT2(a, b) a##b
#define CAT(a, b) CAT2(a, b)

int main() {
  const int n = get<int>(), tile = get<int>(), fb = get<int>(), rb = get<int>(), adj = get<int>(), P = get<int>(),
            rows = get<int>(), ng = get<int>(), nt = get<int>(), G = get<int>();
  std::vector<SweepOp> ops(G);
  for (SweepOp& o : ops) {
    o.kind = get<int8_t>(); o.p0 = get<int8_t>(); o.p1 = get<int8_t>(); o.nang = get<int8_t>();
    for (int j = 0; j < 3; j++) o.src[j] = get<int>();
    for (int j = 0; j < 3; j++) o.slot[j] = get<int>();
    for (int j = 0; j < 3; j++) o.fixed[j] = 0.f;
  }
  std::vector<TermDev> terms(nt);
  std::vector<int> gptr(ng + 1, 0);
  for (TermDev& t : terms) {
    t.pmask_lo = get<uint32_t>(); t.pmask_hi = 0; t.coeff = get<float>(); t.group = get<int>();
    for (int g = t.group + 1; g <= ng; g++) gptr[g]++;
  }
  std::vector<float> params((size_t)rows * P);
  for (float& p : params) p = get<float>();
  const int k = tile ? std::min(n, tile) : n;
  int L = 0;
  LinProgram prog = tile ? lin_tiled_program(ops, n, k, fb, rb, adj, ng == 0, &L)
                         : lin_program(ops, n, n, 0, fb, rb, adj, ng == 0);
  for (TermDev& t : terms) {
    uint32_t m = 0;
    for (int q = 0; q < n; q++)
      if ((t.pmask_lo >> q) & 1u) m ^= prog.map.row[q];
    if (parity32(t.pmask_lo & prog.map.b)) t.coeff = -t.coeff;
    t.pmask_lo = m;
  }
  const size_t dim = (size_t)1 << n;
  std::vector<uint32_t> lin = prog.map.col;
  lin.push_back(prog.map.to_y(0));
  std::vector<double> values((size_t)rows * (ng ? ng : 2 * dim), -7.0), gw;
  std::vector<float> grads((size_t)rows * std::max(P, 1), -7.f);
  int status = 0;
  SweepArgs a{};
  a.ops = ops.data(); a.G = G; a.n = n; a.params = params.data(); a.pstride = P;
  a.terms = terms.data(); a.group_ptr = gptr.data(); a.T = nt; a.n_groups = ng;
  a.output = ng ? TDQ_OUT_EXPVAL : TDQ_OUT_STATE;
  a.values = values.data(); a.grads = grads.data(); a.P = P; a.status = &status; a.ps_copies = 1;
  std::vector<float> odiag((size_t)ng * dim);
  for (int g = 0; g < ng; g++)
    for (size_t y = 0; y < dim; y++)
      odiag[g * dim + y] = diag_weight(terms.data(), gptr[g], gptr[g + 1], (uint32_t)y);
  a.odiag = odiag.data();
  a.rot = prog.rot.data(); a.rot_x = prog.rot_x.data(); a.nrot = (int)prog.rot.size();
  a.lin = lin.data(); a.quarter = ng ? 0 : prog.map.quarter;
#ifdef WHOLE
  const LinTile& t = prog.tiles[0];
  const int nrec = (int)t.coef.size(), threads = std::max(32, std::min(256, (1 << n) >> std::min(fb, n)));
  const size_t gb = adj ? k2_grad_bytes(true, P, threads) : 0;
  const size_t sb = dim * sizeof(c2) * (adj ? 2 : 1) + coef_bytes(nrec, a.nrot) + ((gb + 7) & ~(size_t)7) + 32 * sizeof(double) + 16;
  a.rot_flips = t.flips.data(); a.coef = t.coef.data(); a.norm = t.norm.data();
  launch(rows, threads, smem_raw, sb,
         [&] { tdq_k2_specialised(a, nullptr, 0, nullptr, nullptr, nrec); });
#else
  const int np = (int)prog.tiles.size(), nthr = std::max(32, std::min(256, 1 << (k - std::min(fb, k)))),
            nthr_r = std::max(32, std::min(256, 1 << (k - std::min(rb, k))));
  std::vector<c2> psi(dim * rows, c2{NAN, NAN}), lam(dim * rows, c2{NAN, NAN});
  std::vector<double> gacc((size_t)rows * std::max(P, 1), 0.0), vals((size_t)rows * std::max(ng, 1), 0.0);
  TiledDev d{};
  d.ops = ops.data(); d.psi = psi.data(); d.lam = lam.data(); d.gacc = gacc.data(); d.vals = vals.data();
  d.n = n; d.k = k; d.L = L; d.nrows = rows;
  using K1F = void (*)(SweepArgs, TiledDev, int);
  using K1R = void (*)(SweepArgs, TiledDev);
  const K1F kf[] = {FWD_KERNELS};
  const K1R kr[] = {REV_KERNELS};
  int max_rec = 0, gmax = 0;
  std::vector<int> nacc(np, 0);
  for (int p = 0; p < np; p++) {
    max_rec = std::max(max_rec, (int)prog.tiles[p].coef.size());
    for (int o : prog.tiles[p].ops) nacc[p] += adj && prog.ops[o].slot >= 0;
    gmax = std::max(gmax, 4 * (std::max(nthr, nthr_r) / 32) * std::max(1, nacc[p]));
  }
  auto run = [&](int p, bool rev) {
    const LinTile& t = prog.tiles[p];
    d.ntiles = p == 0 && (np > 1 || ng) ? 1 : 1 << (n - k);
    std::vector<int> off;
    for (int j = 0; j < (1 << (k - L)); j++) {
      uint32_t o = 0;
      for (int i = 0; i < k - L; i++)
        if ((j >> i) & 1) o ^= t.v[L + i];
      off.push_back((int)o);
    }
    std::vector<int8_t> loc8(32, -1);
    d.off = off.data(); d.loc = loc8.data(); d.smask = t.pivots;
    d.rec0 = 0; d.nrec = (int)t.coef.size();
    d.gbytes = 4 * (std::max(nthr, nthr_r) / 32) * std::max(1, nacc[p]);
    a.rot_flips = t.flips.data(); a.coef = t.coef.data(); a.norm = t.norm.data();
    const int units = rows * d.ntiles, ctas = std::min(units, 3);  // uneven shares, rows cut across CTAs
    d.tiles_per_cta = (units + ctas - 1) / ctas;
    const unsigned grid = (units + d.tiles_per_cta - 1) / d.tiles_per_cta;
    d.dbl = 1;
    const bool last = p == np - 1;
    const size_t sm = rev ? k1_smem_bytes(k, L, 1, 1, coef_bytes(max_rec, a.nrot), 0, ng, gmax)
                          : k1_smem_bytes(k, L, p == 0 ? 1 : 2, adj && last ? 1 : 0, coef_bytes(max_rec, a.nrot), 0, ng, gmax);
    if (rev) launch(grid, nthr_r, raw, sm, [&] { kr[p](a, d); });
    else launch(grid, nthr, raw, sm, [&] { kf[p](a, d, last && !adj ? ng == 0 : 1); });
  };
  for (int p = 0; p < np; p++) run(p, false);
  if (adj)
    for (int p = np - 2; p >= 0; p--) run(p, true);
  for (size_t i = 0; i < vals.size() && ng; i++) values[i] = vals[i];
  for (size_t i = 0; i < grads.size(); i++) grads[i] = (float)gacc[i];
  if (!ng)
    for (int r = 0; r < rows; r++)
      for (uint32_t x = 0; x < dim; x++) {
        const c2 v = psi[r * dim + lin_index(a, x)];
        values[(r * dim + x) * 2] = v.x;
        values[(r * dim + x) * 2 + 1] = v.y;
      }
#endif
  printf("status %d\n", status);
  for (double v : values) printf("%.9g ", v);
  printf("\n");
  if (adj)
    for (float g : grads) printf("%.9g ", g);
  printf("\n");
  return 0;
}

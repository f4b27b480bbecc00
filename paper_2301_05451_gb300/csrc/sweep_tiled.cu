// Kernel K1: tiled state sweep through HBM (see sweep_tiled.cuh).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <string>
#include <thread>
#include <utility>
#include <vector>

#include "k1_body.cuh"
#include "sweep_jit.h"
#include "sweep_tiled.cuh"

namespace tdq {

namespace {

template <bool FIRST, bool LAST, bool GRAD>
__global__ void __launch_bounds__(256) k1_forward(SweepArgs a, TiledDev t, int store) {
  k1_forward_body<256, FIRST, LAST, GRAD, InterpTile>(a, t, store);
}

__global__ void __launch_bounds__(256) k1_reverse(SweepArgs a, TiledDev t) { k1_reverse_body<256, InterpTile>(a, t); }

// Copy out the chunk's values, F for the shift rule, gradients, amplitudes.
__global__ void k1_finalize(SweepArgs a, TiledDev t, int nrows, int grad_adj) {
  chain_wait();
  const int lr = blockIdx.x;
  if (lr >= nrows) return;
  const int row = t.row0 + lr;
  const int64_t b = row / a.ps_copies;
  const int kk = row % a.ps_copies;
  if (a.output == TDQ_OUT_EXPVAL) {
    if (threadIdx.x == 0) {
      double F = 0.0;
      for (int g = 0; g < a.n_groups; g++) {
        const double v = t.vals[(int64_t)lr * a.n_groups + g];
        F += (a.gw ? a.gw[b * a.n_groups + g] : 1.0) * v;
        if (kk == 0) a.values[b * a.n_groups + g] = v;
      }
      if (a.ps_copies > 1) a.ps_F[row] = F;
    }
  } else if (kk == 0 && a.output == TDQ_OUT_AMPLITUDE) {
    const c2* psi = t.psi + (size_t)lr * (1u << t.n);
    for (int i = threadIdx.x; i < a.A; i += blockDim.x) {
      const c2 v = psi[a.amp_idx[i]];
      a.values[(b * a.A + i) * 2] = v.x;
      a.values[(b * a.A + i) * 2 + 1] = v.y;
    }
  }
  if (grad_adj)
    for (int j = threadIdx.x; j < a.P; j += blockDim.x) a.grads[b * a.P + j] = (float)t.gacc[(int64_t)lr * a.P + j];
}

// (double)f and (double)f * f without the FP64 pipe, which runs at less than a
// 64th of the FP32 rate and is what a read-out of states waits for (four FP64
// instructions per probability: 160 us for 2^24 of them).  Exact; only
// subnormal and non-finite floats take the conversion.
__device__ __forceinline__ double exact_double(float f) {
  const uint32_t u = __float_as_uint(f), e = (u >> 23) & 255u;
  if ((e == 0u && (u << 1)) || e == 255u) return (double)f;
  const uint32_t hi = (u & 0x80000000u) | (e ? ((u & 0x7fffffffu) >> 3) + (896u << 20) : 0u);
  return __hiloint2double((int)hi, (int)(u << 29));
}
__device__ __forceinline__ double exact_square(float f) {
  const uint32_t u = __float_as_uint(f), e = (u >> 23) & 255u;
  if (e - 1u >= 254u) return (u << 1) ? (double)f * (double)f : 0.0;
  // (2^7 m)^2 with the 24-bit m: in [2^60, 2^62); normalised to bit 62
  const uint32_t m = ((u & 0x7fffffu) | 0x800000u) << 7;
  const uint32_t ph = __umulhi(m, m), pl = m * m, top = ph >> 29;  // (bit 61)
  const uint32_t h = top ? ph : __funnelshift_l(pl, ph, 1), l = top ? pl : pl << 1;
  // mantissa bits 61..9 of (h, l); 2 e - 254 + 1023 - 1 (the leading one adds 1), + 1 for the top half
  return __hiloint2double((int)(((2u * e + 768u + top) << 20) + (h >> 9)), (int)__funnelshift_r(l, h, 9));
}

// The chunk's final states as the output: the whole state (TDQ_OUT_STATE) or
// the probabilities (TDQ_OUT_PROBS) of every row.  Basis index x sits at place
// y(x), a linear map: element by element one of the two sides would be
// scattered, 32 bytes moved for 8 used.  A block moves one coset at a time of
// a space that holds both 2^5 consecutive x and the x of 2^5 consecutive y
// (OutMap): read in runs of y, turned in shared memory, written in runs of x.
// The maps are linear: a thread's elements tid + 256 i differ by constants.
// 20 qubits, 16 rows, 128 MiB read, 128 MiB of probabilities written:
// 77 us, 160 element by element with FP64 conversions.
constexpr int kOutPer = (1 << kOutBits) / 256;  // elements per thread
__global__ void __launch_bounds__(256) k1_state_out(SweepArgs a, TiledDev t, int nrows, const OutMap* __restrict__ m) {
  __shared__ c2 buf[1 << kOutBits];
  __shared__ uint32_t at_yx[2];  // this tile's first y and x
  const int size = 1 << m->bits, tid = threadIdx.x;
  const bool on = tid < size;
  const uint32_t ox = m->x[tid], oy = m->y[tid], at = m->at[tid];
  uint32_t cx[kOutPer], cy[kOutPer], ca[kOutPer];
#pragma unroll
  for (int i = 0; i < kOutPer; i++) {
    cx[i] = m->x[256 * i];
    cy[i] = m->y[256 * i];
    ca[i] = swz(m->at[256 * i]);
  }
  const int per = max(1, size / 256);
  const int64_t dim = (int64_t)1 << t.n, per_row = dim >> m->bits, tot = per_row * nrows;
  const uint32_t other = (uint32_t)(dim - 1) & ~m->pivots;
  for (int64_t tile = blockIdx.x; tile < tot; tile += gridDim.x) {
    const int lr = (int)(tile / per_row);
    const int row = t.row0 + lr;
    const int64_t b = row / a.ps_copies;
    if (row % a.ps_copies) continue;
    if (tid < 32) {  // y of the tile's first x: a bit of x per lane
      const uint32_t x0 = deposit((uint32_t)(tile - (int64_t)lr * per_row), other);
      uint32_t y = tid < t.n && ((x0 >> tid) & 1u) ? (a.lin ? a.lin[tid] : 1u << tid) : 0u;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) y ^= __shfl_xor_sync(0xffffffffu, y, o);
      if (tid == 0) {
        at_yx[0] = y ^ (a.lin ? a.lin[t.n] : 0u) ^ (a.row_frame ? a.row_frame[lr] : 0u);
        at_yx[1] = x0;
      }
    }
    __syncthreads();
    const uint32_t y0 = at_yx[0] ^ oy, x0 = at_yx[1] ^ ox;
    const c2* psi = t.psi + (size_t)lr * dim;
    c2 v[kOutPer];
    if (on) {
#pragma unroll
      for (int i = 0; i < kOutPer; i++)
        if (i < per) v[i] = psi[y0 ^ cy[i]];
#pragma unroll
      for (int i = 0; i < kOutPer; i++)
        if (i < per) buf[swz(tid) ^ swz(256 * i)] = v[i];
    }
    __syncthreads();
    if (on) {
#pragma unroll
      for (int i = 0; i < kOutPer; i++)
        if (i < per) v[i] = buf[swz(at) ^ ca[i]];
      double* out = a.values + (a.output == TDQ_OUT_STATE ? 2 : 1) * b * dim;
#pragma unroll
      for (int i = 0; i < kOutPer; i++) {
        if (i >= per) continue;
        const size_t x = x0 ^ cx[i];
        if (a.output == TDQ_OUT_STATE) {
          out[2 * x] = exact_double(v[i].x);
          out[2 * x + 1] = exact_double(v[i].y);
        } else {
          out[x] = exact_square(v[i].x) + exact_square(v[i].y);
        }
      }
    }
  }
}

// The map of k1_state_out for x = A y (+ a constant).
OutMap out_map(const LinMap& map) {
  OutMap m{};
  const int n = map.n, r = std::min(5, n);
  std::vector<uint32_t> ax(n, 0);  // ax[i]: the x that y's bit i flips
  for (int q = 0; q < n; q++)
    for (int i = 0; i < n; i++) ax[i] |= ((map.row[q] >> i) & 1u) << q;
  // the space in the order of x (consecutive x first) and in the order of y
  LinSpace S;
  std::vector<uint32_t> bx, by;
  auto grow = [](LinSpace& sp, std::vector<uint32_t>& list, uint32_t v, int dim) {
    if ((int)sp.v.size() < dim && sp.reduce(v)) {
      sp.add(v);
      list.push_back(v);
    }
  };
  const int bits = std::min(n, kOutBits);
  for (int i = 0; i < r; i++) grow(S, bx, 1u << i, bits);
  for (int i = 0; i < r; i++) grow(S, bx, ax[i], bits);
  for (int i = r; i < n; i++) grow(S, bx, ax[i], bits);
  m.bits = bits;
  m.pivots = S.pivots();
  LinSpace Y;
  for (int i = 0; i < n; i++)
    if (!S.reduce(ax[i])) grow(Y, by, ax[i], bits);
  for (uint32_t v : bx) grow(Y, by, v, bits);
  auto y_of = [&](uint32_t x) {
    uint32_t y = 0;
    for (int q = 0; q < n; q++)
      if ((x >> q) & 1u) y ^= map.col[q];
    return y;
  };
  // everything is linear: entry l from the entries of its bits; `at` of a basis
  // vector are its coordinates in the other basis
  std::vector<std::pair<uint32_t, int>> rows;  // reduced vectors of `by`, and which they are sums of
  for (int i = 0; i < bits; i++) {
    std::pair<uint32_t, int> v{by[i], 1 << i};
    for (const auto& r : rows)
      if (v.first & r.first & (0u - r.first)) v = {v.first ^ r.first, v.second ^ r.second};
    const uint32_t low = v.first & (0u - v.first);
    for (auto& r : rows)
      if (r.first & low) r = {r.first ^ v.first, r.second ^ v.second};
    rows.push_back(v);
  }
  for (int i = 0; i < bits; i++) {
    int at = 0;
    for (const auto& r : rows)
      if (bx[i] & r.first & (0u - r.first)) at ^= r.second;
    m.x[1 << i] = bx[i];
    m.y[1 << i] = y_of(by[i]);
    m.at[1 << i] = (uint16_t)at;
  }
  for (int l = 1; l < (1 << bits); l++) {
    const int low = l & -l;
    m.x[l] = m.x[l ^ low] ^ m.x[low];
    m.y[l] = m.y[l ^ low] ^ m.y[low];
    m.at[l] = (uint16_t)(m.at[l ^ low] ^ m.at[low]);
  }
  return m;
}

}  // namespace

void tiled_free(TiledSweep& t) {
  for (cudaEvent_t e : t.ev) cudaEventDestroy(e);
  t.ev.clear();
  cudaFree(t.d_ops);
  cudaFree(t.d_off);
  cudaFree(t.d_loc);
  cudaFree(t.d_psi);
  cudaFree(t.d_lam);
  cudaFree(t.d_gacc);
  cudaFree(t.d_vals);
  cudaFree(t.d_ps_gate_pass);
  cudaFree(t.d_ps_rows);
  cudaFree(t.d_ps_first);
  cudaFree(t.d_alt);
  cudaFree(t.d_rpass);
  cudaFree(t.d_dops);
  cudaFree(t.d_rec_ptr);
  cudaFree(t.d_rec_ops);
  cudaFree(t.d_lin);
  cudaFree(t.d_rot);
  cudaFree(t.d_rot_x);
  cudaFree(t.d_rot_flips);
  cudaFree(t.d_coef);
  cudaFree(t.d_norm);
  cudaFree(t.d_out);
  t.d_out = nullptr;
  t.d_coef = nullptr;
  t.d_norm = nullptr;
  cudaFree(t.d_row_frame);
  t.d_lin = t.d_rot_x = t.d_rot_flips = t.d_row_frame = nullptr;
  t.d_rot = nullptr;
  t.d_ps_gate_pass = t.d_ps_rows = t.d_ps_first = nullptr;
  t.d_alt = nullptr;
  t.d_rpass = nullptr;
  t.d_dops = nullptr;
  t.d_rec_ptr = t.d_rec_ops = nullptr;
  t.d_ops = nullptr;
  t.d_off = nullptr;
  t.d_loc = nullptr;
  t.d_psi = t.d_lam = nullptr;
  t.d_gacc = t.d_vals = nullptr;
}

// Needs a gate on bit position p held in the tile?  (diagonal gates never,
// CNOT only for its target)
static void tile_needs(const SweepOp& op, std::vector<int>& need) {
  need.clear();
  switch (op.kind) {
    case K_RZ: case K_Z: case K_CZ: case K_RZZ: break;
    case K_CNOT: need.push_back(op.p1); break;
    default: need.push_back(op.p0); break;
  }
}

tdq_status tiled_plan(TiledSweep& t, const tdq_circuit* c, const std::vector<SweepOp>& ops,
                      const std::vector<int>& ps_gate, int rows, bool adj, int tile_qubits, int fb, int rb,
                      TiledHost& h) {
  t.fb = fb;
  t.rb = rb;
  const int n = c->n;
  t.n = n;
  const int kq = tile_qubits > 0 ? tile_qubits : 12;
  if (kq < 5 || kq > 13) return fail(TDQ_ERR_ARG, "tile_qubits must be in 5..13");
  t.k = std::min(n, kq);
  t.L = std::min(4, t.k);
  t.adj = adj;
  t.rows = rows;
  t.P = c->n_params;
  t.ng = c->n_groups;
  if (t.ng > 1024) return fail(TDQ_ERR_UNSUPPORTED, "tiled sweep: more than 1024 output groups");
  const int G = (int)ops.size();
  // Greedy pass schedule: walk gates in circuit order; take a gate when every
  // earlier gate on its qubits is taken and its non-diagonal bits fit in the
  // tile (growing the tile's bit set up to k); otherwise block its qubits for
  // the rest of this pass.
  std::vector<char> done(G, 0);
  std::vector<int> order;
  int remaining = G, first = 0;
  t.passes.clear();
  std::vector<int> need;
  while (remaining > 0) {
    uint32_t smask = (1u << t.L) - 1u;
    int used = t.L;
    std::vector<char> blocked(n, 0);
    TiledPass ps{0, (int)order.size(), 0};
    while (first < G && done[first]) first++;
    for (int g = first; g < G; g++) {
      if (done[g]) continue;
      const SweepOp& op = ops[g];
      const int pa = op.p0, pb = op.p1;
      if (blocked[pa] || (pb >= 0 && blocked[pb])) {
        blocked[pa] = 1;
        if (pb >= 0) blocked[pb] = 1;
        continue;
      }
      tile_needs(op, need);
      uint32_t add = 0;
      for (int p : need)
        if (!((smask >> p) & 1u)) add |= 1u << p;
      if (used + __builtin_popcount(add) <= t.k) {
        smask |= add;
        used += __builtin_popcount(add);
        done[g] = 1;
        remaining--;
        order.push_back(g);
      } else {
        blocked[pa] = 1;
        if (pb >= 0) blocked[pb] = 1;
      }
    }
    // fill the tile's unused slots with the lowest free positions
    for (int p = 0; p < n && used < t.k; p++)
      if (!((smask >> p) & 1u)) {
        smask |= 1u << p;
        used++;
      }
    ps.smask = smask;
    ps.op_end = (int)order.size();
    if (ps.op_end == ps.op_begin) return fail(TDQ_ERR_STATE, "tiled sweep: empty pass");
    t.passes.push_back(ps);
  }
  // device program in pass order; slot/src stay per op
  std::vector<SweepOp>& pops = h.pops;
  for (int g : order) pops.push_back(ops[g]);
  std::vector<int>& offs = h.offs;
  std::vector<int8_t>& locs = h.locs;
  int maxp = 0;
  for (const TiledPass& ps : t.passes) {
    maxp = std::max(maxp, ps.op_end - ps.op_begin);
    std::vector<int> hi;
    int8_t loc[32];
    for (int p = 0; p < 32; p++) loc[p] = -1;
    int li = 0;
    for (int p = 0; p < n; p++)
      if ((ps.smask >> p) & 1u) {
        loc[p] = (int8_t)li++;
        if (p >= t.L) hi.push_back(p);
      }
    const int nh = t.k - t.L;
    for (int j = 0; j < (1 << nh); j++) {
      int o = 0;
      for (int i = 0; i < nh; i++)
        if ((j >> i) & 1) o |= 1 << hi[i];
      offs.push_back(o);
    }
    for (int p = 0; p < 32; p++) locs.push_back(loc[p]);
  }
  // decoded programs inside every tile pass (op indices are pass-ordered):
  // a fused forward program and, with gradients, a one-op-per-gate reverse one
  Program& prog = h.prog;
  t.max_rec = 0;
  int max_dops = 0;
  for (size_t pi = 0; pi < t.passes.size(); pi++) {
    const int r0 = (int)prog.rec_ptr.size() - 1, d0 = (int)prog.dops.size();
    t.rec_begin.push_back(r0);
    t.fp_begin.push_back((int)prog.passes.size());
    build_program(pops, t.passes[pi].op_begin, t.passes[pi].op_end, &locs[pi * 32], t.k, true, r0, fb, prog);
    t.fp_end.push_back((int)prog.passes.size());
    const int bd0 = (int)prog.dops.size();
    t.bp_begin.push_back((int)prog.passes.size());
    if (adj) build_program(pops, t.passes[pi].op_begin, t.passes[pi].op_end, &locs[pi * 32], t.k, false, r0, rb, prog);
    t.bp_end.push_back((int)prog.passes.size());
    t.bo_begin.push_back(bd0 - d0);
    t.bo_end.push_back((int)prog.dops.size() - d0);
    t.rec_end.push_back((int)prog.rec_ptr.size() - 1);
    for (int q = t.fp_begin.back(); q < t.bp_end.back(); q++) {  // op ranges relative to the tile pass
      prog.passes[q].op_begin -= d0;
      prog.passes[q].op_end -= d0;
    }
    t.dop_begin.push_back(d0);
    t.dop_end.push_back((int)prog.dops.size());
    t.max_rec = std::max(t.max_rec, t.rec_end.back() - r0);
    max_dops = std::max(max_dops, (int)prog.dops.size() - d0);
  }
  t.max_dops = max_dops;
  t.max_pass_ops = maxp;
  // parameter-shift copies refer to gates by index: renumber to pass order
  t.order = order;
  std::vector<int> pos(G, 0);
  std::vector<int>& psp = h.psp;
  for (int i = 0; i < G; i++) pos[order[i]] = i;
  for (int g : ps_gate) psp.push_back(pos[g]);
  return TDQ_OK;
}

tdq_status tiled_lin_plan(TiledSweep& t, const tdq_circuit* c, const std::vector<SweepOp>& ops, int rows, bool adj,
                          int tile_qubits, int fb, int rb, bool exact, LinProgram& prog) {
  t.fb = fb;
  t.rb = rb;
  t.n = c->n;
  const int kq = tile_qubits > 0 ? tile_qubits : 12;
  if (kq < 5 || kq > 13) return fail(TDQ_ERR_ARG, "tile_qubits must be in 5..13");
  t.k = std::min(t.n, kq);
  t.adj = adj;
  t.rows = rows;
  t.P = c->n_params;
  t.ng = c->n_groups;
  if (t.ng > 1024) return fail(TDQ_ERR_UNSUPPORTED, "tiled sweep: more than 1024 output groups");
  prog = lin_tiled_program(ops, t.n, t.k, fb, rb, adj, exact, &t.L);
  t.passes.clear();
  t.max_rec = 0;
  t.max_dops = 0;
  int r0 = 0;
  for (const LinTile& tile : prog.tiles) {
    t.passes.push_back({tile.pivots, 0, 0});
    const int nr = (int)tile.coef.size();
    t.rec_begin.push_back(r0);
    t.rec_end.push_back(r0 += nr);
    t.max_rec = std::max(t.max_rec, nr);
    for (std::vector<int>* v : {&t.fp_begin, &t.fp_end, &t.bp_begin, &t.bp_end, &t.bo_begin, &t.bo_end, &t.dop_begin,
                                &t.dop_end})
      v->push_back(0);
  }
  return TDQ_OK;
}

// Whether a forward kernel over 12-bit tiles runs in CTAs of 128 threads with
// one tile buffer, four per SM (fused with its reverse sweep three), or in two of
// 256 threads with two buffers.  A tile's load, its register passes (a
// barrier each) and its store follow one another, and more CTAs overlap them
// better than a second buffer does: 20-qubit ladder, 481 rows, values 8.81 ->
// 8.00 ms (two CTAs with one buffer 8.95, seven of 64 threads 9.37), fused last
// pass of 64 rows 732 -> 635 us.  A round of four (three) such CTAs takes 1.85 (1.45)
// rounds of two, so the last round's fill decides: 16 qubits, 24 rows, fused pass,
// 2.5 tiles per SM, one round for two 82 -> 47 us; 17 qubits, 16 rows, 3.4 per SM,
// two rounds either way, 106 us in CTAs of 256 and 125 in CTAs of 128.  (Reverse
// kernels stay at two of 256: 1.56 ms against 1.98 at three of 128.)  A pass of few
// register passes over parts of 128-byte lines waits for memory alone, and more
// tiles at once spread it thinner: 20 qubits, 16 rows, three register passes over
// 32-byte runs 94 us in CTAs of 256 and 111 in CTAs of 128; but four, 481 rows, 2.72 ms
// and 2.53, and two over whole lines 1.64 and 1.31.
static bool narrow_pass(const LinTile& tile, double tiles, int sms, bool fused) {
  bool lines = true;
  for (int i = 0; i < 4; i++) lines = lines && tile.v[i] == 1u << i;
  if (!lines && tile.fwd.size() < 4) return false;
  const double wide = std::ceil(tiles / (2.0 * sms));
  return fused ? 1.45 * std::ceil(tiles / (3.0 * sms)) < wide : 1.85 * std::ceil(tiles / (4.0 * sms)) < wide;
}

tdq_status tiled_compile(TiledSweep& t, const tdq_circuit* c, const std::vector<SweepOp>& ops,
                         const std::vector<int>& ps_gate, const std::vector<int>& ps_ang, int copies, int rows, bool adj,
                         int tile_qubits, const LinProgram* lin, int fb, int rb, bool whole_output, double* bytes_row) {
  TiledHost h;
  if (!lin) {
    tdq_status s0 = tiled_plan(t, c, ops, ps_gate, rows, adj, tile_qubits, fb, rb, h);
    if (s0 != TDQ_OK) return s0;
  } else {  // ops in circuit order; every pass's index offsets and table rows
    h.pops = ops;
    h.psp = ps_gate;
    for (const LinTile& tile : lin->tiles) {
      for (int j = 0; j < (1 << (t.k - t.L)); j++) {
        uint32_t o = 0;
        for (int i = 0; i < t.k - t.L; i++)
          if ((j >> i) & 1) o ^= tile.v[t.L + i];
        h.offs.push_back((int)o);
      }
      for (int p = 0; p < 32; p++) h.locs.push_back(-1);
    }
  }
  const bool interpret = lin == nullptr;
  const int n = c->n;
  const std::vector<SweepOp>& pops = h.pops;
  const std::vector<int>& offs = h.offs;
  const std::vector<int8_t>& locs = h.locs;
  const Program& prog = h.prog;
  const std::vector<int>& psp = h.psp;
  auto up = [](void** d, const void* h, size_t bytes) -> tdq_status {
    if (bytes == 0) return TDQ_OK;
    if (cudaMalloc(d, bytes) != cudaSuccess) return fail(TDQ_ERR_OOM, "tiled sweep: cudaMalloc");
    if (cudaMemcpy(*d, h, bytes, cudaMemcpyHostToDevice) != cudaSuccess)
      return fail(TDQ_ERR_CUDA, "tiled sweep: cudaMemcpy");
    return TDQ_OK;
  };
  tdq_status s;
  if (lin) {
    std::vector<uint32_t> map = lin->map.col;
    map.push_back(lin->map.to_y(0));
    if ((s = up((void**)&t.d_lin, map.data(), sizeof(uint32_t) * map.size())) != TDQ_OK) return s;
    t.quarter = lin->exact ? lin->map.quarter : 0;
    t.nrot = (int)lin->rot.size();
    std::vector<uint32_t> flips;
    for (const LinTile& tile : lin->tiles) flips.insert(flips.end(), tile.flips.begin(), tile.flips.end());
    if ((s = up((void**)&t.d_rot, lin->rot.data(), sizeof(CoefRec) * lin->rot.size())) != TDQ_OK) return s;
    if ((s = up((void**)&t.d_rot_x, lin->rot_x.data(), sizeof(uint32_t) * lin->rot_x.size())) != TDQ_OK) return s;
    std::vector<CoefRec> coef;
    std::vector<int> norm;
    for (const LinTile& tile : lin->tiles) {
      for (CoefRec q : tile.coef) {
        if (q.type != C_ROT && q.type != C_PHASE) q.code += (int)norm.size();
        coef.push_back(q);
      }
      norm.insert(norm.end(), tile.norm.begin(), tile.norm.end());
    }
    if ((s = up((void**)&t.d_coef, coef.data(), sizeof(CoefRec) * coef.size())) != TDQ_OK) return s;
    if ((s = up((void**)&t.d_norm, norm.data(), sizeof(int) * norm.size())) != TDQ_OK) return s;
    if ((s = up((void**)&t.d_rot_flips, flips.data(), sizeof(uint32_t) * flips.size())) != TDQ_OK) return s;
  }
  if ((s = up((void**)&t.d_ops, pops.data(), sizeof(SweepOp) * pops.size())) != TDQ_OK) return s;
  if ((s = up((void**)&t.d_off, offs.data(), sizeof(int) * offs.size())) != TDQ_OK) return s;
  if ((s = up((void**)&t.d_loc, locs.data(), locs.size())) != TDQ_OK) return s;
  if (!psp.empty() && (s = up((void**)&t.d_ps_gate_pass, psp.data(), sizeof(int) * psp.size())) != TDQ_OK)
    return s;
  if ((s = up((void**)&t.d_rpass, prog.passes.data(), sizeof(RegPass) * prog.passes.size())) != TDQ_OK) return s;
  if ((s = up((void**)&t.d_dops, prog.dops.data(), sizeof(DOp) * prog.dops.size())) != TDQ_OK) return s;
  if ((s = up((void**)&t.d_rec_ptr, prog.rec_ptr.data(), sizeof(int) * prog.rec_ptr.size())) != TDQ_OK) return s;
  if ((s = up((void**)&t.d_rec_ops, prog.rec_ops.data(), sizeof(int) * prog.rec_ops.size())) != TDQ_OK) return s;
  if (whole_output) {
    LinMap id;
    lin_ops({}, n, &id);
    const OutMap m = out_map(lin ? lin->map : id);
    if ((s = up((void**)&t.d_out, &m, sizeof(m))) != TDQ_OK) return s;
  }
  // resident rows: bounded by a workspace budget of 3/4 of free memory, 64 GiB at most
  size_t freeb = 0, totb = 0;
  cudaMemGetInfo(&freeb, &totb);
  const size_t per_row = ((size_t)1 << n) * sizeof(c2) * (adj ? 2 : 1);
  size_t budget = std::min<size_t>((size_t)64 << 30, freeb / 4 * 3);
  t.chunk_rows = (int)std::max<size_t>(1, std::min<size_t>((size_t)rows, budget / per_row));
  if ((size_t)t.chunk_rows * per_row > freeb) return fail(TDQ_ERR_OOM, "tiled sweep: state does not fit");
  if (cudaMalloc(&t.d_psi, ((size_t)1 << n) * sizeof(c2) * t.chunk_rows) != cudaSuccess)
    return fail(TDQ_ERR_OOM, "tiled sweep: state buffer");
  if (adj && cudaMalloc(&t.d_lam, ((size_t)1 << n) * sizeof(c2) * t.chunk_rows) != cudaSuccess)
    return fail(TDQ_ERR_OOM, "tiled sweep: adjoint buffer");
  if (t.nrot && cudaMalloc(&t.d_row_frame, sizeof(uint32_t) * t.chunk_rows) != cudaSuccess)
    return fail(TDQ_ERR_OOM, "tiled sweep: frame buffer");
  if (cudaMalloc(&t.d_gacc, sizeof(double) * std::max(1, t.P) * t.chunk_rows) != cudaSuccess)
    return fail(TDQ_ERR_OOM, "tiled sweep: gradient buffer");
  if (cudaMalloc(&t.d_vals, sizeof(double) * std::max(1, t.ng) * t.chunk_rows) != cudaSuccess)
    return fail(TDQ_ERR_OOM, "tiled sweep: value buffer");
  // Parameter shift: a copy's state is the unshifted copy's until the tile pass
  // that holds its angle (rotations that a pass has not reached yet commute with
  // what ran before them), so it starts there.  20-qubit ladder, 481 copies,
  // 361 of them in the second pass and 441 in the third: 7.99 -> 6.88 ms, the same bits.
  // Kept to executions whose rows are all resident; one more state per batch entry.
  t.copies = copies;
  t.ps_active.clear();
  if (lin && copies > 1 && t.chunk_rows == rows && lin->tiles.size() > 1 && c->n_groups > 0 &&
      cudaMalloc(&t.d_alt, ((size_t)1 << n) * sizeof(c2) * (rows / copies)) == cudaSuccess) {
    std::vector<int> first(copies, 0), list;
    for (int k = 1; k < copies; k++) {
      const int gate = ps_gate[(k - 1) / 2], ang = ps_ang[(k - 1) / 2];
      for (int p = (int)lin->tiles.size() - 1; p >= 0; p--)
        for (int o : lin->tiles[p].ops)
          if (lin->ops[o].op == gate && lin->ops[o].ang == ang && lin->ops[o].kind <= L_PHASE && lin->ops[o].kind != L_H)
            first[k] = p;
    }
    for (int p = 0; p < (int)lin->tiles.size(); p++) {
      const size_t at = list.size();
      for (int k = 0; k < copies; k++)
        if (first[k] <= p) list.push_back(k);
      t.ps_active.push_back((int)(list.size() - at));
    }
    if ((s = up((void**)&t.d_ps_rows, list.data(), sizeof(int) * list.size())) != TDQ_OK) return s;
    if ((s = up((void**)&t.d_ps_first, first.data(), sizeof(int) * first.size())) != TDQ_OK) return s;
  } else {
    cudaGetLastError();  // (no room: every copy runs every pass)
  }
  // threads: one forward group (2^4 amplitudes) per thread; reverse kernels
  // up to 256 threads (two CTAs per SM)
  t.nthreads = std::max(32, std::min(256, 1 << (t.k - fb)));
  t.nthreads_r = interpret ? t.nthreads : std::max(32, std::min(256, 1 << (t.k - rb)));
  t.kf.clear();
  t.kr.clear();
  t.spec_gbytes.clear();
  const int np = (int)t.passes.size();
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  t.sms = std::max(1, nsm);
  t.threads_f.assign(np, t.nthreads);
  if (!interpret && t.k == 12 && t.nthreads == 256)
    for (int p = 0; p < np; p++)
      if (narrow_pass(lin->tiles[p], std::ldexp((double)t.chunk_rows, p ? n - t.k : 0), t.sms, adj && p == np - 1))
        t.threads_f[p] = 128;
  int gmax = 0, ndops_sm = 0;
  std::vector<int> nacc(np, 0);  // gradient accumulators of every pass
  if (!interpret) {
    const int nw = std::max(t.nthreads, t.nthreads_r) / 32;
    for (int p = 0; p < np; p++) {
      if (adj)
        for (int o : lin->tiles[p].ops) nacc[p] += lin->ops[o].slot >= 0 ? 1 : 0;
      t.spec_gbytes.push_back(4 * nw * std::max(1, nacc[p]));
      gmax = std::max(gmax, t.spec_gbytes.back());
    }
  } else {
    gmax = 24 * t.max_rec;
    ndops_sm = t.max_dops;
  }
  // shared memory per kernel: forward kernels a double-buffered state (psi;
  // the last pass also lambda; one buffer where two do not fit, or in CTAs of
  // 128 threads, see narrow_pass).  Reverse kernels hold psi and lambda in one
  // buffer each: two CTAs of 256 threads
  // per SM then interleave one CTA's tile loads with the other's compute,
  // which measured faster than one double-buffered CTA of 512 threads.
  const int mbytes = interpret ? t.max_rec * (int)sizeof(OpMat) : coef_bytes(t.max_rec, t.nrot);
  auto sizes = [&](int nb) {
    t.smem_f.assign(np, 0);
    for (int p = 0; p < np; p++)
      t.smem_f[p] = k1_smem_bytes(t.k, t.L, p == 0 || t.threads_f[p] < t.nthreads ? 1 : nb, (adj && p == np - 1) ? 1 : 0, mbytes, ndops_sm,
                                  t.ng, gmax);
    t.smem_r = adj ? k1_smem_bytes(t.k, t.L, 1, 1, mbytes, ndops_sm, t.ng, gmax) : 0;
    size_t m = t.smem_r;
    for (size_t v : t.smem_f) m = std::max(m, v);
    return m;
  };
  t.dbl = sizes(2) <= 227 * 1024 ? 1 : 0;
  size_t smax = sizes(t.dbl ? 2 : 1);
  if (smax > 227 * 1024) return fail(TDQ_ERR_UNSUPPORTED, "tiled sweep: tile program too large");
  if (!interpret) {
    // every tile pass as straight-line code, a module per pass; those not in the
    // cache are compiled on a host thread each (failures surface again below)
    std::vector<JitCode> code(np);
    std::vector<int> todo;
    for (int p = 0; p < np; p++) {
      code[p] = k1_code(t, *lin, t.nthreads_r, p);
      if (!jit_cached(code[p])) todo.push_back(p);
    }
    std::atomic<size_t> next{0};
    std::vector<std::thread> pool;
    auto work = [&] {
      try {
        if (cudaSetDevice(dev) != cudaSuccess) return;
        for (size_t i = next++; i < todo.size(); i = next++) {
          const void* k = nullptr;
          jit_kernel(code[todo[i]], ("tdq_k1f_" + std::to_string(todo[i])).c_str(), &k);
        }
      } catch (...) {
      }
    };
    const size_t nt = std::min<size_t>(todo.size(), std::thread::hardware_concurrency());
    pool.reserve(nt);
    try {
      for (size_t w = 0; w < nt && nt > 1; w++) pool.emplace_back(work);
    } catch (...) {  // (as many threads as there are)
    }
    for (std::thread& th : pool) th.join();
    for (int p = 0; p < np; p++) {
      const void* kf = nullptr;
      const void* kr = nullptr;
      const std::string nf = "tdq_k1f_" + std::to_string(p), nr = "tdq_k1r_" + std::to_string(p);
      tdq_status s2 = jit_kernel(code[p], nf.c_str(), &kf);
      if (s2 != TDQ_OK) return s2;
      if (cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)t.smem_f[p]) != cudaSuccess)
        return fail(TDQ_ERR_CUDA, "tiled sweep: cudaFuncSetAttribute");
      if (adj && p + 1 < np) {
        if ((s2 = jit_kernel(code[p], nr.c_str(), &kr)) != TDQ_OK) return s2;
        if (cudaFuncSetAttribute(kr, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)t.smem_r) != cudaSuccess)
          return fail(TDQ_ERR_CUDA, "tiled sweep: cudaFuncSetAttribute");
      }
      t.kf.push_back(kf);
      t.kr.push_back(kr);
    }
  } else {
    const int sm = (int)smax;
    cudaFuncSetAttribute(k1_forward<true, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    cudaFuncSetAttribute(k1_forward<false, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    cudaFuncSetAttribute(k1_forward<true, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    cudaFuncSetAttribute(k1_forward<false, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    cudaFuncSetAttribute(k1_forward<true, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    cudaFuncSetAttribute(k1_forward<false, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    cudaFuncSetAttribute(k1_reverse, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  }
  // resident CTAs per kernel (occupancy of the kernel at its launch shape)
  {
    auto slots = [&](const void* fn, int threads, size_t smem) {
      int nb = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, threads, smem) != cudaSuccess || nb < 1) {
        cudaGetLastError();
        nb = 1;
      }
      return t.sms * nb;
    };
    t.slots_f.assign(np, 0);
    for (int p = 0; p < np; p++) {
      const bool f = p == 0, l = p == np - 1;
      const void* fn = !t.kf.empty() ? t.kf[p]
                       : (f && !l) ? (const void*)k1_forward<true, false, false>
                       : (!f && !l) ? (const void*)k1_forward<false, false, false>
                       : (f && !adj) ? (const void*)k1_forward<true, true, false>
                       : (!adj) ? (const void*)k1_forward<false, true, false>
                       : f ? (const void*)k1_forward<true, true, true>
                           : (const void*)k1_forward<false, true, true>;
      t.slots_f[p] = slots(fn, t.threads_f[p], t.smem_f[p]);
    }
    t.slots_r = t.sms;
    if (adj && np > 1) t.slots_r = slots(!t.kr.empty() ? t.kr[0] : (const void*)k1_reverse, t.nthreads_r, t.smem_r);
  }
  // HBM traffic model per row and launch unit: every pass reads and writes the
  // state (the first pass only writes it, a value-only last pass only reads
  // it); with the reverse sweep each earlier pass reads and writes psi and
  // lambda again.  From |0...0> the specialised passes' first one holds its one
  // nonzero tile, which is all that the second reads and the reverse of the
  // second leaves.
  const double sb = (double)((size_t)1 << n) * sizeof(c2);
  const double part = lin && np > 1 ? std::ldexp(1.0, t.k - n) : 1.0;
  auto in = [&](int p) { return p == 0 ? 0.0 : p == 1 ? part * sb : sb; };
  auto out = [&](int p) { return p == 0 ? part * sb : sb; };
  auto left = [&](int p) { return lin ? in(p) : sb; };  // of psi and lambda each, by the reverse of pass p
  // the FLOPs of each unit (forward passes, then the reverse passes from the
  // second last down): dense gates, or the operations of the specialised
  // passes per amplitude -- rotation 4, H and a pass's scale 2, its phases one
  // product 6; a dot 4 -- psi and lambda both in reverse
  const double dim = std::ldexp(1.0, n);
  const double obs = c->n_groups > 0 ? (3.0 + 2.0 * (double)c->terms.size()) * dim : 0.0;
  std::vector<double> fw(np, 0.0), dots(np, 0.0), bw(np, 0.0);
  for (int p = 0; p < np; p++) {
    for (int o = t.passes[p].op_begin; o < t.passes[p].op_end; o++) {
      fw[p] += gate_fwd_flops(pops[o].kind, dim);
      dots[p] += gate_dot_flops(pops[o].kind, dim);
    }
    bw[p] = 2 * fw[p] + dots[p];
    if (!lin) continue;
    auto count = [&](const LinReg& r, bool rev) {
      double c = r.norm >= 0 ? 2 : 0, dot = 0;
      bool phase = false;
      for (int o : r.ops) {
        const LinOp& g = lin->ops[o];
        c += g.kind == L_RY || g.kind == L_RX ? 4 : g.kind == L_H ? 2 : 0;
        phase |= g.kind == L_PHASE;
        dot += g.slot >= 0 && g.kind != L_PHASE ? 4 : 0;
      }
      c += phase ? 6 : 0;
      return (rev ? 2 * c + dot + (phase ? 4 : 0) : c) * dim * (p == 0 ? part : 1.0);
    };
    for (const LinReg& r : lin->tiles[p].fwd) fw[p] += count(r, false);
    if (adj)
      for (const LinReg& r : lin->tiles[p].rev) bw[p] += count(r, true);
  }
  t.unit_flops.clear();
  t.unit_bytes.clear();
  t.unit_kind.clear();
  for (int p = 0; p < np; p++) {
    const bool l = p == np - 1;
    t.unit_kind.push_back(l && adj ? 1 : 0);
    t.unit_flops.push_back(fw[p] + (l ? obs : 0.0) + (l && adj ? bw[p] + obs : 0.0));
    const double share = t.ps_active.empty() ? 1.0 : (double)t.ps_active[p] / copies;
    t.unit_flops.back() *= share;
    t.unit_bytes.push_back(share * (in(p) + (!l ? out(p) : adj ? 2 * left(p) : c->n_groups > 0 ? 0.0 : out(p))));
  }
  if (adj)
    for (int p = np - 2; p >= 0; p--) {
      t.unit_kind.push_back(2);
      t.unit_flops.push_back(bw[p]);
      t.unit_bytes.push_back(2 * (out(p) + left(p)));
    }
  *bytes_row = 0;
  for (double by : t.unit_bytes) *bytes_row += by;
  return TDQ_OK;
}

static void set_pass(const TiledSweep& t, TiledDev& d, int p) {
  d.fp = t.d_rpass + t.fp_begin[p];
  d.nfp = t.fp_end[p] - t.fp_begin[p];
  d.bp = t.d_rpass + t.bp_begin[p];
  d.nbp = t.bp_end[p] - t.bp_begin[p];
  d.dops = t.d_dops + t.dop_begin[p];
  d.ndops = t.dop_end[p] - t.dop_begin[p];
  d.bo0 = t.bo_begin[p];
  d.bo1 = t.bo_end[p];
  d.rec_ptr = t.d_rec_ptr;
  d.rec_ops = t.d_rec_ops;
  d.rec0 = t.rec_begin[p];
  d.nrec = t.rec_end[p] - t.rec_begin[p];
  if (t.kf.empty()) {
    d.gbytes = 24 * d.nrec;
  } else {  // specialised: no decoded ops in shared memory; per-warp FP32 rows
    d.ndops = 0;
    d.gbytes = t.spec_gbytes[p];
  }
}

// A launch that may be dispatched while the kernel before it in the stream is
// finishing (chained; the kernel waits in chain_wait).
static cudaError_t launch_chained(const void* k, dim3 g, dim3 b, void** args, size_t smem, cudaStream_t st,
                                  bool chained) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = g;
  cfg.blockDim = b;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, k, args);
}

tdq_status tiled_execute(TiledSweep& t, const SweepArgs& a0, int grad, cudaStream_t st,
                         int* launches) {
  SweepArgs a = a0;
  if (a.ps_copies > 1) a.ps_gate = t.d_ps_gate_pass;
  a.lin = t.d_lin;
  a.quarter = t.quarter;
  a.rot = t.d_rot;
  a.rot_x = t.d_rot_x;
  a.rot_flips = t.d_rot_flips;
  a.coef = t.d_coef;
  a.norm = t.d_norm;
  a.nrot = t.nrot;
  a.row_frame = t.d_row_frame;
  const bool adj = grad == TDQ_GRAD_ADJOINT;
  const int np = (int)t.passes.size();
  const int ntiles = 1 << (t.n - t.k);
  for (int row0 = 0; row0 < t.rows; row0 += t.chunk_rows) {
    const int nr = std::min(t.chunk_rows, t.rows - row0);
    if (cudaMemsetAsync(t.d_vals, 0, sizeof(double) * std::max(1, t.ng) * nr, st) != cudaSuccess)
      return fail(TDQ_ERR_CUDA, "tiled sweep: memset");
    if (adj && cudaMemsetAsync(t.d_gacc, 0, sizeof(double) * std::max(1, t.P) * nr, st) != cudaSuccess)
      return fail(TDQ_ERR_CUDA, "tiled sweep: memset");
    // one wave per kernel: as many CTAs as fit on the GPU at once, each
    // with an equal share of the chunk's (row, tile) units
    // (specialised programs from |0...0>: the first pass's one tile at base 0,
    // see k1_forward_body; a lone pass still writes a state output's zeros)
    const bool lone = !a.init && !t.kf.empty() && (np > 1 || a.output == TDQ_OUT_EXPVAL);
    auto grid_for = [&](int slots, TiledDev& dd, int p) {
      dd.ntiles = p == 0 && lone ? 1 : ntiles;
      const int64_t total = (int64_t)dd.nrows * dd.ntiles;
      const int64_t n0 = std::max<int64_t>(1, std::min<int64_t>(total, slots));
      const int64_t upc = (total + n0 - 1) / n0;
      dd.tiles_per_cta = (int)upc;
      return dim3((unsigned)((total + upc - 1) / upc));
    };
    TiledDev d{};
    d.ops = t.d_ops;
    d.psi = t.d_psi;
    d.lam = t.d_lam;
    d.gacc = t.d_gacc;
    d.vals = t.d_vals;
    d.n = t.n;
    d.k = t.k;
    d.L = t.L;
    d.row0 = row0;
    d.nrows = nr;
    d.dbl = t.dbl;
    const int nthr = t.nthreads;  // (generic kernels)
    const int store_last = (a.output != TDQ_OUT_EXPVAL) ? 1 : 0;  // amplitudes, states: read from HBM
    for (int p = 0; p < np; p++) {
      d.off = t.d_off + (size_t)p * (1 << (t.k - t.L));
      d.loc = t.d_loc + (size_t)p * 32;
      d.smask = t.passes[p].smask;
      d.op_begin = t.passes[p].op_begin;
      d.op_end = t.passes[p].op_end;
      set_pass(t, d, p);
      const bool f = p == 0, l = p == np - 1;
      if (!t.ps_active.empty()) {
        d.ps_rows = p ? d.ps_rows + d.ps_active : t.d_ps_rows;
        d.ps_first = t.d_ps_first;
        d.alt = t.d_alt;
        d.ps_active = t.ps_active[p];
        d.pass = p;
        d.nrows = nr / t.copies * d.ps_active;
      }
      const dim3 grid = grid_for(t.slots_f[p], d, p);
      const bool rec = !t.ev.empty() && row0 == 0;
      if (rec) cudaEventRecord(t.ev[2 * p], st);
      if (!t.kf.empty()) {
        int st_flag = (l && !adj) ? store_last : 1;
        void* args[] = {&a, &d, &st_flag};
        // the first pass follows the caller's work and the clears above: unchained
        if (launch_chained(t.kf[p], grid, dim3(t.threads_f[p]), args, t.smem_f[p], st, p > 0) != cudaSuccess)
          return fail(TDQ_ERR_CUDA, "tiled sweep: launch of a specialised pass");
        if (rec) cudaEventRecord(t.ev[2 * p + 1], st);
        (*launches)++;
        continue;
      }
      const size_t sm = t.smem_f[p];
      if (f && !l) k1_forward<true, false, false><<<grid, nthr, sm, st>>>(a, d, 1);
      else if (!f && !l) k1_forward<false, false, false><<<grid, nthr, sm, st>>>(a, d, 1);
      else if (f && l && !adj) k1_forward<true, true, false><<<grid, nthr, sm, st>>>(a, d, store_last);
      else if (!f && l && !adj) k1_forward<false, true, false><<<grid, nthr, sm, st>>>(a, d, store_last);
      else if (f && l && adj) k1_forward<true, true, true><<<grid, nthr, sm, st>>>(a, d, 1);
      else k1_forward<false, true, true><<<grid, nthr, sm, st>>>(a, d, 1);
      if (rec) cudaEventRecord(t.ev[2 * p + 1], st);
      (*launches)++;
    }
    if (adj) {
      for (int p = np - 2; p >= 0; p--) {
        d.off = t.d_off + (size_t)p * (1 << (t.k - t.L));
        d.loc = t.d_loc + (size_t)p * 32;
        d.smask = t.passes[p].smask;
        d.op_begin = t.passes[p].op_begin;
        d.op_end = t.passes[p].op_end;
        set_pass(t, d, p);
        const dim3 grid = grid_for(t.slots_r, d, p);
        const int u = np + (np - 2 - p);  // launch unit of this reverse pass
        const bool rec = !t.ev.empty() && row0 == 0;
        if (rec) cudaEventRecord(t.ev[2 * u], st);
        if (!t.kr.empty()) {
          void* args[] = {&a, &d};
          if (launch_chained(t.kr[p], grid, dim3(t.nthreads_r), args, t.smem_r, st, true) != cudaSuccess)
            return fail(TDQ_ERR_CUDA, "tiled sweep: launch of a specialised pass");
        } else {
          k1_reverse<<<grid, t.nthreads_r, t.smem_r, st>>>(a, d);
        }
        if (rec) cudaEventRecord(t.ev[2 * u + 1], st);
        (*launches)++;
      }
    }
    {
      int nr_ = nr, g = adj ? 1 : 0;
      void* args[] = {&a, &d, &nr_, &g};
      if (launch_chained((const void*)k1_finalize, dim3(nr), dim3(128), args, 0, st, !t.kf.empty()) != cudaSuccess)
        return fail(TDQ_ERR_CUDA, "tiled sweep: launch of the read-out");
    }
    (*launches)++;
    if (a.output == TDQ_OUT_STATE || a.output == TDQ_OUT_PROBS) {
      const int64_t tot = (int64_t)nr << t.n;
      k1_state_out<<<(unsigned)std::min<int64_t>(tot >> std::min(t.n, kOutBits), 8 * t.sms), 256, 0, st>>>(a, d, nr, t.d_out);
      (*launches)++;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(TDQ_ERR_CUDA, std::string("tiled sweep launch: ") + cudaGetErrorString(e));
  }
  return TDQ_OK;
}

}  // namespace tdq

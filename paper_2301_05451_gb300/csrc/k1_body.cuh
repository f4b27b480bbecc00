// K1 bodies: the tiled state sweep through HBM (one launch per tile pass).
// A pass holds k bit positions of the state (always the L lowest, so tiles
// are read in contiguous 2^L-amplitude runs); a tile is the 2^k amplitudes
// that share the bits outside them.  Each CTA loads its tiles into shared
// memory, absorbs the pass's gates there (register passes) and writes them
// back: one HBM read and write of the state per pass instead of one per gate.
//
// The gate program of a pass is a policy, as for K2: InterpTile decodes the
// host-built register passes at run time; a specialised program has them as
// straight-line code (bits, kinds and table rows compile-time constants).
#pragma once

#include "engine.cuh"

namespace tdq {

struct TiledDev {
  const SweepOp* ops;
  const int* off;      // this pass's 2^(k-L) offsets
  const int8_t* loc;   // this pass's 32 local-bit entries
  const RegPass* fp;   // this pass's forward register passes (ops relative to dop0)
  int nfp;
  const RegPass* bp;   // reverse register passes
  int nbp;
  const DOp* dops;     // this pass's decoded ops (forward then reverse)
  int ndops;
  int bo0, bo1;        // reverse ops range (relative)
  const int* rec_ptr;
  const int* rec_ops;
  int rec0, nrec;      // this pass's recipes
  c2* psi;
  c2* lam;
  double* gacc;
  double* vals;
  int n, k, L;
  uint32_t smask;
  int op_begin, op_end;
  int tiles_per_cta, ntiles;  // (tiles_per_cta: (row, tile) units per CTA)
  int row0;
  int nrows;           // rows of the chunk: units are (row, tile), row-major
  int gbytes;          // shared-memory bytes of the gradient partial sums
  int dbl;             // 1: two tile buffers in the forward kernels (loads overlap compute)
  // Parameter shift with shared prefixes (ps_rows: NULL without): copy k is the
  // unshifted copy up to pass ps_first[k].  A pass runs the ps_active copies
  // ps_rows of every batch entry; the unshifted copy, read by those that start
  // here, changes between its row and a second buffer (alt, per entry).
  const int* ps_rows;
  const int* ps_first;
  c2* alt;
  int ps_active, pass;
};

// Spread the bits of t over the positions of mask (lowest first).
__device__ __forceinline__ uint32_t deposit(uint32_t t, uint32_t mask) {
  uint32_t out = 0;
  for (uint32_t m = mask; m && t; m &= m - 1, t >>= 1)
    if (t & 1u) out |= m & (0u - m);
  return out;
}

struct TileShared {
  c2* psi;
  c2* lam;
  c2* psi2;     // second state buffer (double-buffered loads), or NULL
  OpMat* mats;  // [recipes of the pass] (specialised programs: float4 rows)
  DOp* dops;    // [decoded ops of the pass]
  double* red;
  double* vsum;         // [n_groups]
  unsigned char* gpart; // gradient partial sums (policy-defined), gbytes
  int* off;
  int8_t* loc;
};

// layout: psi[2^k] x npsi | lambda[2^k] x nlam | gate tensors[mbytes] | dops[ndops] | red[32] |
//         vsum[ng] | gpart[gbytes] | off[2^(k-L)] | loc[32]
__host__ __device__ __forceinline__ size_t k1_smem_bytes(int k, int L, int npsi, int nlam, int mbytes, int ndops,
                                                        int ng, int gbytes) {
  return (size_t)(1 << k) * sizeof(c2) * (npsi + nlam) + (size_t)mbytes + sizeof(DOp) * ndops +
         (32 + (size_t)ng) * sizeof(double) + (((size_t)gbytes + 7) & ~(size_t)7) + sizeof(int) * (1 << (k - L)) +
         32 + 16;
}

// Specialised programs have the tile's size and buffers as constants (kK tile
// bits, kBuffers state buffers of the forward kernels), so that lambda and
// the second buffer are immediate offsets.
template <class Prog>
__device__ __forceinline__ TileShared carve(unsigned char* raw, int k, int L, int npsi, int nlam, int mbytes,
                                            int ndops, int ng, int gbytes) {
  TileShared s;
  const int nloc = 1 << (Prog::kSpecialised ? Prog::kK : k);
  c2* p = reinterpret_cast<c2*>(raw);
  s.psi = p;
  s.psi2 = npsi > 1 ? p + nloc : nullptr;
  p += npsi * nloc;
  s.lam = nlam > 0 ? p : nullptr;
  p += nlam * nloc;
  s.mats = reinterpret_cast<OpMat*>(p);
  s.dops = reinterpret_cast<DOp*>(reinterpret_cast<unsigned char*>(p) + mbytes);
  s.red = reinterpret_cast<double*>(s.dops + ndops);
  s.vsum = s.red + 32;
  s.gpart = reinterpret_cast<unsigned char*>(s.vsum + ng);
  s.off = reinterpret_cast<int*>(s.gpart + ((gbytes + 7) & ~7));
  s.loc = reinterpret_cast<int8_t*>(s.off + (1 << (k - L)));
  return s;
}

__device__ __forceinline__ uint32_t gidx(const TileShared& s, uint32_t base, uint32_t j, int L) {
  return base ^ (uint32_t)s.off[j >> L] ^ (j & ((1u << L) - 1u));
}

// Diagonal weight of output group g at basis index x: from the table of
// every group's diagonal when the compile made one (read through L2, the
// same for every row), else from the group's Z-product terms.
template <class Prog>
__device__ __forceinline__ float obs_weight(const SweepArgs& a, int g, uint32_t x) {
  if (Prog::kDiag || a.odiag) return a.odiag[((size_t)g << a.n) + x];
  return diag_weight(a.terms, a.group_ptr[g], a.group_ptr[g + 1], x);
}

// Bytes of a pass's gate tensors.
template <class Prog>
__device__ __forceinline__ int k1_mat_bytes(const SweepArgs& a, const TiledDev& t) {
  return Prog::kSpecialised ? coef_bytes(t.nrec, a.nrot) : t.nrec * (int)sizeof(OpMat);
}

// Per-CTA set-up: offsets, local bits, this row's gate tensors (K0), the
// decoded ops (interpreted programs) and zeroed partial sums.
template <class Prog>
__device__ __forceinline__ void k1_setup(const SweepArgs& a, const TiledDev& t, const TileShared& s, int64_t b,
                                         int kk, int* bad) {
  const int noff = 1 << (t.k - t.L);
  for (int i = threadIdx.x; i < noff; i += blockDim.x) s.off[i] = t.off[i];
  if (threadIdx.x < 32) s.loc[threadIdx.x] = t.loc[threadIdx.x];
  // (interpreted programs: shifted gates are numbered in pass order, tiled_compile)
  if constexpr (Prog::kSpecialised)
    build_coefs(a, t.rec0, t.nrec, reinterpret_cast<float4*>(s.mats), b, kk, bad);
  else
    for (int i = threadIdx.x; i < t.nrec; i += blockDim.x)
      s.mats[i] = build_recipe(a, t.ops, t.rec_ptr, t.rec_ops, t.rec0 + i, b, kk, bad);
  for (int i = threadIdx.x; i < t.ndops; i += blockDim.x) s.dops[i] = t.dops[i];
  for (int i = threadIdx.x; i < t.gbytes / 4; i += blockDim.x) reinterpret_cast<float*>(s.gpart)[i] = 0.f;
  for (int g = threadIdx.x; g < a.n_groups; g += blockDim.x) s.vsum[g] = 0.0;
  __syncthreads();
}

// Gate program decoded at run time; gradient shares in FP64 per (recipe, angle).
struct InterpTile {
  static constexpr bool kSpecialised = false;
  static constexpr bool kFirst = false, kSecond = false, kDiag = false;
  static constexpr int kK = 0, kN = 30, kBuffers = 0, kGroups = 0;
  __device__ __forceinline__ static bool in_first(uint32_t) { return true; }
  // f(shared-memory slot, global index) for this thread's elements of a tile
  template <int NT, class F>
  __device__ __forceinline__ static void every(const TiledDev& t, const TileShared& s, uint32_t base, F&& f) {
    for (uint32_t j = threadIdx.x; j < (1u << t.k); j += blockDim.x) f(swz(j), gidx(s, base, j, t.L));
  }
  // buf: offset of the state buffer in use
  __device__ __forceinline__ static void forward(const TiledDev& t, const TileShared& s, uint32_t base, uint32_t buf) {
    const int ngroups = 1 << (t.k - kFwdRegBits);
    for (int i = 0; i < t.nfp; i++) {
      const RegPass rp = t.fp[i];
      for (int grp = threadIdx.x; grp < ngroups; grp += blockDim.x)
        fwd_group<kFwdRegBits>(s.psi + buf, rp, s.dops, s.mats, base, (uint32_t)grp);
      __syncthreads();
    }
  }
  __device__ __forceinline__ static void reverse(const TiledDev& t, const TileShared& s, uint32_t base, uint32_t buf) {
    const int ngroups = 1 << (t.k - kRevRegBits);
    double* gp = reinterpret_cast<double*>(s.gpart);
    for (int i = t.nbp - 1; i >= 0; i--) {
      const RegPass rp = t.bp[i];
      for (int g0 = 0; g0 < ngroups; g0 += blockDim.x)
        adj_group<kRevRegBits, false>(s.psi + buf, s.lam, rp, s.dops, s.mats, base, (uint32_t)(g0 + threadIdx.x),
                                         g0 + (int)threadIdx.x < ngroups, gp);
      __syncthreads();
    }
  }
  // partial sums into the row's gradient columns
  __device__ __forceinline__ static void flush(const SweepArgs& a, const TiledDev& t, const TileShared& s, int lr) {
    __syncthreads();
    const double* gp = reinterpret_cast<const double*>(s.gpart);
    for (int i = t.bo0 + (int)threadIdx.x; i < t.bo1; i += blockDim.x) {
      const DOp d = s.dops[i];
      for (int j = 0; j < d.nang; j++)
        if (d.slot[j] >= 0) atomicAdd(&t.gacc[(int64_t)lr * a.P + d.slot[j]], gp[3 * d.mat + j]);
    }
  }
};

// Element x of a state in HBM (a 32-bit byte offset where the state is small
// enough for one).
template <class Prog>
__device__ __forceinline__ c2* elem(c2* g, uint32_t x) {
  if (Prog::kSpecialised && Prog::kN <= 29) return reinterpret_cast<c2*>(reinterpret_cast<unsigned char*>(g) + (x << 3));
  return g + x;
}

// Starts the asynchronous load of tile `base` of state g into buffer buf
// (one commit group per thread).
// sparse: only the elements on the first pass's space; the others are zero.
// Specialised programs move pairs of neighbours, 16 bytes past L1 (8-byte copies
// keep the load pipe busy that the register passes read shared memory with):
// 20-qubit ladder, 481 rows 9.39 -> 8.81 ms, 64 rows with gradient 4.68 -> 4.46 ms.
template <int NT, class Prog>
__device__ __forceinline__ void k1_issue(c2* buf, c2* g, const TiledDev& t, const TileShared& s, uint32_t base,
                                         bool sparse = false) {
  if constexpr (Prog::kSpecialised)
    Prog::template pairs<NT>(t, s, base, [&](uint32_t j, uint32_t x) {
      if (!(Prog::kSecond && sparse) || Prog::in_first(x)) cp_async16(&buf[j], elem<Prog>(g, x));
      else *reinterpret_cast<float4*>(&buf[j]) = make_float4(0.f, 0.f, 0.f, 0.f);
    });
  else
    Prog::template every<NT>(t, s, base, [&](uint32_t j, uint32_t x) { cp_async8(&buf[j], elem<Prog>(g, x)); });
}

// Writes buffer buf to tile `base` of state g (sparse as above: nothing else).
template <int NT, class Prog>
__device__ __forceinline__ void k1_store(const c2* buf, c2* g, const TiledDev& t, const TileShared& s, uint32_t base,
                                         bool sparse = false) {
  if constexpr (Prog::kSpecialised)
    Prog::template pairs<NT>(t, s, base, [&](uint32_t j, uint32_t x) {
      if (Prog::kSecond && sparse && !Prog::in_first(x)) return;
      *reinterpret_cast<float4*>(elem<Prog>(g, x)) = *reinterpret_cast<const float4*>(&buf[j]);
    });
  else
    Prog::template every<NT>(t, s, base, [&](uint32_t j, uint32_t x) { *elem<Prog>(g, x) = buf[j]; });
}

// The (row, tile) units of this CTA: a contiguous range of the row-major
// unit index, cut into per-row segments: tiles [tile0, tile1) of row lr.  (Not
// a callback: the largest programs' was compiled as a function of its own, and
// spilled 1.6 KB at its register limit.)
struct Segments {
  int64_t u, u1;
  int lr = 0, tile0 = 0, tile1 = 0;
  bool first = true;
  __device__ __forceinline__ explicit Segments(const TiledDev& t) {
    u = (int64_t)blockIdx.x * t.tiles_per_cta;
    u1 = min((int64_t)t.nrows * t.ntiles, u + t.tiles_per_cta);
  }
  __device__ __forceinline__ bool next(const TiledDev& t) {
    if (u >= u1) return false;
    if (!first) __syncthreads();  // the previous row's partial sums are read out
    first = false;
    lr = (int)(u / t.ntiles);
    tile0 = (int)(u - (int64_t)lr * t.ntiles);
    tile1 = (int)min((int64_t)t.ntiles, tile0 + (u1 - u));
    u += tile1 - tile0;
    return true;
  }
};

// Forward pass.  FIRST: the tile starts as the initial state (|0...0> or the
// caller's) instead of being read.  LAST: accumulate the observable groups; with GRAD also form lambda = O_w psi
// and run this pass's reverse sweep at once (psi and lambda then written).
// Tiles after the first of a row segment are read while the previous one is
// being computed (two shared-memory buffers; specialised CTAs of 128 threads have
// one and leave the overlap to the three others of their SM, see narrow_pass).
// NT: threads per CTA (specialised programs).
//
// From |0...0> the state after the first pass is zero outside the pass's tile
// at base 0 (the space V0).  Specialised programs use that at both ends: the
// first pass only visits that tile (the launch has one tile per row); the
// second pass (Prog::kSecond) takes every element outside V0 as zero instead
// of reading it, and its reverse sweep keeps psi and lambda only on V0, all
// that the first pass's reverse sweep visits (its gradient shares are
// products with psi, zero elsewhere).  On the 20-qubit ladder (64 rows) the
// first pass went from 116 to 16 us forward and from 2.9 ms to 59 us in reverse.
template <int NT, bool FIRST, bool LAST, bool GRAD, class Prog>
__device__ __forceinline__ void k1_forward_body(const SweepArgs& a, const TiledDev& t, int store) {
  extern __shared__ __align__(16) unsigned char raw[];
  const int nbuf = FIRST ? 1 : Prog::kSpecialised ? Prog::kBuffers : (t.dbl ? 2 : 1);
  const TileShared s = carve<Prog>(raw, t.k, t.L, nbuf, (GRAD && LAST) ? 1 : 0, k1_mat_bytes<Prog>(a, t), t.ndops,
                                   a.n_groups, t.gbytes);
  const uint32_t dim = 1u << t.n;
  const uint32_t other = (dim - 1u) & ~t.smask;
  // the gate tensors and tables are built while the kernel before finishes
  // (the first kernel of an execution is launched unchained): 17-qubit ladder,
  // 5 rows, 7 passes of 15 to 50 us, 215 -> 143 us; 16 qubits, 24 rows, 218 -> 168
  chain_dispatch();
  bool waited = false;
  for (Segments seg(t); seg.next(t);) {
    const int tile0 = seg.tile0, tile1 = seg.tile1;
    int lr = seg.lr;
    if (Prog::kSpecialised && !GRAD && t.ps_rows)
      lr = lr / t.ps_active * a.ps_copies + t.ps_rows[lr % t.ps_active];
    const int row = t.row0 + lr;
    const int64_t b = row / a.ps_copies;
    const int kk = row % a.ps_copies;
    int bad = 0;
    k1_setup<Prog>(a, t, s, b, kk, &bad);
    if (!waited) chain_wait();
    waited = true;
    if (bad) atomicOr(a.status, 1 << TDQ_ERR_NONFINITE);
    c2* gpsi = t.psi + (size_t)lr * dim;
    c2* glam = GRAD ? t.lam + (size_t)lr * dim : nullptr;
    c2 *gin = gpsi, *gout = gpsi;
    if (Prog::kSpecialised && !GRAD && t.ps_rows) {
      c2 *even = t.psi + (size_t)(lr - kk) * dim, *odd = t.alt + (size_t)b * dim;
      if (kk == 0 || t.ps_first[kk] == t.pass) gin = (t.pass & 1) ? odd : even;
      if (kk == 0) gout = (t.pass & 1) ? even : odd;
    }
    // index part of the row's frame: the observable of y is read at y ^ mu
    uint32_t mu = 0u;
    if constexpr (Prog::kSpecialised && LAST) {
      mu = coef_frame(reinterpret_cast<const float4*>(s.mats), t.nrec, a.nrot);
      if (a.row_frame && threadIdx.x == 0) a.row_frame[lr] = mu;
    }
    if (!FIRST && nbuf == 2 && tile0 < tile1) {
      k1_issue<NT, Prog>(s.psi, gin, t, s, deposit((uint32_t)tile0, other), !a.init);
      cp_async_commit();
    }
    for (int tile = tile0, it = 0; tile < tile1; tile++, it++) {
      const uint32_t base = deposit((uint32_t)tile, other);
      // offset of the state buffer in use
      const uint32_t buf = !FIRST && nbuf == 2 && (it & 1) ? (uint32_t)(s.psi2 - s.psi) : 0u;
      // this thread's elements: f(shared-memory slot, global index)
      auto every = [&](auto&& f) { Prog::template every<NT>(t, s, base, f); };
      if (FIRST && !Prog::kSpecialised && !a.init && base != 0u) {
        // from |0...0>, the pass's gates mix amplitudes within a tile only,
        // so every tile but the one at base 0 stays zero: write it out as
        // zeros (psi, and lambda = O psi = 0 when the reverse sweep is fused)
        // without its gates; nothing in shared memory is touched
        if (store || (LAST && GRAD))
          every([&](uint32_t, uint32_t x) {
            gpsi[x] = {0.f, 0.f};
            if (LAST && GRAD) glam[x] = {0.f, 0.f};
          });
        continue;
      }
      if (FIRST) {
        if (a.init) {
          const c2* p0 = a.init + b * a.init_stride;
          if constexpr (Prog::kSpecialised) {
            const bool wide = (reinterpret_cast<unsigned long long>(p0) & 15u) == 0;  // (the caller's pointer)
            Prog::template pairs<NT>(t, s, base, [&](uint32_t j, uint32_t x) {
              float4 v;
              if (wide) v = *reinterpret_cast<const float4*>(p0 + x);
              else v = make_float4(p0[x].x, p0[x].y, p0[x + 1].x, p0[x + 1].y);
              s.psi[j] = quarter_turns({v.x, v.y}, a.quarter);
              s.psi[j + 1] = quarter_turns({v.z, v.w}, a.quarter);
            });
          } else {
            every([&](uint32_t j, uint32_t x) { s.psi[j] = quarter_turns(p0[x], a.quarter); });
          }
        } else {
          every([&](uint32_t j, uint32_t x) { s.psi[j] = quarter_turns({x == 0u ? 1.f : 0.f, 0.f}, a.quarter); });
        }
      } else if (nbuf == 2) {
        if (tile + 1 < tile1) {  // the buffer of the previous tile is free (barrier at the loop end)
          k1_issue<NT, Prog>((it & 1) ? s.psi : s.psi2, gin, t, s, deposit((uint32_t)(tile + 1), other), !a.init);
          cp_async_commit();
          cp_async_wait<1>();
        } else {
          cp_async_wait<0>();
        }
      } else {  // one buffer: load, then compute
        k1_issue<NT, Prog>(s.psi, gin, t, s, base, !a.init);
        cp_async_commit();
        cp_async_wait<0>();
      }
      __syncthreads();
      Prog::forward(t, s, base, buf);
      if (LAST && a.output == TDQ_OUT_EXPVAL) {
        // the observable's diagonal gives the values (sum |psi|^2 d) and, with
        // gradients, lambda = sum_g w_g d_g psi (a thread's own elements: no
        // barrier between the groups)
        const int ng = Prog::kGroups == 1 ? 1 : a.n_groups;
        for (int g = 0; g < ng; g++) {
          float acc = 0.f;
          const float w = GRAD && a.gw ? (float)a.gw[b * ng + g] : 1.f;
          every([&](uint32_t j, uint32_t x) {
            const c2 v = s.psi[j ^ buf];
            const float d = obs_weight<Prog>(a, g, x ^ mu);
            acc += (v.x * v.x + v.y * v.y) * d;
            if (GRAD) {
              const c2 l = g ? s.lam[j] : c2{0.f, 0.f};
              s.lam[j] = {fmaf(w * d, v.x, l.x), fmaf(w * d, v.y, l.y)};
            }
          });
          acc = warp_sum_f(acc);
          if ((threadIdx.x & 31) == 0) atomicAdd(&s.vsum[g], (double)acc);
        }
        if (GRAD) {
          __syncthreads();
          Prog::reverse(t, s, base, buf);
          if (!(FIRST && Prog::kSpecialised)) {  // nothing reads them after the first pass's reverse sweep
            k1_store<NT, Prog>(s.psi + buf, gpsi, t, s, base, !a.init);
            k1_store<NT, Prog>(s.lam, glam, t, s, base, !a.init);
          }
        }
      }
      if (!(LAST && GRAD) && store) k1_store<NT, Prog>(s.psi + buf, gout, t, s, base);
      __syncthreads();
    }
    if (LAST && a.output == TDQ_OUT_EXPVAL) {
      __syncthreads();
      for (int g = threadIdx.x; g < a.n_groups; g += blockDim.x)
        atomicAdd(&t.vals[(int64_t)lr * a.n_groups + g], s.vsum[g]);
    }
    if (GRAD && LAST) Prog::flush(a, t, s, lr);
  }
}

// Reverse pass over the tiles of one pass (passes before the last), one
// buffer per state: two CTAs per SM overlap one's loads with the other's
// compute.
template <int NT, class Prog>
__device__ __forceinline__ void k1_reverse_body(const SweepArgs& a, const TiledDev& t) {
  extern __shared__ __align__(16) unsigned char raw[];
  const TileShared s = carve<Prog>(raw, t.k, t.L, 1, 1, k1_mat_bytes<Prog>(a, t), t.ndops, a.n_groups, t.gbytes);
  const uint32_t dim = 1u << t.n;
  const uint32_t other = (dim - 1u) & ~t.smask;
  chain_dispatch();
  bool waited = false;
  for (Segments seg(t); seg.next(t);) {
    const int lr = seg.lr, tile0 = seg.tile0, tile1 = seg.tile1;
    const int row = t.row0 + lr;
    const int64_t b = row / a.ps_copies;
    int bad = 0;
    k1_setup<Prog>(a, t, s, b, 0, &bad);
    if (!waited) chain_wait();
    waited = true;
    c2* gpsi = t.psi + (size_t)lr * dim;
    c2* glam = t.lam + (size_t)lr * dim;
    for (int tile = tile0; tile < tile1; tile++) {
      const uint32_t base = deposit((uint32_t)tile, other);
      k1_issue<NT, Prog>(s.psi, gpsi, t, s, base);
      k1_issue<NT, Prog>(s.lam, glam, t, s, base);
      cp_async_commit();
      // the next tile's lines on their way to L2 meanwhile (a thread per
      // 128-byte run of 16 amplitudes)
      if (tile + 1 < tile1) {
        const uint32_t next = deposit((uint32_t)(tile + 1), other);
        for (uint32_t r = threadIdx.x; r < (1u << (t.k - t.L)); r += blockDim.x) {
          const uint32_t x = gidx(s, next, r << t.L, t.L);
          prefetch_l2(gpsi + x);
          prefetch_l2(glam + x);
        }
      }
      cp_async_wait<0>();
      __syncthreads();
      Prog::reverse(t, s, base, 0u);
      if (!Prog::kFirst) {
        k1_store<NT, Prog>(s.psi, gpsi, t, s, base, !a.init);
        k1_store<NT, Prog>(s.lam, glam, t, s, base, !a.init);
      }
      __syncthreads();
    }
    Prog::flush(a, t, s, lr);
  }
}

}  // namespace tdq

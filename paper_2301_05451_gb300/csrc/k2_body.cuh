// K2 body: one CTA holds one row's whole state in shared memory and runs the
// forward sweep, the observable epilogue (K6) and the reverse sweep (K7) of
// the state-sweep contraction path (Sec. 3.2 (e), Sec. 4.1).
//
// The gate program is a policy: InterpProg decodes the host-built register
// passes at run time; a specialised program (generated per circuit, compiled
// at run time) has every pass and gate as straight-line code with its bits as
// compile-time constants.  Both use the same register gate kernels.
#pragma once

#include "engine.cuh"

namespace tdq {

// Gate program read from shared memory at run time.  Gradient shares go to
// FP64 shared-memory sums, one per parameter column.
struct InterpProg {
  static constexpr bool kSpecialised = false;
  using Mat = OpMat;
  const RegPass* passes;
  int npf, npb;
  const DOp* dops;  // in shared memory

  template <int MF>
  __device__ __forceinline__ void forward(c2* psi, const OpMat* mats, int dim) const {
    for (int pi = 0; pi < npf; pi++) {
      const RegPass rp = passes[pi];
      for (int grp = threadIdx.x; grp < (dim >> MF); grp += blockDim.x)
        fwd_group<MF>(psi, rp, dops, mats, 0u, (uint32_t)grp);
      __syncthreads();
    }
  }

  template <int MB>
  __device__ __forceinline__ void reverse(c2* psi, c2* lam, const OpMat* mats, int dim, double* gacc,
                                          float*) const {
    const int nbg = dim >> MB;
    for (int pi = npf + npb - 1; pi >= npf; pi--) {
      const RegPass rp = passes[pi];
      for (int g0 = 0; g0 < nbg; g0 += blockDim.x)  // uniform trip count: warp reductions inside
        adj_group<MB, true>(psi, lam, rp, dops, mats, 0u, (uint32_t)(g0 + threadIdx.x),
                            g0 + (int)threadIdx.x < nbg, gacc);
      __syncthreads();
    }
  }
};

// Shared-memory bytes of the gradient accumulators.
__host__ __device__ constexpr size_t k2_grad_bytes(bool specialised, int P, int nthreads) {
  return specialised ? sizeof(float) * (size_t)P * (size_t)(nthreads / 32) : sizeof(double) * (size_t)P;
}

// Row r of the batch (with parameter shift: sample r / copies, copy r % copies).
// layout: psi[dim] | lambda[dim] (GRAD) | mats[nrec] (specialised: coef_bytes) | dops[ndops] | grad accumulators | red[32] | bad
template <int MF, int MB, bool GRAD, class Prog>
__device__ __forceinline__ void k2_body(const SweepArgs& a, Prog prog, const DOp* gdops, int ndops,
                                        const int* rec_ptr, const int* rec_ops, int nrec, int r) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int dim = 1 << a.n;
  c2* psi = reinterpret_cast<c2*>(smem_raw);
  c2* lam = psi + dim;
  using Mat = typename Prog::Mat;
  Mat* mats = reinterpret_cast<Mat*>(psi + (GRAD ? 2 : 1) * dim);
  DOp* dops = reinterpret_cast<DOp*>(reinterpret_cast<unsigned char*>(mats) +
                                     (Prog::kSpecialised ? coef_bytes(nrec, a.nrot) : (int)sizeof(Mat) * nrec));
  unsigned char* gbase = reinterpret_cast<unsigned char*>(dops + ndops);
  const size_t gbytes = GRAD ? k2_grad_bytes(Prog::kSpecialised, a.P, blockDim.x) : 0;
  double* gacc = reinterpret_cast<double*>(gbase);
  float* gpart = reinterpret_cast<float*>(gbase);
  double* red = reinterpret_cast<double*>(gbase + ((gbytes + 7) & ~(size_t)7));
  int* sbad = reinterpret_cast<int*>(red + 32);

  const int64_t b = r / a.ps_copies;
  const int k = r % a.ps_copies;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid == 0) *sbad = 0;
  __syncthreads();
  // K0: this row's gate tensors (fused products for the forward program)
  int bad = 0;
  if constexpr (Prog::kSpecialised)
    build_coefs(a, 0, nrec, mats, b, k, &bad);
  else
    for (int i = tid; i < nrec; i += nt) mats[i] = build_recipe(a, a.ops, rec_ptr, rec_ops, i, b, k, &bad);
  for (int i = tid; i < ndops; i += nt) dops[i] = gdops[i];
  if (bad) atomicOr(sbad, 1);
  if (a.init) {
    const c2* p0 = a.init + b * a.init_stride;
    for (int x = tid; x < dim; x += nt) psi[swz(x)] = quarter_turns(p0[x], a.quarter);
  } else {
    for (int x = tid; x < dim; x += nt) psi[swz(x)] = quarter_turns({x == 0 ? 1.f : 0.f, 0.f}, a.quarter);
  }
  if (GRAD) {
    if (Prog::kSpecialised)
      for (int j = tid; j < a.P * (nt >> 5); j += nt) gpart[j] = 0.f;
    else
      for (int j = tid; j < a.P; j += nt) gacc[j] = 0.0;
  }
  if (!Prog::kSpecialised) prog.dops = dops;
  __syncthreads();
  prog.template forward<MF>(psi, mats, dim);

  // index part of the row's frame: basis place y sits at y ^ mu
  uint32_t mu = 0u;
  if constexpr (Prog::kSpecialised) mu = coef_frame(mats, nrec, a.nrot);
  // observable epilogue (K6) / amplitude, state or probability read-out
  double Fval = 0.0;
  if (a.output == TDQ_OUT_EXPVAL) {
    for (int g = 0; g < a.n_groups; g++) {
      float acc = 0.f;
      const int t0 = a.group_ptr[g], t1 = a.group_ptr[g + 1];
      if (a.odiag) {
        const float* D = a.odiag + (size_t)g * dim;
        for (int x = tid; x < dim; x += nt) {
          const c2 v = psi[swz(x)];
          acc += (v.x * v.x + v.y * v.y) * D[(uint32_t)x ^ mu];
        }
      } else {
        for (int x = tid; x < dim; x += nt) {
          const c2 v = psi[swz(x)];
          acc += (v.x * v.x + v.y * v.y) * diag_weight(a.terms, t0, t1, (uint32_t)x ^ mu);
        }
      }
      const double tot = block_sum((double)acc, red);
      const double w = a.gw ? a.gw[b * a.n_groups + g] : 1.0;
      Fval += w * tot;
      if (k == 0 && tid == 0 && !a.fine_rows) a.values[b * a.n_groups + g] = tot;
    }
  } else if (k == 0 && a.output == TDQ_OUT_AMPLITUDE) {
    for (int i = tid; i < a.A; i += nt) {
      const c2 v = psi[swz(a.amp_idx[i])];
      a.values[(b * a.A + i) * 2] = v.x;
      a.values[(b * a.A + i) * 2 + 1] = v.y;
    }
  } else if (k == 0 && a.output == TDQ_OUT_STATE) {
    for (int x = tid; x < dim; x += nt) {
      const c2 v = psi[swz(lin_index(a, (uint32_t)x))];
      a.values[(b * dim + x) * 2] = v.x;
      a.values[(b * dim + x) * 2 + 1] = v.y;
    }
  } else if (k == 0 && a.output == TDQ_OUT_PROBS) {
    for (int x = tid; x < dim; x += nt) {
      const c2 v = psi[swz(lin_index(a, (uint32_t)x) ^ mu)];
      a.values[b * dim + x] = (double)v.x * v.x + (double)v.y * v.y;
    }
  }
  if (a.ps_copies > 1 && tid == 0) a.ps_F[r] = Fval;

  if (GRAD) {
    // lambda = O_w psi,  O_w = sum_g w_g O_g (diagonal)
    for (int x = tid; x < dim; x += nt) {
      float d = 0.f;
      for (int g = 0; g < a.n_groups; g++) {
        const float w = a.gw ? (float)a.gw[b * a.n_groups + g] : 1.f;
        d += w * (a.odiag ? a.odiag[(size_t)g * dim + ((uint32_t)x ^ mu)]
                          : diag_weight(a.terms, a.group_ptr[g], a.group_ptr[g + 1], (uint32_t)x ^ mu));
      }
      const c2 v = psi[swz(x)];
      lam[swz(x)] = {d * v.x, d * v.y};
    }
    __syncthreads();
    prog.template reverse<MB>(psi, lam, mats, dim, gacc, gpart);
    if (Prog::kSpecialised) {
      const int nw = nt >> 5;
      for (int j = tid; j < a.P; j += nt) {
        double s = 0.0;
        for (int w = 0; w < nw; w++) s += (double)gpart[w * a.P + j];
        a.grads[b * a.P + j] = (float)s;
      }
    } else {
      for (int j = tid; j < a.P; j += nt) a.grads[b * a.P + j] = (float)gacc[j];
    }
  }
  __syncthreads();
  if (tid == 0 && *sbad) atomicOr(a.status, 1 << TDQ_ERR_NONFINITE);
}

// ------------------------------------------------------------ values of few rows
// An expectation of one row is one number, and where it is small every rounding
// of the state's amplitudes counts: 6 qubits, 36 rotations, one row in float
// leaves 4e-8, 1e-6 of the value in one evaluation out of five.  Where SMs and
// time are left (fine_values, sweep.cu), a second CTA per row takes the values
// from a state of two floats per number (2^-45), while the first sweeps the
// gradients in float.  What bounds it is the chain of gates: a barrier, shared
// memory there and back and some 100 dependent instructions, 0.28 us each.
constexpr int kFineOps = 64;   // gates staged at a time
// CTAs between the rows' and the values' that leave at once: on the SM beside it, a
// value's CTA slows the row's while both fetch cold code (6 qubits, one row, L2
// flushed: 21.2 us; 19.1 with a gap; 18.1 without the values' CTA).
constexpr int kFineGap = 8;

struct df {  // h + l, |l| at most half an ulp of h
  float h, l;
};
// (device: no fused multiply-adds made of these)
#if defined(__CUDACC__) || defined(__CUDACC_RTC__)
__device__ __forceinline__ float add1(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float mul1(float a, float b) { return __fmul_rn(a, b); }
#else
inline float add1(float a, float b) { return a + b; }
inline float mul1(float a, float b) { return a * b; }
#endif
__device__ __forceinline__ df df_norm(float h, float l) {
  const float s = add1(h, l);
  return {s, add1(l, -add1(s, -h))};
}
__device__ __forceinline__ df df_add(df a, df b) {
  const float s = add1(a.h, b.h), v = add1(s, -a.h);
  const float e = add1(add1(a.h, -add1(s, -v)), add1(b.h, -v));
  return df_norm(s, add1(e, add1(a.l, b.l)));
}
__device__ __forceinline__ df df_mul(df a, df b) {
  const float p = mul1(a.h, b.h), e = fmaf(a.h, b.h, -p);
  return df_norm(p, fmaf(a.h, b.l, fmaf(a.l, b.h, e)));
}
__device__ __forceinline__ df df_neg(df a) { return {-a.h, -a.l}; }
// c a + s b, the small parts summed in float
__device__ __forceinline__ df df_turn(df c, df a, df s, df b) {
  const float p = mul1(c.h, a.h), q = mul1(s.h, b.h), t = add1(p, q), v = add1(t, -p);
  const float e = add1(add1(p, -add1(t, -v)), add1(q, -v));
  const float l = fmaf(c.h, a.l, fmaf(c.l, a.h, fmaf(c.h, a.h, -p)));
  const float k = fmaf(s.h, b.l, fmaf(s.l, b.h, fmaf(s.h, b.h, -q)));
  return df_norm(t, add1(e, add1(l, k)));
}

constexpr df df_of(double v) { return {(float)v, (float)(v - (double)(float)v)}; }

// sin x and cos x to 2^-39 (2^-37 at the end of the float reduction), as sincos2
// but with the remainder and the series' leading terms in two floats throughout.
struct SinCosF {
  df s, c;
};
__device__ __forceinline__ SinCosF sincos_df(float x) {
  if (!reducible(x)) {
    const SinCos r = sincos2_far(x);
    return {{r.s, r.sl}, {r.c, r.cl}};
  }
  const float k = quadrant(x), m = mul1(k, 7.54979013e-8f);
  const df r = df_add(df_add({fmaf(-k, 1.5703125f, x), 0.f}, {-mul1(k, 4.83751297e-4f), 0.f}),
                      {-m, -fmaf(k, 7.54979013e-8f, -m)});
  const df p = df_mul(r, r);
  const float sq = fmaf(p.h, fmaf(p.h, fmaf(p.h, 1.60590438e-10f, -2.50521084e-8f), 2.7557319e-6f), -1.98412698e-4f);
  const df sv = df_add(df_of(-1.0 / 6), df_mul(p, df_add(df_of(1.0 / 120), df_mul(p, {sq, 0.f}))));
  const df s = df_add(r, df_mul(r, df_mul(p, sv)));
  const float cq = fmaf(p.h, fmaf(p.h, fmaf(p.h, -1.14707456e-11f, 2.08767570e-9f), -2.75573192e-7f), 2.48015873e-5f);
  const df cv = df_add(df_of(1.0 / 24), df_mul(p, df_add(df_of(-1.0 / 720), df_mul(p, {cq, 0.f}))));
  const df c = df_add({1.f, 0.f}, df_mul(p, df_add({-0.5f, 0.f}, df_mul(p, cv))));
  const int q = (int)k & 3;
  SinCosF o = (q & 1) ? SinCosF{c, s} : SinCosF{s, c};
  if (q & 2) o.s = df_neg(o.s);
  if (q == 1 || q == 2) o.c = df_neg(o.c);
  return o;
}

struct zf {  // a complex number of two dfs
  df x, y;
};
__device__ __forceinline__ zf zf_get(const float4& v) { return {{v.x, v.y}, {v.z, v.w}}; }
__device__ __forceinline__ float4 zf_put(zf v) { return make_float4(v.x.h, v.x.l, v.y.h, v.y.l); }

__host__ __device__ __forceinline__ size_t k2_fine_bytes(int n) {
  return ((size_t)16 << n) + kFineOps * (sizeof(FineOp) + sizeof(float4)) + 32 * sizeof(double);
}

// layout: psi[dim] (x.h, x.l, y.h, y.l) | ops[kFineOps] | coefficients[kFineOps] | red[32]
static __device__ __noinline__ void k2_fine_row(const SweepArgs& a, int64_t b) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const uint32_t dim = 1u << a.n, tid = threadIdx.x, nt = blockDim.x;
  float4* psi = reinterpret_cast<float4*>(smem_raw);
  FineOp* ops = reinterpret_cast<FineOp*>(psi + dim);
  float4* cf = reinterpret_cast<float4*>(ops + kFineOps);
  double* red = reinterpret_cast<double*>(cf + kFineOps);
  for (uint32_t y = tid; y < dim; y += nt) {
    const c2 v = a.init ? a.init[b * a.init_stride + y] : c2{y == 0u ? 1.f : 0.f, 0.f};
    psi[y] = make_float4(v.x, 0.f, v.y, 0.f);
  }
  for (int o0 = 0; o0 < a.nfine; o0 += kFineOps) {
    const int no = a.nfine - o0 < kFineOps ? a.nfine - o0 : kFineOps;
    __syncthreads();
    for (int i = tid; i < no; i += nt) {
      const FineOp q = a.fine[o0 + i];
      ops[i] = q;
      if (q.kind == L_RY || q.kind == L_RX || q.kind == L_PHASE) {
        int bad = 0;
        const float v = coef_angle(a, {q.src, q.fixed, -1, 0}, b, 0, &bad);
        if (bad) atomicOr(a.status, 1 << TDQ_ERR_NONFINITE);
        const SinCosF r = sincos_df(q.kind == L_PHASE ? v : 0.5f * v);
        cf[i] = make_float4(r.c.h, r.c.l, r.s.h, r.s.l);
      }
    }
    __syncthreads();
    FineOp next = ops[0];  // (read ahead of the barrier)
    float4 nextc = cf[0];
    for (int i = 0; i < no;) {
      const FineOp q = next;
      const df c = {nextc.x, nextc.y}, s = {nextc.z, nextc.w}, ns = df_neg(s);
      i++;
      next = ops[min(i, kFineOps - 1)];
      nextc = cf[min(i, kFineOps - 1)];
      const uint32_t bit = q.m ? q.m : q.f, low = bit & (0u - bit), odd = (uint32_t)q.b & 1u;
      if (q.m) {
        // a phase on the same bit goes with it, on the pair's second member
        const bool also = i < no && next.kind == L_PHASE && next.f == q.f && next.b == q.b;
        const df pc = {nextc.x, nextc.y}, ps = {nextc.z, nextc.w};
        if (also) {
          i++;
          next = ops[min(i, kFineOps - 1)];
          nextc = cf[min(i, kFineOps - 1)];
        }
#pragma unroll 2
        for (uint32_t p = tid; p < dim / 2; p += nt) {
          const uint32_t y = ((p & ~(low - 1u)) << 1) | (p & (low - 1u));
          const uint32_t y0 = (((uint32_t)__popc(y & q.f) ^ odd) & 1u) ? y ^ q.m : y, y1 = y0 ^ q.m;
          const zf u = zf_get(psi[y0]), v = zf_get(psi[y1]);
          zf a0, a1;  // (logical 0 and 1)
          if (q.kind == L_RY) {
            a0 = {df_turn(c, u.x, ns, v.x), df_turn(c, u.y, ns, v.y)};
            a1 = {df_turn(c, v.x, s, u.x), df_turn(c, v.y, s, u.y)};
          } else if (q.kind == L_RX) {
            a0 = {df_turn(c, u.x, s, v.y), df_turn(c, u.y, ns, v.x)};
            a1 = {df_turn(c, v.x, s, u.y), df_turn(c, v.y, ns, u.x)};
          } else {  // L_H
            const df r = {0.70710678f, 1.21016175e-8f}, nr = df_neg(r);
            a0 = {df_turn(r, u.x, r, v.x), df_turn(r, u.y, r, v.y)};
            a1 = {df_turn(r, u.x, nr, v.x), df_turn(r, u.y, nr, v.y)};
          }
          if (also) a1 = {df_turn(pc, a1.x, df_neg(ps), a1.y), df_turn(pc, a1.y, ps, a1.x)};
          psi[y0] = zf_put(a0);
          psi[y1] = zf_put(a1);
        }
      } else {
        // the places whose logical bit is 1 (a global phase does not reach the values)
#pragma unroll 2
        for (uint32_t p = tid; p < dim / 2; p += nt) {
          uint32_t y = ((p & ~(low - 1u)) << 1) | (p & (low - 1u));
          if ((((uint32_t)__popc(y & q.f) ^ odd) & 1u) == 0u) y ^= low;
          const zf u = zf_get(psi[y]);
          if (q.kind == L_PHASE)
            psi[y] = zf_put({df_turn(c, u.x, ns, u.y), df_turn(c, u.y, s, u.x)});
          else if (q.kind == L_SIGN || (((uint32_t)__popc(y & q.f2) ^ ((uint32_t)q.b >> 1)) & 1u))
            psi[y] = zf_put({df_neg(u.x), df_neg(u.y)});
        }
      }
      __syncthreads();
    }
  }
  __syncthreads();
  // |psi|^2 in FP64 (in the amplitude's place), then every group's sum
  for (uint32_t y = tid; y < dim; y += nt) {
    const float4 v = psi[y];
    const double x = (double)v.x + (double)v.y, w = (double)v.z + (double)v.w;
    *reinterpret_cast<double*>(&psi[y]) = x * x + w * w;
  }
  for (int g = 0; g < a.n_groups; g++) {
    double acc = 0.0;
    for (uint32_t y = tid; y < dim; y += nt)
      acc += *reinterpret_cast<const double*>(&psi[y]) * (double)a.odiag[(size_t)g * dim + y];
    const double tot = block_sum(acc, red);
    if (tid == 0) a.values[b * a.n_groups + g] = tot;
  }
}

}  // namespace tdq

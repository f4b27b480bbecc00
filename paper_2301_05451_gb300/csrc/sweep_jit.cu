// Specialised sweep programs (see sweep_jit.h) and their run-time compilation.
#include "sweep_jit.h"

#include <cuda_runtime.h>
#include <nvJitLink.h>
#include <nvrtc.h>

#include <algorithm>
#include <atomic>
#include <charconv>
#include <cstdlib>
#include <map>
#include <mutex>
#include <thread>
#include <type_traits>

namespace tdq {

// The device headers the generated source includes, embedded at build time
// (kJitHeaderNames / kJitHeaderSrc / kJitHeaderCount).
#include "jit_headers.inc"

namespace {

// Generated text (half the time of a string stream).
class Text {
 public:
  Text& operator<<(const char* v) {
    b_.append(v);
    return *this;
  }
  Text& operator<<(const std::string& v) {
    b_.append(v);
    return *this;
  }
  template <class T, class = std::enable_if_t<std::is_integral<T>::value>>
  Text& operator<<(T v) {
    char d[24];
    b_.append(d, std::to_chars(d, d + sizeof(d), v).ptr);
    return *this;
  }
  const std::string& str() const { return b_; }

 private:
  std::string b_;
};

// (swz and swz_pair)
uint32_t swz_host(uint32_t x, bool pairs) {
  return pairs ? x ^ ((((x >> 4) ^ (x >> 7) ^ (x >> 10)) & 7u) << 1) : x ^ ((x >> 4) & 15u) ^ ((x >> 8) & 15u);
}

// A sign known at compile time up to group-dependent words: the XOR of the
// words w<i> (top bit) and a constant.
struct Sign {
  bool c = false;
  std::vector<int> w;
  void flip(const Sign& o) {
    c ^= o.c;
    for (int i : o.w) {
      auto it = std::find(w.begin(), w.end(), i);
      if (it == w.end()) w.push_back(i);
      else w.erase(it);
    }
  }
  bool constant() const { return w.empty(); }
  bool zero() const { return w.empty() && !c; }
  std::string str() const {
    std::string s;
    for (int i : w) s += (s.empty() ? "w" : " ^ w") + std::to_string(i);
    if (c) s += s.empty() ? "0x80000000u" : " ^ 0x80000000u";
    return s.empty() ? "0u" : s;
  }
};

// Writes one register pass: the group loop, its loads, gates and stores.
// Diagonal gates are gathered into blocks (an op may pass others it commutes
// with): a block multiplies every class of members that its parities tell
// apart by one product of phases.  The part of the phases that a whole group
// shares, and the scale that the unscaled rotations left out, are one factor
// per group, merged into the pass's largest block.  Signs (Z, CZ with one
// register bit) wait as a frame: a later gate on the bit flips its
// off-diagonal sign, a phase block absorbs them.
class PassWriter {
 public:
  PassWriter(Text& s, const LinProgram& P, const LinTile& t, const LinReg& r, bool rev)
      : s_(s), P_(P), t_(t), r_(r), rev_(rev), N_(1 << r.M) {
    for (int pos : r.grp_pos) varying_ |= t.v[pos];
    const uint32_t all = P.n >= 32 ? ~0u : (1u << P.n) - 1u;
    varying_ |= all & ~t.pivots;
    for (int i = 0; i < r.M; i++) {
      gu_[i] = 0;
      for (int l = 0; l < t.k; l++)
        if ((r.u[i] >> l) & 1u) gu_[i] ^= t.v[l];
    }
  }

  // share(o): where the gradient share of op o goes ("" if nowhere)
  template <class Share>
  void write(int nthreads, const std::string& y0, const std::vector<const char*>& arrays,
             const std::vector<const char*>& regs, Share share) {
    const int groups = 1 << (t_.k - r_.M);
    s_ << "  for (int grp = threadIdx.x; grp < " << groups << "; grp += " << nthreads << ") {\n";
    s_ << "    const uint32_t gb = " << spread() << ";\n    const uint32_t sb = " << (P_.pairs ? "swz_pair" : "swz")
       << "(gb);\n    const uint32_t y0 = " << y0
       << ";\n    (void)y0;\n";
    regs_ = regs;
    for (size_t i = 0; i < arrays.size(); i++) move(arrays[i], regs[i], false);
    plan();
    prelude();
    for (size_t i = 0; i < items_.size(); i++) {
      const std::vector<int>& it = items_[i];
      if (P_.ops[it[0]].kind == L_PHASE) block(it, (int)i == merge_, share);
      else gate(it[0], share);
    }
    if (merge_ < 0 && group_factor_) {
      const char* f = complex_factor_ ? "lin_mul" : "lin_scale";
      for (const char* g : regs)
        for (int j = 0; j < N_; j++) s_ << "    " << f << "(" << g << j << ", " << (complex_factor_ ? "G" : "G.x") << ");\n";
    }
    for (const Frame& f : frame_) flush(f);
    frame_.clear();
    for (size_t i = 0; i < arrays.size(); i++) move(arrays[i], regs[i], true);
    s_ << "  }\n";
  }

 private:
  struct Frame {
    int fr;
    Sign sign;
  };

  // local index of the group's first member: group bit i at local bit grp_pos[i]
  std::string spread() const {
    Text e;
    const int n = (int)r_.grp_pos.size();
    if (n == 0) return "0u * (uint32_t)grp";
    for (int i = 0; i < n;) {
      int j = i + 1;
      while (j < n && r_.grp_pos[j] == r_.grp_pos[i] + (j - i)) j++;
      const uint32_t mask = ((1u << (j - i)) - 1u) << i;
      const int sh = r_.grp_pos[i] - i;
      e << (i ? " | " : "") << "(((uint32_t)grp & " << mask << "u) " << (sh >= 0 ? "<< " : ">> ") << (sh >= 0 ? sh : -sh)
        << ")";
      i = j;
    }
    return e.str();
  }

  uint32_t member(int j) const {  // local index of member j from the group's first
    uint32_t l = 0;
    for (int i = 0; i < r_.M; i++)
      if ((j >> i) & 1) l ^= r_.u[i];
    return l;
  }

  void move(const char* arr, const char* reg, bool store) {
    // (a tile's state buffer in use starts at element `buf`)
    const char* sb = t_.k < P_.n && std::string(arr) == "psi" ? "[sb ^ buf ^ " : "[sb ^ ";
    // members that differ in local bit 0 are neighbours: 16 bytes at a time
    int pair = -1;
    for (int i = 0; i < r_.M; i++)
      if (P_.pairs && r_.u[i] == 1u) pair = i;
    for (int j = 0; j < N_; j++) {
      const uint32_t so = swz_host(member(j), P_.pairs);
      if (pair >= 0) {
        if ((j >> pair) & 1) continue;
        const int j2 = j | (1 << pair);
        if (store)
          s_ << "    *reinterpret_cast<float4*>(&" << arr << sb << so << "u]) = make_float4(" << reg << j << ".x, " << reg
             << j << ".y, " << reg << j2 << ".x, " << reg << j2 << ".y);\n";
        else
          s_ << "    const float4 " << reg << "q" << j << " = *reinterpret_cast<const float4*>(&" << arr << sb << so
             << "u]);\n    c2 " << reg << j << " = {" << reg << "q" << j << ".x, " << reg << "q" << j << ".y}, " << reg << j2
             << " = {" << reg << "q" << j << ".z, " << reg << "q" << j << ".w};\n";
        continue;
      }
      if (store) s_ << "    " << arr << sb << so << "u] = " << reg << j << ";\n";
      else s_ << "    c2 " << reg << j << " = " << arr << sb << so << "u];\n";
    }
  }

  // the op's parity over the members: bit i the parity of f on vector i
  int reg_parity(uint32_t f) const {
    int fr = 0;
    for (int i = 0; i < r_.M; i++) fr |= parity32(f & gu_[i]) << i;
    return fr;
  }
  int reg_mask(uint32_t m) const {  // members j, j ^ mask pair up under m
    for (int j = 1; j < N_; j++) {
      uint32_t g = 0;
      for (int i = 0; i < r_.M; i++)
        if ((j >> i) & 1) g ^= gu_[i];
      if (g == m) return j;
    }
    return 0;
  }
  // the part of the parity that the group shares
  Sign group_sign(uint32_t f, int b) {
    Sign g;
    g.c = b != 0;
    bool moves = (f & ~t_.pivots & (P_.n >= 32 ? ~0u : (1u << P_.n) - 1u)) != 0;
    for (int pos : r_.grp_pos) moves = moves || parity32(f & t_.v[pos]);
    if (!moves) return g;
    const uint32_t m = f & varying_;
    auto it = words_.find(m);
    if (it == words_.end()) {
      it = words_.emplace(m, (int)words_.size()).first;
      s_ << "    const uint32_t w" << it->second << " = ";
      if ((m & (m - 1u)) == 0) {
        int p = 0;
        while (!((m >> p) & 1u)) p++;
        s_ << "(y0 << " << 31 - p << ") & 0x80000000u;\n";
      } else {
        s_ << "(uint32_t)__popc(y0 & " << m << "u) << 31;\n";
      }
    }
    g.w.push_back(it->second);
    return g;
  }

  // order of execution: gates as early as they commute ahead, phases gathered
  void plan() {
    std::vector<int> todo = r_.ops;
    if (rev_) std::reverse(todo.begin(), todo.end());
    items_.clear();
    while (!todo.empty()) {
      int pick = -1;
      for (size_t i = 0; i < todo.size() && pick < 0; i++) {
        if (P_.ops[todo[i]].kind == L_PHASE) continue;
        bool ok = true;
        for (size_t j = 0; j < i && ok; j++) ok = lin_commute(P_.ops[todo[i]], P_.ops[todo[j]]);
        if (ok) pick = (int)i;
      }
      if (pick >= 0) {
        items_.push_back({todo[pick]});
        todo.erase(todo.begin() + pick);
        continue;
      }
      std::vector<int> blk, left;
      for (int o : todo) {
        bool ok = P_.ops[o].kind == L_PHASE;
        for (size_t j = 0; j < left.size() && ok; j++) ok = lin_commute(P_.ops[o], P_.ops[left[j]]);
        (ok ? blk : left).push_back(o);
      }
      items_.push_back(blk);
      todo.swap(left);
    }
  }

  std::string mat(int o) const { return "mats[" + std::to_string(P_.coef[o]) + "]"; }

  // sign words of every op, the group factor G (scale, shared phases, shared
  // signs) and the block it is merged into
  void prelude() {
    complex_factor_ = false;
    bool signs = false;
    std::vector<std::string> phase, flips;
    for (int o : r_.ops) {
      const LinOp& g = P_.ops[o];
      const Sign a = group_sign(g.f, g.b);
      if (g.kind == L_PHASE) {
        // e^{-+i a/2} by the shared sign (conjugate in reverse); constant
        // ones are a global phase, kept for exact programs only
        Sign sg = a;
        sg.c = sg.c == rev_;  // forward, sign 0: (cos, -sin)
        if (!a.constant() || P_.exact)
          phase.push_back("    { const float4 q = " + mat(o) + "; G = cmul(G, {q.x, sx(q.y, " + sg.str() + ")}); }\n");
        if (g.p && P_.exact) phase.push_back("    { const float4 q = " + mat(o) + "; G = cmul(G, {q.x, q.y}); }\n");
      } else if (g.kind == L_CZ) {
        const Sign b = group_sign(g.f2, g.b2);
        if (!a.zero() && !b.zero() && (P_.exact || !a.constant() || !b.constant())) {
          flips.push_back("    gs ^= (" + a.str() + ") & (" + b.str() + ");\n");
          signs = true;
        }
      } else if (g.kind == L_SIGN) {
        if (!a.zero() && (P_.exact || !a.constant())) {
          flips.push_back("    gs ^= " + a.str() + ";\n");
          signs = true;
        }
      }
    }
    // exact programs' rotations of the second form leave their sign to the
    // group factor; their words need the frame at that point, so it is walked
    // here first
    std::vector<Frame> fr;
    for (const std::vector<int>& it : items_) {
      const LinOp& g = P_.ops[it[0]];
      if (g.kind == L_PHASE) {
        std::vector<int> basis;
        std::vector<int> frs;
        for (int o : it) frs.push_back(reg_parity(P_.ops[o].f));
        absorb(frs, fr, nullptr);
        continue;
      }
      if (!g.m) {
        add_frames(g, fr);
        continue;
      }
      const int mj = reg_mask(g.m);
      if (g.kind == L_H) {
        drop_hit(fr, mj, nullptr);
        continue;
      }
      if (!P_.exact) continue;  // one form only
      Sign sg = frame_sign(fr, mj);
      if (g.kind == L_RY) sg.flip(group_sign(g.f, g.b));
      if (!sg.zero() && (P_.exact || !sg.constant())) {
        flips.push_back("    gs ^= __float_as_uint(" + mat(it[0]) + ".w) & (" + sg.str() + ");\n");
        signs = true;
      }
    }
    merge_ = -1;
    size_t big = 0;
    group_factor_ = r_.norm >= 0 || !phase.empty() || signs;
    if (group_factor_)
      for (size_t i = 0; i < items_.size(); i++)
        if (P_.ops[items_[i][0]].kind == L_PHASE && items_[i].size() > big) {
          big = items_[i].size();
          merge_ = (int)i;
        }
    complex_factor_ = !phase.empty() || P_.exact;
    if (!group_factor_) return;
    if (r_.norm >= 0) s_ << "    const float4 nrm = mats[" << r_.norm << "];\n";
    s_ << "    uint32_t gs = 0u;\n";
    for (const std::string& f : flips) s_ << f;
    s_ << "    c2 G = {sx(" << (r_.norm >= 0 ? "nrm.x" : "1.f") << ", gs), "
       << (r_.norm >= 0 && P_.exact ? "sx(nrm.y, gs)" : "0.f") << "};\n";
    for (const std::string& f : phase) s_ << f;
    if (rev_ && r_.norm >= 0) s_ << "    float sc = 1.f;\n";
  }

  Sign frame_sign(const std::vector<Frame>& fr, int mj) const {
    Sign s;
    for (const Frame& f : fr)
      if (cpar(f.fr & mj)) s.flip(f.sign);
    return s;
  }

  static void push_frame(std::vector<Frame>& fr, int bits, const Sign& sign) {
    if (!bits || sign.zero()) return;
    for (size_t i = 0; i < fr.size(); i++)
      if (fr[i].fr == bits) {
        fr[i].sign.flip(sign);
        if (fr[i].sign.zero()) fr.erase(fr.begin() + i);
        return;
      }
    fr.push_back({bits, sign});
  }

  // the frame signs of CZ and SIGN ops (their member-wise product of two
  // register parities is applied by gate())
  void add_frames(const LinOp& g, std::vector<Frame>& fr) {
    const int f0 = reg_parity(g.f);
    Sign one;
    one.c = true;
    if (g.kind == L_SIGN) {
      push_frame(fr, f0, one);
      return;
    }
    const int f1 = reg_parity(g.f2);
    push_frame(fr, f0, group_sign(g.f2, g.b2));
    push_frame(fr, f1, group_sign(g.f, g.b));
  }

  template <class Emit>
  static void drop_frames(std::vector<Frame>& fr, const std::vector<char>& drop, Emit emit) {
    std::vector<Frame> keep;
    for (size_t i = 0; i < fr.size(); i++) {
      if (drop[i]) emit(fr[i]);
      else keep.push_back(fr[i]);
    }
    fr.swap(keep);
  }

  // frames that anticommute with a pairing mask, taken out (applied if `self`)
  void drop_hit(std::vector<Frame>& fr, int mj, PassWriter* self) {
    std::vector<char> d;
    for (const Frame& f : fr) d.push_back((char)cpar(f.fr & mj));
    drop_frames(fr, d, [&](const Frame& f) {
      if (self) self->flush(f);
    });
  }

  // frames in the span of a block's parities, taken out into `out`
  static void absorb(const std::vector<int>& frs, std::vector<Frame>& fr, std::vector<Frame>* out) {
    std::vector<int> basis;
    for (int f : frs)
      if (f) add_basis(basis, f);
    std::vector<char> d;
    for (const Frame& f : fr) d.push_back((char)(combo(basis, f.fr) >= 0));
    drop_frames(fr, d, [&](const Frame& f) {
      if (out) out->push_back(f);
    });
  }

  static bool add_basis(std::vector<int>& basis, int f) {
    if (combo(basis, f) >= 0) return false;
    basis.push_back(f);
    return true;
  }
  // f as an XOR of basis vectors (bit i: vector i), or -1
  static int combo(const std::vector<int>& basis, int f) {
    for (int c = 0; c < (1 << basis.size()); c++) {
      int x = 0;
      for (size_t i = 0; i < basis.size(); i++)
        if ((c >> i) & 1) x ^= basis[i];
      if (x == f) return c;
    }
    return -1;
  }

  void flush(const Frame& f) {
    for (const char* g : regs_)
      for (int j = 0; j < N_; j++)
        if (cpar(f.fr & j)) s_ << "    lin_neg(" << g << j << ", " << f.sign.str() << ");\n";
  }

  template <class Share>
  void gate(int o, Share share) {
    const LinOp& g = P_.ops[o];
    if (!g.m) {
      if (g.kind == L_CZ) {
        const int f0 = reg_parity(g.f), f1 = reg_parity(g.f2);
        for (const char* a : regs_)
          for (int j = 0; j < N_; j++)
            if (cpar(f0 & j) && cpar(f1 & j)) s_ << "    lin_neg(" << a << j << ", 0x80000000u);\n";
      }
      add_frames(g, frame_);
      return;
    }
    const int mj = reg_mask(g.m), fr = reg_parity(g.f);
    if (g.kind == L_H) {
      drop_hit(frame_, mj, this);
      s_ << "    {\n    const float2 hs = bc2(sx(1.f, " << group_sign(g.f, g.b).str() << ")), hn = bc2(-hs.x);\n";
      for (const char* a : regs_)
        pairs(mj, fr, [&](int j, int k) { s_ << "    h_pair(" << a << j << ", " << a << k << ", hs, hn);\n"; });
      s_ << "    }\n";
      if (rev_ && r_.norm >= 0) s_ << "    sc *= 0.70710678118654752f;\n";
      return;
    }
    Sign sg = frame_sign(frame_, mj);
    if (g.kind == L_RY) sg.flip(group_sign(g.f, g.b));
    s_ << "    {\n    const float4 q = " << mat(o) << ";\n";
    const std::string dst = rev_ ? share(o) : "";
    const bool ry = g.kind == L_RY;
    if (!dst.empty()) {
      const char* type = ry ? "float2" : "float";
      const char* zero = ry ? "make_float2(0.f, 0.f)" : "0.f";
      s_ << "    " << type << " gp = " << zero << ", gn = " << zero << ";\n";
      pairs(mj, ry ? fr : mj & -mj, [&](int j, int k) {
        s_ << "    dot_" << (ry ? "y" : "x") << "(p" << j << ", p" << k << ", l" << j << ", l" << k << ", gp, gn);\n";
      });
      s_ << "    lin_share(" << dst << ", sx(sc * sc * (" << (ry ? "(gp.x + gp.y) - (gn.x + gn.y)" : "gp - gn") << "), " << sg.str()
         << " ^ __float_as_uint(q.w)));\n";
    }
    if (rev_) {
      Sign inv;
      inv.c = true;
      sg.flip(inv);
    }
    s_ << "    const float v = sx(q.x, " << sg.str() << ");\n" << (P_.exact ? "    if (__float_as_uint(q.w) == 0u) {\n" : "");
    if (ry) s_ << "    const float2 t = bc2(v), nt = bc2(-v);\n";
    for (const char* a : regs_)
      pairs(mj, ry ? fr : mj & -mj, [&](int j, int k) {
        s_ << "    " << (ry ? "ry_t(" : "rx_t(") << a << j << ", " << a << k << (ry ? ", t, nt);\n" : ", v);\n");
      });
    if (P_.exact) {
      s_ << "    } else {\n";
      for (const char* a : regs_)
        pairs(mj, ry ? fr : mj & -mj, [&](int j, int k) {
          s_ << "    " << (ry ? "ry_u(" : "rx_u(") << a << j << ", " << a << k << ", v);\n";
        });
      s_ << "    }\n";
    }
    if (rev_ && r_.norm >= 0) s_ << "    sc *= q.y;\n";
    s_ << "    }\n";
  }

  // f(j, j ^ mj) over the members of even parity fr
  template <class F>
  void pairs(int mj, int fr, F f) {
    for (int j = 0; j < N_; j++)
      if (!cpar(fr & j)) f(j, j ^ mj);
  }

  // a block of phases (see the class comment); merge: G multiplies every member
  template <class Share>
  void block(const std::vector<int>& ops, bool merge, Share share) {
    s_ << "    {\n";
    // gradient shares: Im(conj(l) p) summed per class of up to three parities
    std::vector<int> withg;
    if (rev_)
      for (int o : ops)
        if (!share(o).empty()) withg.push_back(o);
    for (size_t c0 = 0; c0 < withg.size(); c0 += 3) {
      const size_t c1 = std::min(withg.size(), c0 + 3);
      std::vector<int> basis;
      for (size_t i = c0; i < c1; i++)
        if (int f = reg_parity(P_.ops[withg[i]].f)) add_basis(basis, f);
      const int nc = 1 << basis.size();
      s_ << "    {\n";
      for (int c = 0; c < nc; c++) s_ << (c ? ", v" : "    float v") << c << " = 0.f";
      s_ << ";\n";
      for (int j = 0; j < N_; j++) {
        int cls = 0;
        for (size_t i = 0; i < basis.size(); i++) cls |= cpar(basis[i] & j) << i;
        s_ << "    v" << cls << " = lin_im(l" << j << ", p" << j << ", v" << cls << ");\n";
      }
      for (size_t i = c0; i < c1; i++) {
        const LinOp& g = P_.ops[withg[i]];
        const int cm = combo(basis, reg_parity(g.f));
        s_ << "    lin_share(" << share(withg[i]) << ", sx(" << (r_.norm >= 0 ? "sc * sc * (" : "(");
        for (int c = 0; c < nc; c++) s_ << (cpar(cm & c) ? " - " : c ? " + " : "") << "v" << c;
        // (the angle's sign in the row's frame; without rotations there is no frame)
        s_ << "), " << group_sign(g.f, g.b).str();
        if (!P_.rot.empty()) s_ << " ^ sig[" << P_.coef[withg[i]] << "]";
        s_ << "));\n";
      }
      s_ << "    }\n";
    }
    // phases per register parity, in class space
    std::vector<int> frs, basis;
    for (int o : ops) frs.push_back(reg_parity(P_.ops[o].f));
    std::vector<Frame> signs;
    absorb(frs, frame_, &signs);
    for (int f : frs)
      if (f) add_basis(basis, f);
    struct Elem {
      int cm;
      std::string name;  // phase, or ""
      Sign sign;
    };
    std::vector<Elem> el;
    for (size_t i = 0; i < ops.size(); i++) {
      if (!frs[i]) continue;  // shared by the group: in G
      const LinOp& g = P_.ops[ops[i]];
      Sign sg = group_sign(g.f, g.b);
      if (rev_) sg.c = !sg.c;
      const std::string nm = "h" + std::to_string(i);
      s_ << "    const c2 " << nm << " = {" << mat(ops[i]) << ".z, sx(" << mat(ops[i]) << ".w, " << sg.str() << ")};\n";
      el.push_back({combo(basis, frs[i]), nm, Sign()});
    }
    for (const Frame& f : signs) el.push_back({combo(basis, f.fr), "", f.sign});
    int tmp = 0;
    classes(basis, el, 0, 0, merge ? "G" : "", &tmp, merge);
    if (merge && rev_ && r_.norm >= 0) s_ << "    sc *= nrm.z;\n";
    s_ << "    }\n";
  }

  template <class Elem>
  void classes(const std::vector<int>& basis, const std::vector<Elem>& el, size_t i, int cls, std::string ph, int* tmp,
               bool merge) {
    if (i < basis.size()) {
      classes(basis, el, i + 1, cls, ph, tmp, merge);
      for (const Elem& e : el)
        if (e.cm == (1 << i) && !e.name.empty()) ph = times(ph, e.name, tmp);
      classes(basis, el, i + 1, cls | (1 << i), ph, tmp, merge);
      return;
    }
    Sign sg;
    for (const Elem& e : el) {
      if (!cpar(e.cm & cls)) continue;
      if (e.name.empty()) sg.flip(e.sign);
      else if (e.cm & (e.cm - 1)) ph = times(ph, e.name, tmp);
    }
    if (!ph.empty() && !sg.zero()) {
      const std::string nm = "t" + std::to_string((*tmp)++);
      s_ << "    c2 " << nm << " = " << ph << ";\n    lin_neg(" << nm << ", " << sg.str() << ");\n";
      ph = nm;
    }
    for (const char* g : regs_)
      for (int j = 0; j < N_; j++) {
        int c = 0;
        for (size_t b = 0; b < basis.size(); b++) c |= cpar(basis[b] & j) << b;
        if (c != cls) continue;
        if (!ph.empty()) s_ << "    lin_mul(" << g << j << ", " << ph << ");\n";
        else if (!sg.zero()) s_ << "    lin_neg(" << g << j << ", " << sg.str() << ");\n";
      }
  }

  std::string times(const std::string& a, const std::string& b, int* tmp) {
    if (a.empty()) return b;
    const std::string nm = "t" + std::to_string((*tmp)++);
    s_ << "    const c2 " << nm << " = cmul(" << a << ", " << b << ");\n";
    return nm;
  }

  Text& s_;
  const LinProgram& P_;
  const LinTile& t_;
  const LinReg& r_;
  const bool rev_;
  const int N_;
  uint32_t gu_[4];        // the pass's vectors as index masks
  uint32_t varying_ = 0;  // index bits that the group base can have
  std::map<uint32_t, int> words_;
  std::vector<std::vector<int>> items_;
  std::vector<Frame> frame_;
  std::vector<const char*> regs_;
  bool group_factor_ = false, complex_factor_ = false;
  int merge_ = -1;
};

// The index of a group's first member: its tile's base XOR its local index
// through the tile's vectors (whole states: the local index).
std::string group_index(const LinProgram& P, const LinTile& t, int L) {
  if (t.k == P.n) return "gb";
  const std::string low = std::to_string((1u << L) - 1u);
  return "base ^ (gb & " + low + "u) ^ (uint32_t)s.off[gb >> " + std::to_string(L) + "]";
}

void emit_fwd_pass(Text& s, const LinProgram& P, const LinTile& t, const LinReg& r, int L, int nthreads) {
  s << "  {\n";
  PassWriter(s, P, t, r, false).write(nthreads, group_index(P, t, L), {"psi"}, {"a"}, [](int) { return std::string(); });
  s << "  }\n  __syncthreads();\n";
}

// One reverse register pass: gradient shares go to accumulator index
// acc_index(op) of the per-warp rows gpart[warp * stride + index], reduced
// over the warp for up to 32 accumulators at once (grad_share_multi; their
// index tables are declared into `decl`).
template <class F>
void emit_rev_pass(Text& s, Text& decl, int* uid, const LinProgram& P, const LinTile& t,
                   const LinReg& r, int L, int nthreads, int stride, F acc_index) {
  // The pass's gradient shares, summed per accumulator index in registers
  // gs<chunk>[position] (a chunk holds at most 32 distinct indices; shares of
  // gates that use one parameter add into one register), then reduced over
  // the warp a chunk at a time by grad_share_multi, whose K lanes add to
  // gpart[warp * stride + table[j]] in one instruction (a read-add-write of
  // shared memory): no table may hold an index twice, or two lanes would read
  // the same old value and one addition would be lost.  A chunk of g indices
  // is padded to K = 2^ceil(log2 g) with indices the chunk does not use (the
  // padding lanes add zero there); if fewer than K - g are free, it is cut
  // into power-of-two chunks instead.
  std::vector<int> distinct;
  for (int o : r.ops)
    if (P.ops[o].slot >= 0) {
      const int idx = acc_index(o);
      if (std::find(distinct.begin(), distinct.end(), idx) == distinct.end()) distinct.push_back(idx);
    }
  std::vector<std::vector<int>> chunks;
  std::map<int, std::pair<int, int>> place;  // accumulator index -> chunk, position
  for (size_t at = 0; at < distinct.size();) {
    const int g = (int)std::min<size_t>(32, distinct.size() - at);
    int kk = 1;
    while (kk < g) kk <<= 1;
    if (kk > stride) kk >>= 1;  // too few free indices: the largest power of two below g
    const int take = std::min(kk, g);
    for (int i = 0; i < take; i++) place[distinct[at + i]] = {(int)chunks.size(), i};
    chunks.emplace_back(distinct.begin() + at, distinct.begin() + at + take);
    std::vector<int>& ch = chunks.back();
    // padding: the lowest accumulator indices the chunk does not use
    for (int cand = 0; (int)ch.size() < kk && cand < stride; cand++)
      if (std::find(ch.begin(), ch.end(), cand) == ch.end()) ch.push_back(cand);
    at += take;
  }
  s << "  {\n";
  for (size_t c = 0; c < chunks.size(); c++) {
    s << "  float gs" << c << "[" << chunks[c].size() << "] = {";
    for (size_t j = 0; j < chunks[c].size(); j++) s << (j ? ", " : "") << "0.f";
    s << "};\n";
  }
  PassWriter(s, P, t, r, true)
      .write(nthreads, group_index(P, t, L), {"psi", "lam"}, {"p", "l"}, [&](int o) {
        if (P.ops[o].slot < 0) return std::string();
        const auto& at = place.at(acc_index(o));
        return "gs" + std::to_string(at.first) + "[" + std::to_string(at.second) + "]";
      });
  for (size_t c = 0; c < chunks.size(); c++) {
    const int id = (*uid)++;
    decl << "__constant__ int tdq_gi_" << id << "[" << chunks[c].size() << "] = {";
    for (size_t j = 0; j < chunks[c].size(); j++) decl << (j ? ", " : "") << chunks[c][j];
    decl << "};\n";
    s << "  grad_share_multi<" << chunks[c].size() << ">(gpart, " << stride << ", tdq_gi_" << id << ", gs" << c << ");\n";
  }
  s << "  __syncthreads();\n  }\n";
}

}  // namespace

// The program struct `sname` of one circuit; constant tables go to decl,
// numbered from *uid.
static void k2_prog_struct(Text& s, Text& decl, int* uid, const LinProgram& P, int nparams,
                           int nthreads, bool grad, const std::string& sname) {
  const LinTile& t = P.tiles[0];
  s << "struct " << sname << " {\n"
    << "  static constexpr bool kSpecialised = true;\n  using Mat = float4;\n  const DOp* dops;\n";
  s << "  template <int MF>\n  __device__ __forceinline__ void forward(c2* psi, const float4* mats, int) const {\n";
  for (size_t pi = 0; pi < t.fwd.size(); pi++) {
    s << "  // forward pass " << pi << "\n";
    emit_fwd_pass(s, P, t, t.fwd[pi], 0, nthreads);
  }
  s << "  }\n";
  s << "  template <int MB>\n  __device__ __forceinline__ void reverse(c2* psi, c2* lam, const float4* mats, int, "
       "double*, float* gpart) const {\n  const uint32_t* sig = reinterpret_cast<const uint32_t*>(mats + "
    << t.coef.size() << ");\n  (void)sig;\n";
  if (grad)
    for (int pi = (int)t.rev.size() - 1; pi >= 0; pi--) {
      s << "  // reverse pass " << pi << "\n";
      emit_rev_pass(s, decl, uid, P, t, t.rev[pi], 0, nthreads, nparams, [&](int o) { return P.ops[o].slot; });
    }
  s << "  }\n};\n";
}

std::string k2_specialised_source(const LinProgram& prog, bool grad, int nthreads, int nparams, const char* name,
                                  bool fine) {
  Text s, decl;
  int uid = 0;
  k2_prog_struct(s, decl, &uid, prog, nparams, nthreads, grad, "SpecProg");
  s << "}  // namespace tdq\n";
  Text out;
  out << "#include \"k2_body.cuh\"\nnamespace tdq {\n" << decl.str() << s.str();
  const int minb = nthreads >= 256 ? 2 : 1;
  out << "extern \"C\" __global__ void __launch_bounds__(" << nthreads << ", " << minb << ") " << name
    << "(tdq::SweepArgs a, const tdq::DOp* gdops, int ndops, const int* rec_ptr, const int* rec_ops, int nrec) {\n"
    << (fine ? "  if (a.fine_rows && (int)blockIdx.x >= a.fine_rows) {\n"
               "    const int f = (int)blockIdx.x - a.fine_rows - tdq::kFineGap;\n"
               "    if (f >= 0) tdq::k2_fine_row(a, f);\n    return;\n  }\n"
             : "")
    << "  tdq::k2_body<0, 0, " << (grad ? "true" : "false")
    << ", tdq::SpecProg>(a, tdq::SpecProg{nullptr}, gdops, 0, rec_ptr, rec_ops, nrec, blockIdx.x);\n}\n";
  return out.str();
}

std::vector<std::string> k2_multi_modules(const std::vector<K2Part>& parts, bool grad, int nthreads,
                                          const char* name) {
  std::vector<std::string> mods(1);
  int uid = 0;  // constant tables numbered across modules: their names stay unique at link time
  for (size_t c = 0; c < parts.size(); c++) {
    Text s, decl;
    k2_prog_struct(s, decl, &uid, *parts[c].prog, parts[c].P, nthreads, grad, "SpecProg_" + std::to_string(c));
    Text out;
    out << "#include \"k2_body.cuh\"\nnamespace tdq {\n" << decl.str() << s.str() << "}  // namespace tdq\n";
    // the circuit's row body: a function of its own, linked to the launch module
    out << "__device__ __noinline__ void tdq_multi_row_" << c
        << "(const tdq::SweepArgs& a, const tdq::MultiCirc& m, int r) {\n  tdq::k2_body<0, 0, "
        << (grad ? "true" : "false") << ", tdq::SpecProg_" << c << ">(a, tdq::SpecProg_"
        << c << "{nullptr}, nullptr, 0, m.rec_ptr, m.rec_ops, m.nrec, r);\n}\n";
    mods.push_back(out.str());
  }
  Text out;
  out << "#include \"sweep_common.cuh\"\n";
  for (size_t c = 0; c < parts.size(); c++)
    out << "__device__ void tdq_multi_row_" << c << "(const tdq::SweepArgs& a, const tdq::MultiCirc& m, int r);\n";
  // persistent CTAs take (circuit, row) items from a counter until none is left
  out << "extern \"C\" __global__ void __launch_bounds__(" << nthreads << ", 1) " << name
      << "(const tdq::MultiCirc* __restrict__ mc, const int2* __restrict__ items, int n_items, int* next,\n"
      << "    const float* params, const float* inputs, double* values, const double* gw, float* grads) {\n"
      << "  __shared__ int s_item;\n"
      << "  for (;;) {\n"
      << "    __syncthreads();\n"
      << "    if (threadIdx.x == 0) s_item = atomicAdd(next, 1);\n"
      << "    __syncthreads();\n"
      << "    const int it = s_item;\n"
      << "    if (it >= n_items) return;\n"
      << "    const int2 w = items[it];\n"
      << "    const tdq::MultiCirc& m = mc[w.x];\n"
      << "    tdq::SweepArgs a = m.a;\n"
      << "    a.params = params + m.p_off;\n"
      << "    a.inputs = inputs ? inputs + m.x_off : nullptr;\n"
      << "    a.values = values + m.v_off;\n"
      << "    a.gw = gw ? gw + m.v_off : nullptr;\n"
      << "    a.grads = grads ? grads + m.g_off : nullptr;\n"
      << "    switch (w.x) {\n";
  for (size_t c = 0; c < parts.size(); c++)
    out << "      case " << c << ": tdq_multi_row_" << c << "(a, m, w.y); break;\n";
  out << "      default: break;\n    }\n  }\n}\n";
  mods[0] = out.str();
  return mods;
}

// pairs(f): f(shared-memory slot, global index) for this thread's pairs of
// neighbours of a tile (both even; see swz_pair), every(f) for its elements.
// A thread's local indices are 2 (tid + NT i): the part of both indices that
// tid gives is computed once per tile, the rest are constants.
static void emit_every(Text& s, const LinTile& t, int L) {
  s << "  template <int NT, class F>\n  __device__ __forceinline__ static void pairs(const TiledDev&, const TileShared& s, "
       "uint32_t base, F&& f) {\n"
    << "    constexpr uint32_t v[" << t.k << "] = {";
  for (int i = 0; i < t.k; i++) s << (i ? ", " : "") << t.v[i] << "u";
  s << "};\n    const uint32_t j = 2u * threadIdx.x;\n    if (2 * NT > " << (1 << t.k) << " && j >= " << (1 << t.k)
    << "u) return;\n"
    << "    const uint32_t y = base ^ (j & " << (1u << L) - 1u << "u) ^ (uint32_t)s.off[j >> " << L
    << "], z = swz_pair(j);\n"
    << "#pragma unroll\n    for (uint32_t i = 0; i < " << (1 << t.k) << "u; i += 2 * NT) {\n"
    << "      uint32_t x = 0;\n#pragma unroll\n      for (int q = 0; q < " << t.k
    << "; q++) x ^= ((i >> q) & 1u) ? v[q] : 0u;\n"
    << "      f(z ^ swz_pair(i), y ^ x);\n    }\n  }\n"
    << "  template <int NT, class F>\n  __device__ __forceinline__ static void every(const TiledDev& t, const TileShared& s, "
       "uint32_t base, F&& f) {\n    pairs<NT>(t, s, base, [&](uint32_t j, uint32_t x) {\n      f(j, x);\n"
       "      f(j | 1u, x | 1u);\n    });\n  }\n";
}

// in_first(x): whether index x lies in the first pass's space (the remainder
// of x by the space's basis is zero).
static void emit_in_first(Text& s, const LinTile& t, int n) {
  const uint32_t out = (n >= 32 ? ~0u : (1u << n) - 1u) & ~t.pivots;
  s << "  __device__ __forceinline__ static bool in_first(uint32_t x) {\n    uint32_t r = x & " << out << "u;\n";
  for (uint32_t v : t.v) {
    if (!(v & out)) continue;
    int p = 0;
    while (!((v & t.pivots) >> p & 1u)) p++;
    s << "    if ((x >> " << p << ") & 1u) r ^= " << (v & out) << "u;\n";
  }
  s << "    return r == 0u;\n  }\n";
}

std::string k1_specialised_source(const TiledSweep& t, const LinProgram& prog, int nthreads_r, int only) {
  Text s, decl;
  int uid = 0;
  const int np = (int)prog.tiles.size();
  for (int p = 0; p < np; p++) {
    if (only >= 0 && p != only) continue;
    const LinTile& tile = prog.tiles[p];
    const int nthreads = t.threads_f[p];
    // gradient accumulators of the pass: one per angle with a slot
    std::map<int, int> acc;
    std::vector<int> slots;
    if (t.adj)
      for (int o : tile.ops)
        if (prog.ops[o].slot >= 0) {
          acc[o] = (int)slots.size();
          slots.push_back(prog.ops[o].slot);
        }
    const int na = std::max(1, (int)slots.size());
    s << "__constant__ int tdq_slots_" << p << "[" << na << "] = {";
    for (int i = 0; i < na; i++) s << (i ? ", " : "") << (i < (int)slots.size() ? slots[i] : 0);
    s << "};\n";
    s << "struct TilePass" << p << " {\n  static constexpr bool kSpecialised = true, kFirst = "
      << (p == 0 ? "true" : "false") << ", kSecond = " << (p == 1 ? "true" : "false") << ", kDiag = "
      << (t.diag ? "true" : "false") << ";\n  static constexpr int kK = " << t.k << ", kN = " << t.n
      << ", kBuffers = " << (t.dbl && nthreads == t.nthreads ? 2 : 1) << ", kGroups = " << t.ng << ";\n";
    emit_in_first(s, prog.tiles[0], t.n);
    emit_every(s, tile, t.L);
    s << "  __device__ __forceinline__ static void forward(const TiledDev&, const TileShared& s, uint32_t base, "
         "uint32_t buf) {\n"
      << "  c2* psi = s.psi;\n  const float4* mats = reinterpret_cast<const float4*>(s.mats);\n";
    for (const LinReg& r : tile.fwd) emit_fwd_pass(s, prog, tile, r, t.L, nthreads);
    s << "  }\n";
    s << "  __device__ __forceinline__ static void reverse(const TiledDev&, const TileShared& s, uint32_t base, "
         "uint32_t buf) {\n"
      << "  c2* psi = s.psi;\n  c2* lam = s.lam;\n  const float4* mats = reinterpret_cast<const float4*>(s.mats);\n"
      << "  float* gpart = reinterpret_cast<float*>(s.gpart);\n"
      << "  const uint32_t* sig = reinterpret_cast<const uint32_t*>(mats + " << tile.coef.size()
      << ");\n  (void)sig;\n";
    // (the fused last pass runs its reverse program with the forward kernel's threads)
    for (int q = (int)tile.rev.size() - 1; q >= 0; q--)
      emit_rev_pass(s, decl, &uid, prog, tile, tile.rev[q], t.L, p == np - 1 ? nthreads : nthreads_r, na,
                    [&](int o) { return acc.at(o); });
    s << "  }\n";
    s << "  __device__ __forceinline__ static void flush(const SweepArgs& a, const TiledDev& t, const TileShared& s, "
         "int lr) {\n"
      << "  __syncthreads();\n  const float* gp = reinterpret_cast<const float*>(s.gpart);\n"
      << "  const int nw = blockDim.x >> 5;\n"
      << "  for (int i = threadIdx.x; i < " << (int)slots.size() << "; i += blockDim.x) {\n"
      << "    double v = 0.0;\n    for (int w = 0; w < nw; w++) v += (double)gp[w * " << na << " + i];\n"
      << "    atomicAdd(&t.gacc[(int64_t)lr * a.P + tdq_slots_" << p << "[i]], v);\n  }\n  }\n};\n";
  }
  s << "}  // namespace tdq\n";
  Text out;
  out << "#include \"k1_body.cuh\"\nnamespace tdq {\n" << decl.str() << s.str();
  for (int p = 0; p < np; p++) {
    if (only >= 0 && p != only) continue;
    const bool f = p == 0, l = p == np - 1;
    const int nthreads = t.threads_f[p];
    const int minb = nthreads < t.nthreads ? (l && t.adj ? 3 : 4) : nthreads >= 256 ? 2 : 1;
    out << "extern \"C\" __global__ void __launch_bounds__(" << nthreads << ", " << minb << ") tdq_k1f_" << p
      << "(tdq::SweepArgs a, tdq::TiledDev t, int store) {\n  tdq::k1_forward_body<" << nthreads << ", "
      << (f ? "true" : "false") << ", " << (l ? "true" : "false") << ", " << ((l && t.adj) ? "true" : "false")
      << ", tdq::TilePass" << p
      << ">(a, t, store);\n}\n";
    if (t.adj && !l)
      out << "extern \"C\" __global__ void __launch_bounds__(" << nthreads_r << ", " << (nthreads_r <= 256 ? 2 : 1)
          << ") tdq_k1r_" << p
        << "(tdq::SweepArgs a, tdq::TiledDev t) {\n  tdq::k1_reverse_body<" << nthreads_r << ", tdq::TilePass" << p << ">(a, t);\n}\n";
  }
  return out.str();
}

namespace {

struct JitCache {
  std::mutex mu;
  std::map<std::string, cudaLibrary_t> libs;  // by key
};

JitCache& cache() {
  static JitCache* c = new JitCache();  // never destroyed: kernels outlive static teardown order
  return *c;
}

std::string nvrtc_log(nvrtcProgram p) {
  size_t n = 0;
  if (nvrtcGetProgramLogSize(p, &n) != NVRTC_SUCCESS || n == 0) return "";
  std::string log(n, '\0');
  nvrtcGetProgramLog(p, &log[0]);
  return log;
}

}  // namespace

JitCode k2_code(const LinProgram& prog, bool grad, int nthreads, int nparams, const char* name, bool fine) {
  std::string key = "k2";
  for (int v : {(int)grad, nthreads, nparams, (int)fine}) key += ' ' + std::to_string(v);
  return {key + name + lin_key(prog), [=, &prog] {
            return std::vector<std::string>{k2_specialised_source(prog, grad, nthreads, nparams, name, fine)};
          }};
}

JitCode k1_code(const TiledSweep& t, const LinProgram& prog, int nthreads_r, int pass) {
  std::string key = "k1";
  for (int v : {t.n, t.k, t.L, (int)t.adj, (int)t.diag, t.ng, t.dbl, t.nthreads, t.threads_f[pass], nthreads_r, pass})
    key += ' ' + std::to_string(v);
  return {key + lin_key(prog), [=, &t, &prog] {
            return std::vector<std::string>{k1_specialised_source(t, prog, nthreads_r, pass)};
          }};
}

bool jit_cached(const JitCode& code) {
  JitCache& C = cache();
  std::lock_guard<std::mutex> lk(C.mu);
  return C.libs.count(code.key) > 0;
}

tdq_status jit_kernel(const JitCode& code, const char* name, const void** kernel) {
  *kernel = nullptr;
  int dev = 0;
  TDQ_CUDA_TRY(cudaGetDevice(&dev));
  int maj = 0, min = 0;
  TDQ_CUDA_TRY(cudaDeviceGetAttribute(&maj, cudaDevAttrComputeCapabilityMajor, dev));
  TDQ_CUDA_TRY(cudaDeviceGetAttribute(&min, cudaDevAttrComputeCapabilityMinor, dev));
  if (maj != 10 || min != 3)
    return fail(TDQ_ERR_UNSUPPORTED, "specialised sweep: built for sm_103a, device is sm_" +
                                         std::to_string(maj) + std::to_string(min));
  // one compilation per key, all its kernels; NVRTC runs outside the lock
  // so that different sources compile concurrently
  JitCache& C = cache();
  cudaLibrary_t lib = nullptr;
  {
    std::lock_guard<std::mutex> lk(C.mu);
    auto it = C.libs.find(code.key);
    if (it != C.libs.end()) lib = it->second;
  }
  if (!lib) {
    const std::string src = code.modules()[0];
    nvrtcProgram p;
    if (nvrtcCreateProgram(&p, src.c_str(), "tdq_specialised.cu", kJitHeaderCount, kJitHeaderSrc,
                           kJitHeaderNames) != NVRTC_SUCCESS)
      return fail(TDQ_ERR_CUDA, "specialised sweep: nvrtcCreateProgram failed");
    const char* opts[] = {"-arch=sm_103a", "-std=c++17", "-default-device", "-lineinfo"};
    const nvrtcResult r = nvrtcCompileProgram(p, 4, opts);
    const std::string log = nvrtc_log(p);
    if (std::getenv("TDQ_JIT_LOG") && !log.empty()) fprintf(stderr, "%s\n", log.c_str());
    if (r != NVRTC_SUCCESS) {
      nvrtcDestroyProgram(&p);
      return fail(TDQ_ERR_CUDA, std::string("specialised sweep: compilation failed: ") + nvrtcGetErrorString(r) +
                                    "\n" + log.substr(0, 4000));
    }
    size_t n = 0;
    nvrtcGetCUBINSize(p, &n);
    std::string cubin(n, '\0');
    nvrtcGetCUBIN(p, &cubin[0]);
    nvrtcDestroyProgram(&p);
    TDQ_CUDA_TRY(cudaLibraryLoadData(&lib, cubin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0));
    std::lock_guard<std::mutex> lk(C.mu);
    auto ins = C.libs.emplace(code.key, lib);
    if (!ins.second) {  // another thread compiled the same code meanwhile
      cudaLibraryUnload(lib);
      lib = ins.first->second;
    }
  }
  cudaKernel_t k = nullptr;
  TDQ_CUDA_TRY(cudaLibraryGetKernel(&k, lib, name));
  *kernel = reinterpret_cast<const void*>(k);
  return TDQ_OK;
}


// One module compiled to relocatable device code (a cubin for linking), its
// functions held to maxrreg registers (0: no limit).
static tdq_status jit_module(const std::string& src, int maxrreg, std::string* cubin, std::string* err) {
  nvrtcProgram p;
  if (nvrtcCreateProgram(&p, src.c_str(), "tdq_module.cu", kJitHeaderCount, kJitHeaderSrc, kJitHeaderNames) !=
      NVRTC_SUCCESS) {
    *err = "nvrtcCreateProgram failed";
    return TDQ_ERR_CUDA;
  }
  const std::string rr = "--maxrregcount=" + std::to_string(maxrreg);
  const char* opts[] = {"-arch=sm_103a", "-std=c++17", "-default-device", "-lineinfo", "-rdc=true", rr.c_str()};
  const nvrtcResult r = nvrtcCompileProgram(p, maxrreg > 0 ? 6 : 5, opts);
  if (r != NVRTC_SUCCESS) {
    *err = std::string("compilation failed: ") + nvrtcGetErrorString(r) + "\n" + nvrtc_log(p).substr(0, 4000);
    nvrtcDestroyProgram(&p);
    return TDQ_ERR_CUDA;
  }
  size_t n = 0;
  nvrtcGetCUBINSize(p, &n);
  cubin->assign(n, '\0');
  nvrtcGetCUBIN(p, &(*cubin)[0]);
  nvrtcDestroyProgram(&p);
  return TDQ_OK;
}

tdq_status jit_link_kernel(const JitCode& code, const char* name, int maxrreg, const void** kernel) {
  *kernel = nullptr;
  int dev = 0;
  TDQ_CUDA_TRY(cudaGetDevice(&dev));
  int maj = 0, min = 0;
  TDQ_CUDA_TRY(cudaDeviceGetAttribute(&maj, cudaDevAttrComputeCapabilityMajor, dev));
  TDQ_CUDA_TRY(cudaDeviceGetAttribute(&min, cudaDevAttrComputeCapabilityMinor, dev));
  if (maj != 10 || min != 3)
    return fail(TDQ_ERR_UNSUPPORTED, "specialised sweep: built for sm_103a, device is sm_" + std::to_string(maj) +
                                         std::to_string(min));
  const std::string key = std::to_string(maxrreg) + ' ' + code.key;
  JitCache& C = cache();
  cudaLibrary_t lib = nullptr;
  {
    std::lock_guard<std::mutex> lk(C.mu);
    auto it = C.libs.find(key);
    if (it != C.libs.end()) lib = it->second;
  }
  if (!lib) {
    const std::vector<std::string> mods = code.modules();
    // every module on its own host thread, then one link
    std::vector<std::string> cubins(mods.size()), errs(mods.size());
    std::vector<tdq_status> st(mods.size(), TDQ_OK);
    std::atomic<size_t> next{0};
    const size_t nt = std::max<size_t>(1, std::min<size_t>(mods.size(), std::thread::hardware_concurrency()));
    std::vector<std::thread> pool;
    for (size_t w = 0; w < nt; w++)
      pool.emplace_back([&] {
        for (size_t i = next++; i < mods.size(); i = next++) {
          try {
            st[i] = jit_module(mods[i], maxrreg, &cubins[i], &errs[i]);
          } catch (...) {
            st[i] = TDQ_ERR_OOM;
            errs[i] = "host allocation";
          }
        }
      });
    for (auto& t : pool) t.join();
    for (size_t i = 0; i < mods.size(); i++)
      if (st[i] != TDQ_OK) return fail(st[i], "specialised sweep, module " + std::to_string(i) + ": " + errs[i]);
    nvJitLinkHandle h;
    const char* lopts[] = {"-arch=sm_103a"};
    if (nvJitLinkCreate(&h, 1, lopts) != NVJITLINK_SUCCESS) return fail(TDQ_ERR_CUDA, "nvJitLinkCreate failed");
    auto link_fail = [&](const std::string& what) {
      size_t n = 0;
      std::string log;
      if (nvJitLinkGetErrorLogSize(h, &n) == NVJITLINK_SUCCESS && n > 1) {
        log.assign(n, '\0');
        nvJitLinkGetErrorLog(h, &log[0]);
      }
      nvJitLinkDestroy(&h);
      return fail(TDQ_ERR_CUDA, "specialised sweep: " + what + "\n" + log.substr(0, 4000));
    };
    for (size_t i = 0; i < cubins.size(); i++)
      if (nvJitLinkAddData(h, NVJITLINK_INPUT_CUBIN, cubins[i].data(), cubins[i].size(),
                           ("module" + std::to_string(i)).c_str()) != NVJITLINK_SUCCESS)
        return link_fail("adding module " + std::to_string(i));
    if (nvJitLinkComplete(h) != NVJITLINK_SUCCESS) return link_fail("link failed");
    size_t n = 0;
    if (nvJitLinkGetLinkedCubinSize(h, &n) != NVJITLINK_SUCCESS) return link_fail("linked size");
    std::string cubin(n, '\0');
    if (nvJitLinkGetLinkedCubin(h, &cubin[0]) != NVJITLINK_SUCCESS) return link_fail("linked cubin");
    nvJitLinkDestroy(&h);
    TDQ_CUDA_TRY(cudaLibraryLoadData(&lib, cubin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0));
    std::lock_guard<std::mutex> lk(C.mu);
    auto ins = C.libs.emplace(key, lib);
    if (!ins.second) {
      cudaLibraryUnload(lib);
      lib = ins.first->second;
    }
  }
  cudaKernel_t k = nullptr;
  TDQ_CUDA_TRY(cudaLibraryGetKernel(&k, lib, name));
  *kernel = reinterpret_cast<const void*>(k);
  return TDQ_OK;
}

}  // namespace tdq

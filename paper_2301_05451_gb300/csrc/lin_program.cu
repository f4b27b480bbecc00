// Scheduling of gate programs in a linear frame (see lin_program.h).
#include "lin_program.h"

#include <algorithm>

namespace tdq {

void LinSpace::add(uint32_t m) {
  m = reduce(m);
  int p = 31;
  while (!((m >> p) & 1u)) p--;
  for (uint32_t& w : v)
    if ((w >> p) & 1u) w ^= m;
  v.push_back(m);
  pivot.push_back(p);
}

std::vector<LinOp> lin_ops(const std::vector<SweepOp>& ops, int n, LinMap* map) {
  LinMap& A = *map;
  A.n = n;
  A.row.assign(n, 0);
  A.col.assign(n, 0);
  A.b = 0;
  A.quarter = 0;
  for (int q = 0; q < n; q++) A.row[q] = A.col[q] = 1u << q;
  std::vector<LinOp> out;
  auto put = [&](LinKind kind, int q, int op, int ang, int slot, bool p) {
    LinOp o{};
    o.kind = kind;
    o.m = kind == L_RY || kind == L_RX || kind == L_H ? A.col[q] : 0u;
    o.f = A.row[q];
    o.b = (uint8_t)((A.b >> q) & 1u);
    o.p = p;
    o.op = op;
    o.ang = ang;
    o.slot = slot;
    out.push_back(o);
  };
  for (int i = 0; i < (int)ops.size(); i++) {
    const SweepOp& g = ops[i];
    switch (g.kind) {
      case K_CNOT:
        A.row[g.p1] ^= A.row[g.p0];
        A.b ^= ((A.b >> g.p0) & 1u) << g.p1;
        A.col[g.p0] ^= A.col[g.p1];
        break;
      case K_X: A.b ^= 1u << g.p0; break;
      case K_Y:  // Y = i X Z
        put(L_SIGN, g.p0, -1, 0, -1, false);
        A.b ^= 1u << g.p0;
        A.quarter = (A.quarter + 1) & 3;
        break;
      case K_Z: put(L_SIGN, g.p0, -1, 0, -1, false); break;
      case K_H: put(L_H, g.p0, -1, 0, -1, false); break;
      case K_RX: put(L_RX, g.p0, i, 0, g.slot[0], false); break;
      case K_RY: put(L_RY, g.p0, i, 0, g.slot[0], false); break;
      case K_RZ: put(L_PHASE, g.p0, i, 0, g.slot[0], false); break;
      case K_U3:
        put(L_PHASE, g.p0, i, 2, g.slot[2], true);
        put(L_RY, g.p0, i, 0, g.slot[0], false);
        put(L_PHASE, g.p0, i, 1, g.slot[1], true);
        break;
      case K_RZZ:  // a phase by the parity of the two bits
        put(L_PHASE, g.p0, i, 0, g.slot[0], false);
        out.back().f ^= A.row[g.p1];
        out.back().b ^= (uint8_t)((A.b >> g.p1) & 1u);
        break;
      default:  // K_CZ
        put(L_CZ, g.p0, -1, 0, -1, false);
        out.back().f2 = A.row[g.p1];
        out.back().b2 = (uint8_t)((A.b >> g.p1) & 1u);
    }
  }
  return out;
}

// Pauli products (x mask, z parity) that generate an op; at most two.
static int generators(const LinOp& o, uint32_t (&x)[2], uint32_t (&z)[2]) {
  switch (o.kind) {
    case L_RY: x[0] = o.m; z[0] = o.f; return 1;
    case L_RX: x[0] = o.m; z[0] = 0; return 1;
    case L_H: x[0] = o.m; z[0] = 0; x[1] = 0; z[1] = o.f; return 2;
    case L_CZ: x[0] = x[1] = 0; z[0] = o.f; z[1] = o.f2; return 2;
    default: x[0] = 0; z[0] = o.f; return 1;
  }
}

bool lin_commute(const LinOp& a, const LinOp& b) {
  uint32_t ax[2], az[2], bx[2], bz[2];
  const int na = generators(a, ax, az), nb = generators(b, bx, bz);
  for (int i = 0; i < na; i++)
    for (int j = 0; j < nb; j++)
      if (parity32(ax[i] & bz[j]) ^ parity32(az[i] & bx[j])) return false;
  return true;
}

namespace {

// Takes ops of `todo` (program order) whose masks fit a space of at most dim
// vectors grown from `space`; an op may pass earlier ones left behind that it
// commutes with.  mask(o): the op's mask in the space's coordinates.
// The first op always fits; what else may be taken:
struct TakeCaps {  // (0: any number)
  int slots;     // gradient slots
  int rows;      // angles
  int unscaled;  // gates that leave their factor to the pass's scale
};
template <class Mask>
void take(const std::vector<LinOp>& ops, std::vector<int>& todo, int dim, LinSpace& space, TakeCaps caps, Mask mask,
          std::vector<int>* taken) {
  std::vector<int> left;
  int ns = 0, nr = 0, nu = 0;
  for (int o : todo) {
    bool ok = true;
    for (size_t i = 0; i < left.size() && ok; i++) ok = lin_commute(ops[o], ops[left[i]]);
    const int s = ops[o].slot >= 0 ? 1 : 0, r = ops[o].op >= 0 ? 1 : 0, u = ops[o].m ? 1 : 0;
    if (!taken->empty() && ((caps.slots && ns + s > caps.slots) || (caps.rows && nr + r > caps.rows) ||
                            (caps.unscaled && nu + u > caps.unscaled)))
      ok = false;
    if (ok && ops[o].m) {
      const uint32_t m = mask(ops[o].m);
      if (space.reduce(m)) {
        if ((int)space.v.size() < dim) space.add(m);
        else ok = false;
      }
    }
    if (ok) {
      taken->push_back(o);
      ns += s;
      nr += r;
      nu += u;
    } else {
      left.push_back(o);
    }
  }
  todo.swap(left);
}

// Gates that a register pass leaves unscaled at most: each grows the amplitudes by
// up to sqrt 2, so by 2^24 in a pass, and the scale that takes it back is at least
// 2^-24 (its square, for the shares of a reverse pass, 2^-48).  Chains of hundreds
// of gates on one or two qubits would overflow; a pass of a wider circuit is full
// long before.
constexpr int kUnscaled = 48;

// Register passes over the tile's ops.  A pass's group index bits are sent to
// the local bits outside U's pivots so that 16 consecutive groups read 16
// different shared-memory slots (see swz and swz_pair: local bit p moves slot
// bit p mod 4, or 0 and 1 + (p - 1) mod 3, for p < 12), as far as the free bits
// allow.  In pairs, local bit 0 is a pivot only of the vector 1: the members
// are then read two at a time.
std::vector<LinReg> reg_passes(const std::vector<LinOp>& ops, const LinTile& t, const LinSpace& V, int mreg,
                               int max_slots, bool pairs) {
  auto slot_bit = [&](int l) { return !pairs ? l & 3 : l ? 1 + (l - 1) % 3 : 0; };
  std::vector<LinReg> out;
  const int M = std::min(mreg, t.k);
  auto local = [&](uint32_t m) {  // coordinates of m in the tile's basis
    uint32_t l = 0;
    for (int i = 0; i < t.k; i++)
      if ((m >> V.pivot[i]) & 1u) l |= 1u << i;
    return l;
  };
  std::vector<int> todo = t.ops;
  while (!todo.empty()) {
    LinReg r;
    r.M = M;
    LinSpace U;
    take(ops, todo, M, U, {max_slots, 0, kUnscaled}, local, &r.ops);
    for (int l = 0; l < t.k && (int)U.v.size() < M; l++)
      if (U.reduce(1u << l)) U.add(1u << l);
    // order by pivot; the pivots are free to choose: prefer those that leave
    // every slot bit a local bit outside them
    for (int i = 0; i < M; i++) r.u[i] = U.v[i];
    uint32_t piv = U.pivots();
    int best = -1;
    std::vector<int> choice(M), pick(M);
    // all pivot sets (one local bit per basis vector, re-reduced) are tried
    // greedily: move a pivot to another set bit of its vector when that frees
    // a slot bit no free local bit reaches
    auto reach = [&](uint32_t p) {
      uint32_t any = pairs ? 1u : 0u;  // (bit 0: read in pairs where it is a pivot)
      for (int l = 0; l < std::min(t.k, 12); l++)
        if (!((p >> l) & 1u)) any |= 1u << slot_bit(l);
      return __builtin_popcount(any);
    };
    best = reach(piv);
    for (int round = 0; round < M && best < 4; round++)
      for (int i = 0; i < M && best < 4; i++)
        for (int l = 0; l < t.k; l++) {
          if (!((U.v[i] >> l) & 1u) || l == U.pivot[i] || (pairs && l == 0)) continue;
          const uint32_t p2 = (piv & ~(1u << U.pivot[i])) | (1u << l);
          if (reach(p2) <= best) continue;
          for (int j = 0; j < M; j++)
            if (j != i && ((U.v[j] >> l) & 1u)) U.v[j] ^= U.v[i];
          U.pivot[i] = l;
          piv = p2;
          best = reach(p2);
          break;
        }
    for (int i = 0; i < M; i++) r.u[i] = U.v[i];
    std::vector<int> free_pos;
    for (int l = 0; l < t.k; l++)
      if (!((piv >> l) & 1u)) free_pos.push_back(l);
    // the first four group bits: free local bits of different slot bits
    std::vector<char> used(free_pos.size(), 0);
    uint32_t slots = 0;
    for (size_t i = 0; i < free_pos.size() && r.grp_pos.size() < 4; i++)
      if (free_pos[i] < 12 && !((slots >> slot_bit(free_pos[i])) & 1u)) {
        slots |= 1u << slot_bit(free_pos[i]);
        used[i] = 1;
        r.grp_pos.push_back(free_pos[i]);
      }
    for (size_t i = 0; i < free_pos.size(); i++)
      if (!used[i]) r.grp_pos.push_back(free_pos[i]);
    out.push_back(r);
  }
  return out;
}

CoefRec angle_record(const std::vector<SweepOp>& gates, const LinOp& g) {
  const SweepOp& op = gates[g.op];
  return {op.src[g.ang], op.fixed[g.ang], 4 * g.op + g.ang, g.kind == L_PHASE ? C_PHASE : C_ROT};
}

// The rows' sign flips and the final index part: the Pauli product of every
// rotation, carried through the ops after it (CZ and H change it, the others
// commute or flip sign with it).
void frame_tables(const std::vector<SweepOp>& gates, LinProgram& P) {
  std::vector<int> rots;
  for (int i = 0; i < (int)P.ops.size(); i++)
    if (P.ops[i].kind == L_RY || P.ops[i].kind == L_RX) {
      rots.push_back(i);
      P.rot.push_back(angle_record(gates, P.ops[i]));
    }
  const int words = ((int)rots.size() + 31) / 32;
  std::vector<int> tile_of(P.ops.size(), -1);
  for (int t = 0; t < (int)P.tiles.size(); t++) {
    P.tiles[t].flips.assign(P.tiles[t].coef.size() * (size_t)words, 0u);
    for (int o : P.tiles[t].ops) tile_of[o] = t;
  }
  for (int j = 0; j < (int)rots.size(); j++) {
    uint32_t x = P.ops[rots[j]].m, z = P.ops[rots[j]].kind == L_RY ? P.ops[rots[j]].f : 0u;
    for (int i = rots[j] + 1; i < (int)P.ops.size(); i++) {
      const LinOp& g = P.ops[i];
      if (g.kind == L_CZ) {
        const uint32_t add = (parity32(g.f & x) ? g.f2 : 0u) ^ (parity32(g.f2 & x) ? g.f : 0u);
        z ^= add;
      } else if (g.kind == L_H) {
        if (parity32(g.f & x) ^ parity32(z & g.m)) {
          x ^= g.m;
          z ^= g.f;
        }
      } else if (P.coef[i] >= 0) {
        const uint32_t gz = g.kind == L_RX ? 0u : g.f;
        if (parity32(x & gz) ^ parity32(z & g.m))
          P.tiles[tile_of[i]].flips[(size_t)P.coef[i] * words + j / 32] |= 1u << (j & 31);
      }
    }
    P.rot_x.push_back(x);
  }
}

}  // namespace

LinProgram lin_program(const std::vector<SweepOp>& gates, int n, int k, int L, int mf, int mr, bool adj, bool exact) {
  LinProgram P;
  P.n = n;
  P.exact = exact;
  P.pairs = L > 0;
  P.ops = lin_ops(gates, n, &P.map);
  P.coef.assign(P.ops.size(), -1);
  std::vector<int> todo;
  for (int i = 0; i < (int)P.ops.size(); i++) todo.push_back(i);
  do {
    LinTile t;
    t.k = k;
    LinSpace V;
    for (int i = 0; i < L; i++) V.add(1u << i);
    // A tile pass keeps at most kTileSlots gradient accumulators, 32 bytes each,
    // and the tables of kTileRows angles, 16 to 20 bytes each, beside its states in
    // shared memory.  A whole state is one tile whatever its angles: where its
    // tables do not fit, it is not run as one.
    constexpr int kTileSlots = 512, kTileRows = 2048;
    take(P.ops, todo, k, V, {L > 0 && adj ? kTileSlots : 0, L > 0 ? kTileRows : 0, 0}, [](uint32_t m) { return m; },
         &t.ops);
    for (int p = 0; p < n && (int)V.v.size() < k; p++)
      if (V.reduce(1u << p)) V.add(1u << p);
    // local bits in the order of their pivots (the L lowest first)
    std::vector<int> order(k);
    for (int i = 0; i < k; i++) order[i] = i;
    std::sort(order.begin(), order.end(), [&](int a, int b) { return V.pivot[a] < V.pivot[b]; });
    LinSpace W;
    for (int i : order) {
      W.v.push_back(V.v[i]);
      W.pivot.push_back(V.pivot[i]);
    }
    t.v = W.v;
    t.pivots = W.pivots();
    t.fwd = reg_passes(P.ops, t, W, mf, 0, P.pairs);
    if (adj) t.rev = reg_passes(P.ops, t, W, mr, kRevPassSlots, P.pairs);
    // the gate-tensor table: one row per angle, one per register pass with
    // unscaled gates
    for (int o : t.ops) {
      const LinOp& g = P.ops[o];
      if (g.kind != L_RY && g.kind != L_RX && g.kind != L_PHASE) continue;
      P.coef[o] = (int)t.coef.size();
      t.coef.push_back(angle_record(gates, g));
    }
    for (std::vector<LinReg>* rs : {&t.fwd, &t.rev})
      for (LinReg& r : *rs) {
        int nh = 0, nd = 0;
        const int first = (int)t.norm.size();
        for (int o : r.ops) {
          nh += P.ops[o].kind == L_H ? 1 : 0;
          nd += P.ops[o].m ? 1 : 0;
          if (P.ops[o].kind == L_RY || P.ops[o].kind == L_RX)
            t.norm.push_back(2 * P.coef[o] + (P.ops[o].kind == L_RX ? 1 : 0));
        }
        if (!nd) continue;
        r.norm = (int)t.coef.size();
        t.coef.push_back({(int)t.norm.size() - first, 0.f, first, (exact ? C_NORM_EXACT : C_NORM) + (nh << 8)});
      }
    P.tiles.push_back(t);
  } while (!todo.empty());
  if (!exact) frame_tables(gates, P);
  return P;
}

std::string lin_key(const LinProgram& P) {
  std::string k;
  auto put = [&](uint64_t v) { k.append(reinterpret_cast<const char*>(&v), sizeof(v)); };
  auto list = [&](const auto& v) {
    put(v.size());
    if (!v.empty()) k.append(reinterpret_cast<const char*>(v.data()), v.size() * sizeof(v[0]));
  };
  put(P.n);
  put((P.pairs ? 1u : 0u) | (P.exact ? 2u : 0u) | (P.rot.empty() ? 4u : 0u));
  put(P.ops.size());
  for (const LinOp& o : P.ops) {
    put(o.kind | o.b << 8 | o.b2 << 16 | (o.p ? 1 : 0) << 24 | (uint64_t)o.m << 32);
    put(o.f | (uint64_t)o.f2 << 32);
    put(o.slot);
  }
  list(P.coef);
  put(P.tiles.size());
  for (const LinTile& t : P.tiles) {
    put(t.k);
    put(t.pivots);
    put(t.coef.size());
    list(t.v);
    list(t.ops);
    for (const std::vector<LinReg>* rs : {&t.fwd, &t.rev}) {
      put(rs->size());
      for (const LinReg& r : *rs) {
        put(r.M);
        put(r.norm);
        for (int i = 0; i < r.M; i++) put(r.u[i]);
        list(r.grp_pos);
        list(r.ops);
      }
    }
  }
  return k;
}

// A tile is read in runs of 2^L amplitudes.  Runs of 128 bytes (L = 4) need the
// fewest cache lines per read, but bits held for them are taken from the
// gates; 32-byte runs (L = 2) still fill the sectors that memory moves, and a
// line's other runs belong to neighbouring tiles, read next.  What a choice
// costs: every tile pass but the first (which visits one tile per row) moves
// the state once, about 3, 4 or 5 register passes' worth at L = 4, 3, 2 (20
// qubits, 16 rows, forward: 45 us at L = 4, 60 to 90 at L = 2, a register pass
// 11), and runs its register passes.  20-qubit ladder, 64 rows, value and
// gradient: L = 4, 6 tile passes and 18 register passes after the first, 5.6
// ms; L = 2, 4 and 14, 4.9 ms; its 481 shifted circuits 11.3 -> 9.4 ms.
LinProgram lin_tiled_program(const std::vector<SweepOp>& ops, int n, int k, int mf, int mr, bool adj, bool exact,
                             int* L) {
  LinProgram best;
  int best_cost = -1;
  for (int l = std::min(4, k); l >= std::min(2, k); l--) {
    LinProgram p = lin_program(ops, n, k, l, mf, mr, adj, exact);
    const int move = 7 - l;
    int cost = 0;
    for (size_t t = 1; t < p.tiles.size(); t++)
      cost += move + (int)p.tiles[t].fwd.size() + (adj ? 2 * (move + (int)p.tiles[t].rev.size()) : 0);
    if (best_cost >= 0 && cost >= best_cost) continue;
    best_cost = cost;
    best = std::move(p);
    *L = l;
  }
  return best;
}

}  // namespace tdq

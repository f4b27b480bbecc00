// Gate programs in a linear frame of the basis index, for the specialised
// sweep kernels.
//
// The state buffer is indexed by y, the circuit's basis index by x; the two
// are related by an affine map over GF(2), x = A y + b, that starts as the
// identity.  CNOT and X only change the map (CNOT adds the control's row of A
// to the target's, X flips a bit of b), so they never touch the state.  Every
// other gate acts through two bit vectors: flipping logical bit q alone flips
// y by the mask m = A^-1 e_q, and the bit's value is the parity of f & y
// (f = row q of A) xor b_q.  A one-qubit gate pairs y with y ^ m; diagonal
// gates are phases by parities of f & y.  U3(t, p, l) is written as its exact
// factors P(l), RY(t), P(p), with P(a) = diag(1, e^{ia}).
//
// A tile is a coset of a subspace V of the index space (it always holds the
// lowest index bits, so that a tile is read in contiguous runs); a register
// group is a coset of a subspace U of the tile's local indices.  An op fits
// when its mask lies in the subspace; ops are taken ahead of others that they
// commute with (as Pauli products).
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include "engine.cuh"

namespace tdq {

struct LinOp {
  LinKind kind;
  uint32_t m;      // pairing mask (RY, RX, H), else 0
  uint32_t f, f2;  // parities that give the logical bit(s): f (all kinds), f2 (CZ)
  uint8_t b, b2;   // constants added to them
  bool p;          // PHASE: P(a) instead of diag(e^{-ia/2}, e^{ia/2})
  int op, ang;     // gate of the program and its angle (RY, RX, PHASE)
  int slot;        // parameter column receiving the gradient, or -1
};

// x = A y + b of a finished program.
struct LinMap {
  int n = 0;
  std::vector<uint32_t> row;  // A: parity of row[q] & y (xor bit q of b) is bit q of x
  std::vector<uint32_t> col;  // A^-1: flipping bit q of x flips y by col[q]
  uint32_t b = 0;
  int quarter = 0;            // global phase i^quarter left out (Y = i X Z)
  uint32_t to_y(uint32_t x) const {
    uint32_t y = 0;
    x ^= b;
    for (int q = 0; q < n; q++)
      if ((x >> q) & 1u) y ^= col[q];
    return y;
  }
};

inline int parity32(uint32_t v) { return __builtin_popcount(v) & 1; }

// The ops of a gate list on n index bits, and the map at its end.
std::vector<LinOp> lin_ops(const std::vector<SweepOp>& ops, int n, LinMap* map);

bool lin_commute(const LinOp& a, const LinOp& b);

// Subspace of GF(2)^n as a reduced basis: vector i has a 1 at pivot[i], where
// every other vector has a 0.
struct LinSpace {
  std::vector<uint32_t> v;
  std::vector<int> pivot;
  uint32_t reduce(uint32_t m) const {
    for (size_t i = 0; i < v.size(); i++)
      if ((m >> pivot[i]) & 1u) m ^= v[i];
    return m;
  }
  // extend by m (not in the space), with the highest bit of its remainder as pivot
  void add(uint32_t m);
  uint32_t pivots() const {
    uint32_t r = 0;
    for (int p : pivot) r |= 1u << p;
    return r;
  }
};

// A register pass: groups of 2^M local indices (cosets of U), the ops
// absorbed there in program order, and the pass's place in the gate-tensor
// table.
struct LinReg {
  int M;
  uint32_t u[4];                // basis of U (local indices)
  std::vector<int> grp_pos;     // local bit of group-index bit i (k - M of them)
  std::vector<int> ops;
  int norm = -1;                // table row of the pass's scale, or -1
};

// A tile pass: local bit i of the tile moves the index by v[i] (v[0..L) the
// lowest index bits); tiles are numbered by the bits outside `pivots`.
struct LinTile {
  int k = 0;
  std::vector<uint32_t> v;
  uint32_t pivots = 0;
  std::vector<int> ops;
  std::vector<LinReg> fwd, rev;
  std::vector<uint32_t> flips;  // programs with a frame: SweepArgs::rot_flips of the table's rows
  std::vector<CoefRec> coef;    // gate-tensor table
  std::vector<int> norm;        // SweepArgs::norm of its scale rows
};

struct LinProgram {
  int n = 0;
  bool pairs = false;        // tiles move in pairs of neighbours (swz_pair), whole states in swz order
  bool exact = false;        // keep the global phase (state and amplitude outputs): no frame
  std::vector<CoefRec> rot;  // with a frame: SweepArgs::rot and rot_x
  std::vector<uint32_t> rot_x;
  std::vector<LinOp> ops;
  std::vector<int> coef;     // table row of every op in its tile pass, or -1
  std::vector<LinTile> tiles;
  LinMap map;
};

// All that a program's generated code depends on, as bytes: equal for equal code.
std::string lin_key(const LinProgram& P);

// Program of n index bits in tiles of k bits, the L lowest in every tile (L = 0,
// k = n: the whole state, one tile); register passes of at most mf (forward)
// and, with adj, mr (reverse) bits.
LinProgram lin_program(const std::vector<SweepOp>& ops, int n, int k, int L, int mf, int mr, bool adj, bool exact);

// Tiled program: the number of lowest index bits that every tile holds is
// chosen here (4 .. 2, returned in *L): fewer leave a tile more directions of
// its own.
LinProgram lin_tiled_program(const std::vector<SweepOp>& ops, int n, int k, int mf, int mr, bool adj, bool exact,
                             int* L);

}  // namespace tdq

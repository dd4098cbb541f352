// Programs of the expression interpreter (interp.cu): what a program is, and how
// a tree becomes one.  Host code only, so that a program can be checked without
// a GPU.
#pragma once

#include <string.h>

#include "internal.h"

namespace su3s {

constexpr int kIRegs = 12;     // limit of an accepted tree (interp_program)
constexpr int kIRegsRun = 24;  // registers a program that runs may have
constexpr int kIMax = 48;

enum IOp : int8_t { I_LOAD = 0, I_MMUL = 1, I_MVMUL = 2, I_RMUL = 3, I_ADD = 4, I_SUB = 5, I_SCALE = 6, I_ADJ = 7 };

struct IIns {
  int8_t op, dst, a, b;
  int8_t w;    // width in reals of the result (18, 6, 1)
  int8_t arg;  // leaf slot (LOAD, with kind in b) / factor index (SCALE)
  int8_t adj;  // products: 1 the left operand's adjoint, 2 the right one's
  int8_t pad;
};

struct IProg {
  int32_t n;
  int32_t root;
  int32_t root_kind;
  int32_t nregs;   // registers the program uses (shared memory is sized to them)
  int32_t nloads;  // its loads in order: leaf slot and width in reals
  int8_t load_leaf[kMaxLeaves], load_w[kMaxLeaves];
  IIns ins[kIMax];
};

// Two sites per thread in the pair arithmetic: lattices of at least kPairSites
// site vectors, programs of at most kPairRegs registers (see k_interp_pair).
constexpr int64_t kPairSites = 300000;
constexpr int kPairRegs = 3;

struct Builder {
  IProg prog;
  bool busy[kIRegsRun] = {};
  int holds[kIRegsRun] = {};       // operations that have yet to read the register
  int leaf_reg[kMaxLeaves];
  int uses_left[kMaxLeaves] = {};  // leaf nodes of each slot not generated yet
  const Canon* c;
  int limit = kIRegsRun;
  bool hold = true;   // operands stay until they are read (false: counting only)
  bool reuse = true;  // results in place
  bool fold = true;   // adjoints of a product's operands folded into it
  int nscal = 0;
  int err = 0;

  int alloc() {
    for (int r = 0; r < limit; ++r)
      if (!busy[r]) {
        busy[r] = true;
        if (r + 1 > prog.nregs) prog.nregs = r + 1;
        return r;
      }
    err = 1;
    return 0;
  }
  // whether register r is still to be read: by an operation whose other operand
  // is being generated, or as a leaf that occurs again
  bool kept(int r) const {
    if (holds[r] > 0) return true;
    for (int l = 0; l < kMaxLeaves; ++l)
      if (leaf_reg[l] == r && uses_left[l] > 0) return true;
    return false;
  }
  // free register r unless it is still to be read
  void release(int r) {
    if (!kept(r)) busy[r] = false;
  }
  // register of an element-by-element result: an operand's own if it is not
  // needed any more (a leaf's register then holds the leaf no longer)
  int in_place(int a, int b) {
    const int d = !reuse ? -1 : !kept(a) ? a : !kept(b) ? b : -1;
    if (d < 0) return alloc();
    for (int l = 0; l < kMaxLeaves; ++l)
      if (leaf_reg[l] == d) leaf_reg[l] = -1;
    return d;
  }
  void emit(IIns in) {
    if (prog.n >= kIMax) {
      err = 2;
      return;
    }
    prog.ins[prog.n++] = in;
  }
  static int8_t width(int kind) { return kind == SU3S_MATRIX ? 18 : kind == SU3S_VECTOR ? 6 : 1; }

  int slot_of(const su3s_field* f) {
    for (size_t i = 0; i < c->leaves.size(); ++i)
      if (c->leaves[i] == f) return (int)i;
    return 0;
  }

  void count_uses(const su3s_expr* e) {
    if (e->op == 0) {
      ++uses_left[slot_of(e->f)];
      return;
    }
    if (e->a) count_uses(e->a);
    if (e->b) count_uses(e->b);
  }

  // returns the register holding the node's value
  int gen(const su3s_expr* e) {
    if (err) return 0;
    switch (e->op) {
      case 0: {  // a leaf: loaded at its first use
        const int l = slot_of(e->f);
        if (leaf_reg[l] < 0) {
          const int r = alloc();
          leaf_reg[l] = r;
          const int kind = e->f->kind;
          emit(IIns{I_LOAD, (int8_t)r, 0, (int8_t)kind, width(kind), (int8_t)l, 0, 0});
          if (!err) {
            prog.load_leaf[prog.nloads] = (int8_t)l;
            prog.load_w[prog.nloads++] = width(kind);
          }
        }
        --uses_left[l];
        return leaf_reg[l];
      }
      case 4: {
        int k = nscal++;  // factors numbered in the canonical (pre-order) order
        int a = gen(e->a);
        int d = in_place(a, a);
        emit(IIns{I_SCALE, (int8_t)d, (int8_t)a, 0, width(e->kind), (int8_t)k, 0, 0});
        if (a != d) release(a);
        return d;
      }
      case 5: {
        int a = gen(e->a);
        int d = alloc();
        emit(IIns{I_ADJ, (int8_t)d, (int8_t)a, 0, 18, 0, 0, 0});
        release(a);
        return d;
      }
      default: {
        const su3s_expr *ea = e->a, *eb = e->b;
        int8_t adj = 0, op;
        if (e->op == 1) {
          op = e->kind == SU3S_MATRIX ? I_MMUL : e->kind == SU3S_VECTOR ? I_MVMUL : I_RMUL;
          // a product reads the adjoint of an operand from the operand itself
          for (; fold && ea->op == 5; ea = ea->a) adj ^= 1;
          for (; fold && eb->op == 5; eb = eb->a) adj ^= 2;
        } else {
          op = e->op == 2 ? I_ADD : I_SUB;
        }
        int a = gen(ea);
        const bool again = kept(a);
        if (hold) ++holds[a];   // the right operand's steps come before this one reads it
        int b = gen(eb);
        if (hold) --holds[a];
        // A product takes a register of its own, or that of a leaf on its left whose
        // last use was in its right operand.  Not an adjoint's: the two-sites kernel
        // stores row i of a product before it reads column i + 1 of such an operand
        // (a row is read before the one above it is stored).
        const bool left = reuse && again && !kept(a) && !(op == I_MMUL && (adj & 1));
        int d = e->op != 1 ? in_place(a, b) : left ? in_place(a, a) : alloc();
        emit(IIns{op, (int8_t)d, (int8_t)a, (int8_t)b, width(e->kind), 0, adj, 0});
        if (a != d) release(a);
        if (b != d) release(b);
        return d;
      }
    }
  }
};

// The program of a tree, and whether it is one for two sites per thread (large:
// such programs are wanted).  Returns 0, or non-zero where the tree is too large.
// The limits on a tree are those of a plain program (one register per result,
// adjoints as steps of their own) that gives a leaf's register back as soon as
// its last use is generated.  A program that runs keeps it until the last
// operation that reads it, with results in place where they can be, and may have
// more registers for that (9 at most among random trees of 8 leaves); it has no
// more steps.
inline int interp_program(const su3s_expr* e, const Canon& c, bool large, IProg* prog, bool* pairs) {
  *pairs = false;
  for (int pass = 0; pass < 3; ++pass) {
    // 0: the limits; 1: two sites per thread, adjoints read in place; 2: one site
    if (pass == 1 && !large) continue;
    Builder bld;
    memset(&bld.prog, 0, sizeof bld.prog);
    bld.c = &c;
    bld.limit = pass > 0 ? kIRegsRun : kIRegs;
    bld.hold = bld.reuse = pass > 0;
    bld.fold = pass == 1;
    for (int l = 0; l < kMaxLeaves; ++l) bld.leaf_reg[l] = -1;
    bld.count_uses(e);
    bld.prog.root = bld.gen(e);
    bld.prog.root_kind = c.kind;
    if (bld.err) return bld.err;
    *prog = bld.prog;
    int products = 0;
    for (int i = 0; i < prog->n; ++i) products += prog->ins[i].op == I_MMUL || prog->ins[i].op == I_MVMUL;
    *pairs = pass == 1 && prog->nregs <= kPairRegs && products <= 2;
    if (*pairs) break;
  }
  return 0;
}

}  // namespace su3s

// Programs of the expression interpreter against the trees they stand for, without a GPU: random
// trees of matrices, vectors and reals in which fields occur several times, each program run step
// by step on integers (exact, modulo 2^64) and compared with the tree's own value.
//   interp_programs <trees> <seed>
// prints the trees checked, or the first whose program is wrong.
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>

#include <memory>
#include <string>
#include <vector>

#include "interp_prog.h"

using namespace su3s;

namespace {

struct Rng {
  uint64_t s;
  uint32_t next() {   // 64-bit linear congruential generator, upper half
    s = s * 6364136223846793005ull + 1442695040888963407ull;
    return (uint32_t)(s >> 33);
  }
  int below(int n) { return (int)(next() % (uint32_t)n); }
};

using U = uint64_t;
struct Value {
  U re[9] = {}, im[9] = {};   // a matrix, the first three of a vector, the first real
};

int elems(int kind) { return kind == SU3S_MATRIX ? 9 : kind == SU3S_VECTOR ? 3 : 1; }

void cmadd(Value& z, int k, const Value& x, int i, const Value& y, int j) {
  z.re[k] += x.re[i] * y.re[j] - x.im[i] * y.im[j];
  z.im[k] += x.re[i] * y.im[j] + x.im[i] * y.re[j];
}
Value product(const Value& x, const Value& y, int kind) {
  Value z;
  const int nc = kind == SU3S_MATRIX ? 3 : 1;
  if (kind == SU3S_REAL) z.re[0] = x.re[0] * y.re[0];
  else
    for (int i = 0; i < 3; ++i)
      for (int k = 0; k < nc; ++k)
        for (int j = 0; j < 3; ++j) cmadd(z, nc * i + k, x, 3 * i + j, y, nc * j + k);
  return z;
}
Value combine(const Value& x, const Value& y, U sg, int kind) {
  Value z;
  for (int e = 0; e < elems(kind); ++e) {
    z.re[e] = x.re[e] + sg * y.re[e];
    z.im[e] = x.im[e] + sg * y.im[e];
  }
  return z;
}
Value scaled(const Value& x, double s, int kind) { return combine(Value(), x, (U)(int64_t)s, kind); }
Value adjoint(const Value& x) {
  Value z;
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      z.re[3 * i + j] = x.re[3 * j + i];
      z.im[3 * i + j] = 0 - x.im[3 * j + i];
    }
  return z;
}

struct Forest {
  std::vector<std::unique_ptr<su3s_expr>> nodes;
  std::vector<su3s_field> fields;
  std::vector<Value> values;
  Rng rng;
  int nscal = 0;

  su3s_expr* node(int op, int kind, const su3s_expr* a = nullptr, const su3s_expr* b = nullptr) {
    nodes.emplace_back(new su3s_expr);
    su3s_expr* e = nodes.back().get();
    e->op = op;
    e->kind = kind;
    e->a = a;
    e->b = b;
    return e;
  }
  // A tree of `uses` leaf nodes and the given kind.
  su3s_expr* tree(int uses, int kind) {
    const int unary = rng.below(5);
    if (unary == 0 && kind == SU3S_MATRIX) return node(5, kind, tree(uses, kind));
    if (unary == 1 && nscal < kMaxScalars) {
      ++nscal;
      const double s = (double)((rng.below(9) - 4) * 3 + 1);
      su3s_expr* e = node(4, kind, tree(uses, kind));
      e->s = s;
      return e;
    }
    if (uses == 1) {
      int l;
      do l = rng.below((int)fields.size());
      while (fields[l].kind != kind);
      su3s_expr* e = node(0, kind);
      e->f = &fields[l];
      return e;
    }
    const int left = 1 + rng.below(uses - 1), op = 1 + rng.below(3);
    const int ka = op == 1 && kind == SU3S_VECTOR ? (int)SU3S_MATRIX : kind;
    su3s_expr* a = tree(left, ka);
    return node(op, kind, a, tree(uses - left, kind));
  }
  Value value(const su3s_expr* e) const {
    switch (e->op) {
      case 0: return values[e->f - fields.data()];
      case 1: return product(value(e->a), value(e->b), e->kind);
      case 2: return combine(value(e->a), value(e->b), 1, e->kind);
      case 3: return combine(value(e->a), value(e->b), (U)-1, e->kind);
      case 4: return scaled(value(e->a), e->s, e->kind);
      default: return adjoint(value(e->a));
    }
  }
  std::string text(const su3s_expr* e) const {
    switch (e->op) {
      case 0: return std::string(1, (char)('a' + (e->f - fields.data())));
      case 4: return std::to_string((int)e->s) + "*" + text(e->a);
      case 5: return "adj(" + text(e->a) + ")";
      default: return "(" + text(e->a) + (e->op == 1 ? "*" : e->op == 2 ? "+" : "-") + text(e->b) + ")";
    }
  }
};

// Leaves by first appearance and real factors in pre-order, as canonicalize numbers them.
void canon(const su3s_expr* e, Canon* c) {
  if (e->op == 0) {
    for (su3s_field* f : c->leaves)
      if (f == e->f) return;
    c->leaves.push_back(e->f);
    return;
  }
  if (e->op == 4) c->scalars.push_back(e->s);
  if (e->a) canon(e->a, c);
  if (e->b) canon(e->b, c);
}

// What is wrong with a program: empty if nothing.
std::string check(const Forest& f, const su3s_expr* e, const Canon& c, const IProg& p, bool pairs) {
  std::vector<Value> reg(kIRegsRun);
  int loads = 0;
  if (p.nregs > kIRegsRun) return "too many registers";
  for (int pc = 0; pc < p.n; ++pc) {
    const IIns in = p.ins[pc];
    const int kind = in.w == 18 ? SU3S_MATRIX : in.w == 6 ? SU3S_VECTOR : SU3S_REAL;
    if (in.dst < 0 || in.dst >= p.nregs || in.a < 0 || in.a >= p.nregs) return "register out of range";
    const Value x = (in.adj & 1) ? adjoint(reg[in.a]) : reg[in.a];
    switch (in.op) {
      case I_LOAD:
        if (p.load_leaf[loads] != in.arg || p.load_w[loads] != in.w) return "list of loads";
        ++loads;
        reg[in.dst] = f.values[c.leaves[in.arg] - f.fields.data()];
        break;
      case I_SCALE: reg[in.dst] = scaled(x, c.scalars[in.arg], kind); break;
      case I_ADJ:
        if (pairs && in.dst == in.a) return "an adjoint over its operand";
        reg[in.dst] = adjoint(x);
        break;
      case I_ADD:
      case I_SUB: reg[in.dst] = combine(x, reg[in.b], in.op == I_ADD ? 1 : (U)-1, kind); break;
      default:
        // two sites per thread: rows are stored before an adjoint's last columns are read
        if (pairs && in.op == I_MMUL && in.dst == in.a && (in.adj & 1)) return "a product over its operand";
        reg[in.dst] = product(x, (in.adj & 2) ? adjoint(reg[in.b]) : reg[in.b], kind);
    }
  }
  if (loads != p.nloads) return "number of loads";
  const Value want = f.value(e), got = reg[p.root];
  for (int k = 0; k < elems(e->kind); ++k)
    if (want.re[k] != got.re[k] || want.im[k] != got.im[k]) return "value";
  return "";
}

}  // namespace

int main(int argc, char** argv) {
  const int trees = argc > 1 ? atoi(argv[1]) : 1000;
  Rng seeds{argc > 2 ? strtoull(argv[2], nullptr, 10) : 1};
  int done = 0, reused = 0, refused = 0, two = 0, most = 0;
  while (done < trees) {
    Forest f;
    f.rng.s = ((uint64_t)seeds.next() << 32) | seeds.next();
    const int kind = f.rng.below(4);   // matrices twice as often
    const int root = kind == 1 ? SU3S_VECTOR : kind == 2 ? SU3S_REAL : SU3S_MATRIX;
    const int nf = 1 + f.rng.below(kMaxLeaves);
    f.fields.resize(nf);
    f.values.resize(nf);
    // the first field has the root's kind, a vector tree has a matrix where it can
    for (int i = 0; i < nf; ++i) {
      f.fields[i].kind = root == SU3S_VECTOR && (i & 1) ? (int)SU3S_MATRIX : root;
      for (int k = 0; k < 9; ++k) {
        f.values[i].re[k] = f.rng.next();
        f.values[i].im[k] = root == SU3S_REAL ? 0 : f.rng.next();
      }
    }
    if (root == SU3S_VECTOR && nf < 2) continue;
    const su3s_expr* e = f.tree(2 + f.rng.below(7), root);
    Canon c;
    canon(e, &c);
    c.kind = e->kind;
    int uses = 0;
    for (auto& n : f.nodes) uses += n->op == 0;
    reused += uses > (int)c.leaves.size();
    ++done;
    for (int large = 0; large < 2; ++large) {
      IProg p;
      bool pairs = false;
      if (interp_program(e, c, large != 0, &p, &pairs)) {
        ++refused;
        continue;
      }
      two += pairs;
      if (p.nregs > most) most = p.nregs;
      const std::string bad = check(f, e, c, p, pairs);
      if (!bad.empty()) {
        printf("%s: %s (%s)\n", bad.c_str(), f.text(e).c_str(), pairs ? "two sites per thread" : "one site per thread");
        return 1;
      }
    }
  }
  printf("ok %d trees, %d with a field twice, %d refused, %d for two sites per thread, %d registers at most\n", done,
         reused, refused, two, most);
  return 0;
}

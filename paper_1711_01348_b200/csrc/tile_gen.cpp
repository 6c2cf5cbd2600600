// Tile programs (tile.h) from the term of a kernel (host only).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <functional>
#include <memory>

#include "gen.h"

namespace tad {

namespace {

constexpr double TILE_COPY = 9, TILE_START = 300, TILE_FIXED = 3500;      // issue slots (schedule)
// Sums of products are pushed inside from here on (us, tile / contractions: sum_k x_ik y_jk + u_ik v_jk, 340 x 340 x 340 128 / 25, 1000 x 1000 x 40
// 105 / 18; below, 300 x 200 x 9 and 64 x 64 x 64, a tile 8.3 and 7.3, a point program 38 and 7.4)
constexpr double TILE_APART_LEAST = double(1 << 22);
constexpr int64_t TILE_MIN_SUM = 4;           // fewer terms than this: nothing to share between the values of a tile

// How often a term is written out as a tree, and whether a sum lies at or below an instance
struct Trees {
    std::vector<char> sum_in;
    std::vector<double> nodes;                // (an expression may share a lot)
    void grow(const Gen &g)
    {
        for (int i = (int)nodes.size(); i < (int)g.inst.size(); ++i) {
            const Inst &in = g.inst[i];
            sum_in.push_back(in.op == I_SUM || (in.a >= 0 && sum_in[in.a]) || (in.b >= 0 && sum_in[in.b]));
            nodes.push_back(1 + (in.a >= 0 ? nodes[in.a] : 0) + (in.b >= 0 ? nodes[in.b] : 0));
        }
    }
};

struct Choice { int p, q, l; bool q_sum; double worth; };

// What a kernel sums and over which variables, read off its instances without a change to them
struct Analysis {
    const Gen &g;
    const TadpProgram &prog;
    std::vector<int64_t> lo, ext;
    Trees trees;
    int leaf = -1, term = -1;
    std::vector<int> outer, factors;
    float cfac = 1.f;
    std::vector<Choice> choices;

    Analysis(const Gen &gen, const Kernel &kern) : g(gen), prog(kern.prog), lo(TADP_MAX_VARS, 0), ext(TADP_MAX_VARS, 1) {}
    bool run(int root, int scale, const std::vector<std::vector<TadpRow>> &lower, const std::vector<std::vector<TadpRow>> &upper);
    int least_steps(const Choice &c) const;
    bool apart() const;
};

struct Tiler {
    Gen g;                                    // (a copy: combined factors become instances of it)
    const TadpProgram &prog;
    const std::vector<int64_t> &lo, &ext;
    const std::vector<int> &outer, &factors;
    const int leaf;
    const float cfac;
    Trees trees;
    int p = -1, q = -1, l = -1;
    bool q_sum = false;
    std::vector<int> z;
    TadtProgram T{};
    std::vector<TadeStep> steps;
    std::vector<int> load_at;                 // load of g -> load of T
    int n_loads = 0, n_code = 0, n_imm = 0;
    std::vector<int> op_inst;

    Tiler(const Analysis &a) : g(a.g), prog(a.prog), lo(a.lo), ext(a.ext), outer(a.outer), factors(a.factors), leaf(a.leaf), cfac(a.cfac), trees(a.trees) {}

    // which of p, q, l an instance varies with
    int cls(int i) const
    {
        const uint32_t d = g.inst[i].deps;
        auto bit = [&](int v) { return v >= 0 && ((d >> v) & 1u) && ext[v] > 1; };
        return (bit(p) ? 1 : 0) | (bit(q) ? 2 : 0) | (bit(l) ? 4 : 0);
    }
    bool add_load(int id)
    {
        if ((int)load_at.size() < (int)g.loads.size()) load_at.resize(g.loads.size(), -1);
        if (load_at[id] >= 0) return true;
        if (n_loads >= TADT_LOADS) return false;
        const TadpLoad &L = g.loads[id];
        TadtLoad t{};
        int64_t base = L.base, mn = L.base, mx = L.base;
        for (int v = 0; v < TADP_MAX_VARS; ++v) {
            if (!L.coef[v]) continue;
            const int64_t first = (int64_t)L.coef[v] * lo[v], span = (int64_t)L.coef[v] * (ext[v] - 1);
            base += first;
            mn += first + std::min<int64_t>(0, span); mx += first + std::max<int64_t>(0, span);
            if (ext[v] == 1) continue;
            if (v == p) t.cp = L.coef[v];
            else if (v == q) t.cq = L.coef[v];
            else if (v == l) t.cl = L.coef[v];
            else {
                const auto it = std::find(z.begin(), z.end(), v);
                if (it == z.end()) return false;
                t.cz[it - z.begin()] = L.coef[v];
            }
        }
        // every offset the kernel can form must lie inside the tensor
        if (mn < 0 || mx >= L.limit) return false;
        t.ptr = L.ptr; t.base = to_i32(base);
        load_at[id] = n_loads;
        T.loads[n_loads++] = t;
        return true;
    }
    // appends the program of an instance; sum: the instance that stands for the finished sum
    bool program(int i, int sum, int32_t &at, int32_t &n)
    {
        std::vector<TadeStep> st;
        trees.grow(g);
        if (trees.nodes[i] > 4 * TADT_STEPS || !elementwise_steps_of(g, i, st, sum)) return false;
        at = (int32_t)steps.size();
        for (TadeStep &s : st) {
            if (s.op == E_LD && s.a >= 0) { if (!add_load(s.a)) return false; s.a = (int16_t)load_at[s.a]; }
            steps.push_back(s);
        }
        n = (int32_t)st.size();
        return (int)steps.size() <= TADT_STEPS;
    }

    // ---- operands ----
    int kind_of(int i) const
    {
        const int c = cls(i);
        if (c == 2 && q_sum) return TK_COL;                   // (another one for every tile)
        return c == 4 || c == 5 ? TK_ROW : c == 6 ? TK_COL : c == 2 ? TK_COLC : c == 3 ? TK_MAT : TK_ROWC;
    }
    bool is_operand(int i) const { return cls(i) != 7 && !trees.sum_in[i]; }
    // c times powers of loads
    bool monomial(int i, int e, double &c, std::vector<std::pair<int, int>> &powers) const
    {
        const Inst &in = g.inst[i];
        switch (in.op) {
        case I_LOAD:
            for (auto &pw : powers) if (pw.first == in.load) return false;
            powers.push_back({in.load, e});
            if (powers.size() == 2 && powers[1].second > 1) std::swap(powers[0], powers[1]);
            return powers.size() <= 2;
        case I_MULC: if (e != 1) return false; c *= in.imm; return monomial(in.a, e, c, powers);
        case I_NEG: if (e != 1) return false; c = -c; return monomial(in.a, e, c, powers);
        case I_SQR: return e == 1 && monomial(in.a, 2, c, powers);
        case I_POWI: return e == 1 && in.ipow == 3 && monomial(in.a, 3, c, powers);
        case I_MUL: return e == 1 && monomial(in.a, 1, c, powers) && monomial(in.b, 1, c, powers);
        default: return false;
        }
    }
    int operand(int i)
    {
        for (size_t o = 0; o < op_inst.size(); ++o) if (op_inst[o] == i) return (int)o;
        if ((int)op_inst.size() >= TADT_OPS) return -1;
        TadtOperand O{};
        O.kind = (int16_t)kind_of(i);
        for (int o : op_inst) if (O.kind == TK_MAT && kind_of(o) == TK_MAT) return -1;      // one in registers
        O.load1 = -1; O.e = 1; O.c = 1.f;
        std::vector<std::pair<int, int>> powers;                 // (load, exponent)
        double cf = 1;
        if (O.kind != TK_MAT && trees.nodes[i] < 16 && monomial(i, 1, cf, powers) && (powers.size() == 1 || (powers.size() == 2 && powers[1].second == 1))) {
            for (auto &pw : powers) if (!add_load(pw.first)) return -1;
            O.load0 = (int16_t)load_at[powers[0].first]; O.e = (int16_t)powers[0].second; O.c = (float)cf;
            if (powers.size() == 2) O.load1 = (int16_t)load_at[powers[1].first];
        } else {
            int32_t at, n;
            if (!program(i, -1, at, n)) return -1;
            O.step0 = (int16_t)at; O.n_steps = (int16_t)n;
        }
        if (O.kind == TK_ROW || O.kind == TK_COL) {
            // the order in which a tile is staged: along what is consecutive in the largest tensor it reads
            const TadtLoad *big = nullptr;
            std::vector<int> st{i};
            while (!st.empty()) {
                const Inst &c = g.inst[st.back()];
                st.pop_back();
                if (c.op == I_LOAD) {
                    const TadtLoad &L = T.loads[load_at[c.load]];
                    const int cv = O.kind == TK_ROW ? L.cp : L.cq, bv = !big ? 0 : O.kind == TK_ROW ? big->cp : big->cq;
                    if (!big || (cv != 0 && L.cl != 0 && (bv == 0 || big->cl == 0))) big = &L;
                }
                if (c.a >= 0) st.push_back(c.a);
                if (c.b >= 0) st.push_back(c.b);
            }
            const int cv = !big ? 0 : O.kind == TK_ROW ? big->cp : big->cq;
            O.along_l = big && big->cl != 0 && std::abs(big->cl) <= (cv == 0 ? 1 : std::abs(cv)) ? 1 : 0;
        }
        T.op[op_inst.size()] = O;
        op_inst.push_back(i);
        return (int)op_inst.size() - 1;
    }

    // ---- the core ----
    bool code(int op, int o = 0, int o2 = 0)
    {
        if (o < 0 || o2 < 0 || n_code >= 8) return false;
        T.core |= tadt_step(op, o, o2) << (8 * n_code++);
        return true;
    }
    bool imm_step(int op, float v)
    {
        if (n_imm >= 4) return false;
        T.imm[n_imm] = v;
        return code(op, n_imm++);
    }
    // values that the evaluation of i holds at once: operands are read in one step, also where they are subtracted
    int need(int i) const { return values_held(g, i, [this](int j) { return is_operand(j); }, true); }
    // the operand that comes first when both are: what stays in registers, rows, columns
    bool before(int a, int b) const
    {
        auto rank = [&](int i) { const int c = kind_of(i); return c == TK_MAT ? 0 : c == TK_ROW ? 1 : c == TK_COL ? 2 : 3; };
        return rank(a) <= rank(b);
    }
    bool emit(int i)
    {
        if (is_operand(i)) return code(T_LD, operand(i));
        const Inst in = g.inst[i];
        auto fn = [&](int f) { return emit(in.a) && code(T_FN, f & 3, f >> 2); };
        switch (in.op) {
        case I_NEG: return emit(in.a) && code(T_NEG);
        case I_SQR: return emit(in.a) && code(T_SQR);
        case I_MULC: return emit(in.a) && imm_step(T_MULC, in.imm);
        case I_ADDC: return emit(in.a) && imm_step(T_ADDC, in.imm);
        case I_POWI: return in.ipow == 3 && emit(in.a) && code(T_CUBE);
        case I_EXP: return fn(F_EXP);
        case I_LOG: return fn(F_LOG);
        case I_SIN: return fn(F_SIN);
        case I_COS: return fn(F_COS);
        case I_TANH: return fn(F_TANH);
        case I_SINH: return fn(F_SINH);
        case I_COSH: return fn(F_COSH);
        case I_ADD: case I_MUL: {
            int a = in.a, b = in.b;
            if (is_operand(a) && is_operand(b) ? before(b, a) && !before(a, b) : is_operand(a)) std::swap(a, b);
            // (a is what is evaluated into X; b an operand, or evaluated with a kept in Y)
            if (is_operand(b)) {
                if (!emit(a)) return false;
                const int o = operand(b);
                // X * o + o2 in one step
                const int last = n_code > 0 ? (int)(T.core >> (8 * (n_code - 1))) & 255 : 0;
                if (in.op == I_ADD && (last & 15) == T_MUL && (last >> 6) == 0 && o >= 0) {
                    T.core &= ~(uint64_t(255) << (8 * --n_code));
                    return code(T_FMA, (last >> 4) & 3, o);
                }
                return code(in.op == I_ADD ? T_ADD : T_MUL, o);
            }
            if (need(a) < need(b)) std::swap(a, b);
            if (need(a) > 2 || need(b) != 1) return false;
            return emit(a) && code(T_PUSH) && emit(b) && code(T_BINY, in.op == I_ADD ? 0 : 2);
        }
        case I_SUB:
            if (is_operand(in.b)) {
                // a - b as a + (-b), -b staged: the same sum, and the cores that are built cover differences too
                if (std::find(op_inst.begin(), op_inst.end(), in.b) != op_inst.end()) return emit(in.a) && code(T_SUB, operand(in.b));
                const int minus = g.neg(in.b);
                trees.grow(g);
                if (is_operand(in.a) && before(minus, in.a) && !before(in.a, minus)) return code(T_LD, operand(minus)) && code(T_ADD, operand(in.a));
                return emit(in.a) && code(T_ADD, operand(minus));
            }
            if (is_operand(in.a)) return emit(in.b) && code(T_RSUB, operand(in.a));
            return need(in.a) <= 2 && need(in.b) == 1 && emit(in.a) && code(T_PUSH) && emit(in.b) && code(T_BINY, 1);
        case I_DIV:
            return need(in.a) <= 2 && need(in.b) == 1 && emit(in.a) && code(T_PUSH) && emit(in.b) && code(T_BINY, 3);
        default: return false;
        }
    }

    bool build(int root, int scale, const Choice &c);
    void schedule();
    double slots = 0;                         // estimate of schedule()
};

// the sum, its factors, and which variables can be p, q and l, the most promising choice first
bool Analysis::run(int root, int scale, const std::vector<std::vector<TadpRow>> &lower, const std::vector<std::vector<TadpRow>> &upper)
{
    trees.grow(g);
    for (int v = 0; v < g.n_outer; ++v) { lo[v] = prog.outer_lo[v]; ext[v] = prog.outer_ext[v]; if (ext[v] < 1) return false; }
    std::vector<int> sums;
    for (int c = 0; c < g.kappa; ++c) {
        int64_t a = INT64_MIN, b = INT64_MAX;
        for (const std::vector<TadpRow> *rows : {&lower[c], &upper[c]})
            for (const TadpRow &r : *rows) {
                for (int v = 0; v < TADP_MAX_VARS; ++v) if (r.coef[v]) return false;
                if (rows == &lower[c]) a = std::max(a, ceil_div(r.c0, r.den)); else b = std::min(b, floor_div(r.c0, r.den));
            }
        if (a == INT64_MIN || b == INT64_MAX || b < a) return false;
        const int v = g.n_outer + g.zorder[c];
        lo[v] = a; ext[v] = b - a + 1;
        sums.push_back(v);
    }
    // ---- the sum: the loops around the term, or the one sum inside an element-wise expression ----
    term = root;
    if (g.kappa == 0) {
        if (scale >= 0 || trees.nodes[root] > 1000) return false;
        bool several = false;
        std::function<void(int)> outermost = [&](int i) {
            const Inst &in = g.inst[i];
            if (in.op == I_SUM) { several = several || (leaf >= 0 && leaf != i); leaf = i; return; }
            for (int c : {in.a, in.b}) if (c >= 0) outermost(c);
        };
        outermost(root);
        if (leaf < 0 || several) return false;
        term = leaf;
    }
    while (g.inst[term].op == I_SUM) {
        const Inst &in = g.inst[term];
        if (in.hi < in.lo) return false;
        lo[in.var] = in.lo; ext[in.var] = in.hi - in.lo + 1;
        sums.push_back(in.var);
        term = in.a;
    }
    if (trees.sum_in[term] || trees.nodes[term] > 1000) return false;
    for (int v = 0; v < g.n_outer; ++v) if (ext[v] > 1) outer.push_back(v);
    sums.erase(std::remove_if(sums.begin(), sums.end(), [&](int v) { return ext[v] == 1; }), sums.end());
    for (int v : sums) if (!(g.inst[term].deps & (1u << v))) return false;
    // ---- factors of the term ----
    {
        std::vector<int> todo{term};
        while (!todo.empty()) {
            const int i = todo.back(); todo.pop_back();
            const Inst &in = g.inst[i];
            if (in.op == I_MUL) { todo.push_back(in.a); todo.push_back(in.b); }
            else if (in.op == I_MULC) { cfac *= in.imm; todo.push_back(in.a); }
            else if (in.op == I_NEG) { cfac = -cfac; todo.push_back(in.a); }
            else factors.push_back(i);
        }
    }
    auto out_step = [&](int v) { return prog.out_coef[v] ? std::abs((int64_t)prog.out_coef[v]) : INT64_MAX; };
    auto couples = [&](int a, int b, int c) { for (int f : factors) { const uint32_t d = g.inst[f].deps; if ((d >> a & 1u) && (d >> b & 1u) && (d >> c & 1u)) return true; } return false; };
    if (sums.size() == 1 && ext[sums[0]] >= TILE_MIN_SUM && (int)outer.size() <= 2 + TADT_Z) {
        // two output variables, the larger ones first; the output is written along q
        for (size_t i = 0; i < outer.size(); ++i)
            for (size_t j = i + 1; j < outer.size(); ++j) {
                const int a = outer[i], b = outer[j];
                const bool flip = out_step(a) < out_step(b);
                if (couples(a, b, sums[0])) choices.push_back({flip ? b : a, flip ? a : b, sums[0], false, (double)ext[a] * (double)ext[b]});
            }
    } else if (sums.size() == 2 && (int)outer.size() <= 1 + TADT_Z) {
        // one output variable; l is the sum that leaves most of the factors outside (the largest tensor is then read once)
        for (int i = 0; i < 2; ++i)
            for (int a : outer) {
                if (ext[sums[i]] < TILE_MIN_SUM || !couples(a, sums[0], sums[1])) continue;
                double outside = 0;
                for (int f : factors) {
                    const uint32_t d = g.inst[f].deps;
                    if ((d >> sums[i]) & 1u) continue;
                    double n = 1;
                    for (int v = 0; v < TADP_MAX_VARS; ++v) if ((d >> v) & 1u) n *= (double)ext[v];
                    outside += n;
                }
                choices.push_back({a, sums[1 - i], sums[i], true, outside * 1e9 + (double)ext[a]});
            }
    }
    choices.erase(std::remove_if(choices.begin(), choices.end(), [&](const Choice &c) { return least_steps(c) > 8; }), choices.end());
    std::stable_sort(choices.begin(), choices.end(), [](const Choice &a, const Choice &b) { return a.worth > b.worth; });
    return !choices.empty();
}

// Steps that the core takes at least: one for what couples the three variables, but for a sum behind a product; the first load, the sum
int Analysis::least_steps(const Choice &c) const
{
    const uint32_t all = 1u << c.p | 1u << c.q | 1u << c.l;
    auto coupled = [&](int i) { return (g.inst[i].deps & all) == all; };
    std::function<int(int)> steps = [&](int i) -> int {
        if (!coupled(i)) return 0;
        const Inst &in = g.inst[i];
        if (in.a < 0 || (in.op == I_POWI && in.ipow != 3)) return 99;
        if (in.b < 0) return 1 + steps(in.a);
        int own = in.op == I_DIV ? 2 : 1;
        if (in.op == I_ADD && coupled(in.a) != coupled(in.b)) {
            const Inst &m = g.inst[coupled(in.a) ? in.a : in.b];
            if (m.op == I_MUL && coupled(m.a) != coupled(m.b)) own = 0;
        }
        return own + steps(in.a) + steps(in.b);
    };
    int n = 2;
    for (int f : factors) n += steps(f);
    return n;
}

// A sum of rounded values (products of loads, functions) and at most one exact one (a load, a constant): nothing would be multiplied out
// to push the summation inside, and each part's sum carries the rounding errors that the term has.  Exact values that nearly cancel
// leave none in the term but all of theirs in the parts (a + 10 and b - 10, 300 x 300 x 300, error against 64 bits: (a + b)^2 as written 4e-8, in
// parts 5e-5; the gradients of (a - b)^3 1e-7 and 7e-5).
bool Analysis::apart() const
{
    std::function<bool(int)> product = [&](int i) -> bool {
        const Inst &in = g.inst[i];
        if (in.op == I_MUL) return product(in.a) && product(in.b);
        if (in.op == I_MULC || in.op == I_NEG || in.op == I_SQR || in.op == I_POWI) return product(in.a);
        return in.op != I_ADD && in.op != I_SUB && in.op != I_ADDC && in.op != I_SUM;
    };
    int exact = 0;
    std::function<bool(int)> sum = [&](int i) -> bool {
        const Inst &in = g.inst[i];
        if (in.op == I_ADD || in.op == I_SUB) return sum(in.a) && sum(in.b);
        if (in.op == I_ADDC) ++exact;
        if (in.op == I_ADDC || in.op == I_MULC || in.op == I_NEG) return sum(in.a);
        exact += in.op == I_LOAD || in.op == I_CONST;
        return product(i);
    };
    return sum(term) && exact <= 1;
}

bool Tiler::build(int root, int scale, const Choice &choice)
{
    p = choice.p; q = choice.q; l = choice.l; q_sum = choice.q_sum;
    for (int v : outer) if (v != p && v != q) z.push_back(v);
    // ---- factors: outside the sum over l (q summed), rows, columns, the core ----
    std::vector<int> post, rows, cols, core;
    bool coupled = false;
    for (int f : factors) {
        const int c = cls(f);
        coupled = coupled || c == 7;
        if (q_sum && !(c & 4)) post.push_back(f);
        else if (c == 5 || c == 4) rows.push_back(f);
        else if (c == 6) cols.push_back(f);
        else core.push_back(f);
    }
    if (!coupled) return false;                               // a product of operands: a contraction
    auto product = [&](const std::vector<int> &fs) { int r = fs[0]; for (size_t i = 1; i < fs.size(); ++i) r = g.bin(I_MUL, r, fs[i]); return r; };
    int body = product(core);
    if (!cols.empty() && !rows.empty()) body = g.bin(I_MUL, body, product(cols));
    int last = !rows.empty() ? product(rows) : !cols.empty() ? product(cols) : -1;
    const bool outside = q_sum && !post.empty();              // a constant factor goes where it costs nothing
    if (last >= 0 && !outside) last = g.mulc(last, cfac);
    trees.grow(g);
    if (is_operand(body) || need(body) > 2 || !emit(body)) return false;
    if (cfac != 1.f && !outside && last < 0 && !imm_step(T_MULC, cfac)) return false;
    if (last >= 0 ? !code(T_ACC, operand(last), 1) : !code(T_ACC)) return false;
    if (outside && !program(g.mulc(product(post), cfac), -1, T.post0, T.n_post)) return false;
    // ---- from the sum to the output ----
    T.epi0 = (int32_t)steps.size();
    if (g.kappa == 0) {
        if (!program(root, leaf, T.epi0, T.n_epi)) return false;
    } else {
        if (scale >= 0 && !program(scale, -1, T.epi0, T.n_epi)) return false;
        TadeStep s{};
        s.op = E_LD; s.a = TADT_SUM; s.b = scale >= 0 ? 2 : 0;
        steps.push_back(s);
        ++T.n_epi;
    }
    if ((int)steps.size() > TADT_STEPS) return false;
    std::copy(steps.begin(), steps.end(), T.steps);
    // neither the tail nor the factors outside vary with l, nor the tail of summed columns with q
    for (int s = 0; s < (int)steps.size(); ++s) {
        const bool tail = s >= T.epi0, factor = T.n_post && s >= T.post0 && s < T.post0 + T.n_post;
        if ((!tail && !factor) || steps[s].op != E_LD || steps[s].a < 0) continue;
        const TadtLoad &L = T.loads[steps[s].a];
        if (L.cl || (q_sum && tail && L.cq)) return false;
    }
    // ---- the output ----
    int64_t obase = prog.out_base, mn = prog.out_base, mx = prog.out_base;
    for (int v = 0; v < g.n_outer; ++v) {
        const int64_t first = (int64_t)prog.out_coef[v] * lo[v], span = (int64_t)prog.out_coef[v] * (ext[v] - 1);
        obase += first;
        mn += first + std::min<int64_t>(0, span); mx += first + std::max<int64_t>(0, span);
        if (ext[v] == 1) continue;
        if (v == p) T.out_cp = prog.out_coef[v];
        else if (v == q) T.out_cq = prog.out_coef[v];
        else T.out_cz[std::find(z.begin(), z.end(), v) - z.begin()] = prog.out_coef[v];
    }
    if (mn < 0 || mx >= prog.out_limit) return false;
    T.out_base = to_i32(obase);
    T.accumulate = prog.accumulate;
    T.p_ext = to_i32(ext[p]); T.q_ext = to_i32(ext[q]); T.l_ext = to_i32(ext[l]);
    for (int d = 0; d < TADT_Z; ++d) T.z_ext[d] = d < (int)z.size() ? to_i32(ext[z[d]]) : 1;
    T.q_sum = q_sum ? 1 : 0;
    T.n_loads = n_loads; T.n_ops = (int32_t)op_inst.size();
    for (int o = 0; o < T.n_ops; ++o) { T.n_rows += T.op[o].kind == TK_ROW; T.n_cols += T.op[o].kind == TK_COL; }
    auto kinds = [&](std::initializer_list<int> want) {
        int o = 0;
        for (int kd : want) { if (o >= T.n_ops || T.op[o].kind != kd) return false; ++o; }
        return o == T.n_ops;
    };
    if (T.core == TADT_SQUARES && kinds({TK_ROW, TK_COL})) T.path = 1;
    else if (T.core == TADT_SQUARES_FMA && kinds({TK_ROW, TK_COL, TK_ROWC, TK_ROW}) && !q_sum) T.path = 2;
    else if (T.core == TADT_WEIGHTED && kinds({TK_MAT, TK_COL, TK_ROW}) && !q_sum) T.path = 3;
    schedule();
    return T.n_blocks > 0;
}

// Tile, groups and shares with the least estimated time.  A thread's values cost their multiply-adds (about thirty issue slots
// a step where the core is read step by step), the staging about nine issue slots an element of every operand, both shared by
// the blocks that are resident; a block by itself is bound by its start, its copies and the sums of groups and shares.
void Tiler::schedule()
{
    double best = -1;
    TadtProgram pick = T;
    for (int tm : {4, 8})
    for (int ct = 1; ct <= 32; ++ct)
        for (int rt = 1; rt <= 32; rt *= 2) {
            if ((tm == 8 && !T.path) || ct * rt > TADT_NT || (ct > 8 && ct % 4)) continue;
            const int bm = tm * rt, bn = 4 * ct;
            if (bm / 2 >= T.p_ext || 4 * (ct - 1) >= T.q_ext || bm > 128) continue;      // a smaller one would do
            for (int lg = TADT_NT / (ct * rt); lg >= 1; lg = lg > 1 ? 1 : 0)
            for (int shares : {1, TADT_SHARES}) {
                if (lg * ct * rt < 128) continue;
                TadtProgram c = T;
                c.tm = tm; c.ct = ct; c.rt = rt; c.lg = lg; c.shares = shares;
                c.ct_mul = (uint32_t)((65536 + ct - 1) / ct); c.rt_mul = (uint32_t)((65536 + rt - 1) / rt);
                c.tiles_p = (T.p_ext + bm - 1) / bm; c.tiles_q = (T.q_ext + bn - 1) / bn;
                const double blocks = (double)c.tiles_p * (T.q_sum ? 1 : c.tiles_q) * T.z_ext[0] * T.z_ext[1];
                if (blocks * shares >= 2147483647.0) continue;
                if (shares > 1 && (T.q_sum ? c.tiles_q < 2 : T.l_ext < 2 * shares)) continue;
                const int l_per = T.q_sum ? T.l_ext : (T.l_ext + shares - 1) / shares;
                const int q_per = T.q_sum ? (c.tiles_q + shares - 1) / shares : 1;
                // the longest piece that leaves room for another one; one that holds all of l needs none
                const auto bytes = [&](int chunk, int buffers) {
                    size_t held = 0;
                    for (int o = 0; o < T.n_ops; ++o) held += T.op[o].kind == TK_ROWC ? (size_t)bm : T.op[o].kind == TK_COLC ? (size_t)bn : 0;
                    return 4 * std::max((size_t)buffers * chunk * (T.n_rows * (size_t)(bm + 4) + T.n_cols * (size_t)(bn + 4)) + held,
                                        (size_t)TADT_NT * tm * (T.q_sum ? 1 : 4));
                };
                c.chunk = l_per; c.buffers = T.q_sum ? 2 : 1;
                if (l_per > 256 || bytes(l_per, c.buffers) > TADT_SMEM) {
                    c.buffers = 2; c.chunk = 256;
                    while (c.chunk > 4 && (c.chunk >= l_per || bytes(c.chunk, 2) > TADT_SMEM)) c.chunk /= 2;
                }
                c.smem = (int32_t)bytes(c.chunk, c.buffers);
                if (c.smem > TADT_SMEM) continue;
                const double pieces = std::ceil((double)l_per / c.chunk);
                // issue slots of a warp, eight warps on four schedulers
                const double slots = 4.0 * tm, per_value = T.path == 1 || T.path == 3 ? 2 * slots + 5 : T.path == 2 ? 4 * slots + 8 : 30.0 * n_code;
                const double arith = pieces * std::ceil((double)c.chunk / lg) * per_value;
                const double copies = ((double)T.n_rows * bm / (T.q_sum && pieces == 1 ? q_per : 1) + (double)T.n_cols * bn) * l_per / TADT_NT * TILE_COPY;
                const double tail = T.q_sum ? 4 * slots : (T.n_epi * 2.5 + 6) * slots / (lg * shares);
                const double per_tile = 2 * (arith + copies + tail) * q_per + 2 * pieces * q_per * (100 + 60 * T.n_ops) + (T.q_sum ? 1400.0 * q_per : 0);    // (a tile's factor is waited for)
                const double fixed = TILE_FIXED + (shares > 1 ? 1500 : 0) + (lg > 1 ? 300 + lg * 12 : 0);
                // a block alone on its SM issues in about half of its slots, two in three quarters; clusters leave some SMs to one
                const double total = blocks * shares, room = shares > 1 ? 264 : 296, cost = 2 * TILE_START + per_tile;
                const double time = fixed + cost * (total <= room / 2 ? 1.8 : total <= 4 * room ? 2.7 * std::ceil(total / room) : 2.7 * (total / room + 0.5));
                if (best < 0 || time < best) { best = time; pick = c; pick.n_blocks = (int32_t)blocks; }
            }
        }
    T = pick;
    slots = best;
}

}  // namespace

std::string tile_listing(const TadtProgram &T)
{
    static const char *const core[] = {"END", "LD", "ADD", "SUB", "RSUB", "MUL", "FMA", "SQR", "CUBE", "NEG", "MULC", "ADDC", "PUSH", "BINY", "FN", "ACC"};
    static const char *const steps[] = {"END", "LD", "PUSH", "CONST", "NEG", "SQR", "CUBE", "MULC", "ADDC", "ADDY", "SUBY", "MULY", "DIVY", "FN"};
    static const char *const kinds[] = {"ROW", "COL", "ROWC", "COLC", "MAT"};
    std::string text;
    char line[160];
    auto add = [&](auto... v) { std::snprintf(line, sizeof line, v...); text += line; };
    for (int i = 0; i < T.n_loads; ++i)
        add(";   load %d ptr=%d base=%d p=%d q=%d l=%d z=%d,%d\n", i, T.loads[i].ptr, T.loads[i].base, T.loads[i].cp, T.loads[i].cq, T.loads[i].cl, T.loads[i].cz[0], T.loads[i].cz[1]);
    for (int i = 0; i < T.n_ops; ++i) {
        const TadtOperand &o = T.op[i];
        if (o.n_steps) add(";   operand %d %s steps=%d+%d\n", i, kinds[o.kind], o.step0, o.n_steps);
        else add(";   operand %d %s %.9g load %d ^ %d load %d\n", i, kinds[o.kind], o.c, o.load0, o.e, o.load1);
    }
    for (uint64_t c = T.core; c; c >>= 8) {
        const int op = (int)c & 15, o = (int)(c >> 4) & 3;
        add(";   core %s %d %d %.9g\n", core[op], o, (int)(c >> 6) & 3, op == T_MULC || op == T_ADDC ? T.imm[o] : 0.f);
    }
    const int last = std::max({T.epi0 + T.n_epi, T.post0 + T.n_post, [&] { int n = 0; for (int i = 0; i < T.n_ops; ++i) n = std::max(n, T.op[i].step0 + T.op[i].n_steps); return n; }()});
    for (int i = 0; i < last; ++i) add(";   step %d %s %d %d %.9g\n", i, steps[T.steps[i].op], T.steps[i].a, T.steps[i].b, T.steps[i].imm);
    add(";   post=%d+%d tail=%d+%d out base=%d p=%d q=%d z=%d,%d of %d,%d accumulate=%d\n", T.post0, T.n_post, T.epi0, T.n_epi, T.out_base, T.out_cp, T.out_cq,
        T.out_cz[0], T.out_cz[1], T.z_ext[0], T.z_ext[1], T.accumulate);
    return text;
}

bool try_tile(Gen &g, Kernel &k, int root, int scale, const std::vector<std::vector<TadpRow>> &lower, const std::vector<std::vector<TadpRow>> &upper,
              const std::vector<TadpRow> &guards, double min_space, double max_space, bool may_factor, TileElse &other, std::vector<Kernel> &spare)
{
    other = TILE_NO_OTHER;
    if (g.p.opt.debug_bounds || root < 0 || !guards.empty()) return false;
    // the number of points, ahead of any work: the outputs, loops with fixed ranges, one sum inside the term
    double points = 1, outs = 1;
    for (int v = 0; v < g.n_outer; ++v) outs *= (double)std::max(1, k.prog.outer_ext[v]);
    points = outs;
    for (int c = 0; c < g.kappa; ++c) {
        int64_t a = INT64_MIN, b = INT64_MAX;
        for (const TadpRow &r : lower[c]) a = std::max(a, ceil_div(r.c0, r.den));
        for (const TadpRow &r : upper[c]) b = std::min(b, floor_div(r.c0, r.den));
        for (const std::vector<TadpRow> *rows : {&lower[c], &upper[c]})
            for (const TadpRow &r : *rows) for (int v = 0; v < TADP_MAX_VARS; ++v) if (r.coef[v]) return false;
        if (a == INT64_MIN || b == INT64_MAX || b < a) return false;
        points *= (double)(b - a + 1);
    }
    for (const Inst &in : g.inst) if (in.uses && in.op == I_SUM) points *= (double)std::max<int64_t>(1, in.hi - in.lo + 1);
    if (points < min_space || points > max_space) return false;
    Analysis all(g, k);
    if (!all.run(root, scale, lower, upper)) return false;
    if (may_factor && points > TILE_APART_LEAST && all.apart()) other = TILE_APART;
    std::unique_ptr<Tiler> found;
    for (const Choice &c : all.choices) {
        found.reset(new Tiler(all));
        if (found->build(root, scale, c)) break;
        found.reset();
    }
    if (!found) { other = TILE_NO_OTHER; return false; }
    const Tiler &t = *found;
    // Taken where it is estimated to be faster than what else would run it.  Microseconds of a tile program, fitted to 840 kernels of 2 to
    // 5000 rows, columns and terms (of the estimate / measured 90 % lie between 0.63 and 1.36); of a point program, see point_time.  A
    // built core is given twice that, the others 15 % more: gradients that are tile programs share a launch.
    // (us, tile / point: 2000 batches of 4 x 4 sums of 8 squares 31 / 9.5, of tanh 42 / 10; tanh, 64 x 64 x 17 7.1 / 6.3 and its gradients 14 / 7.3;
    // tanh, 64 x 1000 x 17 10 / 65.)  Beyond 2^21 outputs the interpreter is at its best, 0.001 ns a point and step, and a tile of which short
    // sums or few rows leave little is not (5 x 3655 x 4 in 149 batches, a sum: 80 / 32).
    const double us = t.T.path ? 1.1 + t.slots / 1275 : std::max(1.0, 0.29 * t.n_code - 4 + t.slots / 700);
    const double steps = 2 + all.trees.nodes[all.term] + (scale >= 0 ? all.trees.nodes[scale] : 0);
    const bool chain = g.kappa == 0 && g.inst[root].op != I_SUM;
    const TadpLoad *big = nullptr;
    for (const TadpLoad &L : g.loads) if (!big || L.limit > big->limit) big = &L;
    bool along = false, across = false;
    for (int v = 0; v < (int)g.vars.size(); ++v) if (std::abs(big->coef[v]) == 1 && all.ext[v] > 1) (v < g.n_outer ? across : along) = true;
    const bool serial = chain && t.T.q_sum && g.inst[all.leaf].hi - g.inst[all.leaf].lo < 3;      // (a short sum of sums stays in its thread)
    if (other == TILE_NO_OTHER && !serial && us > (t.T.path ? 2.0 : 1.15) * point_time(outs, points / outs, steps, chain, g.kappa >= 1, along && !across)) other = TILE_POINTS;
    const bool streams = outs >= double(1 << 21) && us > 4 + 1.2e-6 * t.n_code * points;
    if (other != TILE_NO_OTHER || streams) {
        spare = {k};
        spare[0].tile = {t.T};
        spare[0].prog.zsplit = 1;
        return false;
    }
    k.tile = {t.T};
    k.prog.zsplit = 1;
    k.vec = 0; k.vec_u = 0;
    char line[240];
    std::snprintf(line, sizeof line, "; tile program: %d x %d outputs%s, sums of %d, core %llx%s, tiles of %d x %d, %d groups, %d blocks, %d shares, pieces of %d\n",
                  t.T.p_ext, t.T.q_ext, t.T.q_sum ? " (columns summed)" : "", t.T.l_ext, (unsigned long long)t.T.core, t.T.path ? " (built)" : "",
                  t.T.tm * t.T.rt, 4 * t.T.ct, t.T.lg, t.T.n_blocks, t.T.shares, t.T.chunk);
    k.listing = line;
    return true;
}

}  // namespace tad

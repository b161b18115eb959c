// lower.cpp -- register stages rewritten for the in-place stage engine (lean_stage.cuh).
//
// A plan describes a stage by its sub-ops (DevSub): real 2x2 matrices with two unit entries,
// diagonal tables, controlled phases, X.  The engine wants few kinds of records, each a straight
// run of in-place updates, so the stage is rewritten here, in FP64, without changing what it
// computes (Eq. 2-3 reassociated):
//
//  * complex64: a real 2x2 matrix S with s11 != 0 is D L, L two shears and D a real diagonal:
//      v1 += y v0;  v0 += x v1;   y = s10 / s11,  x = s01 s11 / det,  D = diag(det / s11, s11),
//    two FMAs per pair that overwrite their inputs -- no copy through a temporary, which the
//    unit-entry forms need when both results use both old values.  |s11| >= |s10| is had by
//    exchanging the rows first where it does not hold, and the exchange (an X on that bit) is
//    not executed: from there on the bit is held "flipped" (slot s of the registers holds
//    logical index s ^ F), later sub-ops are written for slots, and the stage stores through
//    addresses XORed with F.  Uncontrolled X gates become such flips too.
//  * complex128: S = s00 [[1, x], [y, +-1]], with the same exchange of rows, two FMAs per pair as well,
//    both from the old values.  The copy through a temporary is free beside FP64 arithmetic, and the
//    factor is the same for both values of the bit, so it needs no multiply of its own.  In
//    double-float form the second shear would round on top of the first and D would round once more:
//    layered circuits of 16 to 22 qubits are 2.0e-14 to 2.7e-14 off so, 2.2e-14 to 3.1e-14 with shears
//    (26 qubits, 12 layers: 37.7 against 36.6 ms).
//  * The factors D are carried along: past a shear pair on the same bit by D^-1 L D (real again,
//    and x y stays the same, so the relative rounding of each update does not change), past
//    everything else freely, until the next diagonal table takes them in.  A stage without a
//    table gets one real scaling at its end.
//  * Phases that can reach a table without crossing a record that does not commute with them
//    join it.
//  * Shear pairs on distinct register bits that can be brought together form one record.
//  * Conditional diagonals whose factor is s(h) prod_j phi_j(h)^(e_j), h the condition bits (CP, RZZ, CZ and
//    what was fused from them), are collected from the plan's unmerged sub-ops at as few places as
//    possible and run as one separable record there: RB + 1 numbers per setting of a group of up to
//    eight conditions instead of 2^RB, so hundreds of conditional phases on dozens of outside bits
//    cost one walk over the register elements.  Tables with that many conditions would not fit, and
//    one table per few of them is what bounded such stages: qaoa23 complex64 826 -> 575 us, qft28
//    complex128 82.6 -> 76.6 ms.
#include "lower.h"

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

namespace qs {

namespace {

// Condition bits up to which a table grows to take in a conditional phase.  A sign costs three
// integer instructions per element as a record of its own; FP32 tables double in size per bit.
// (qs_options.merge_bits limits what is put together here as it does the planner's own tables.)
int limited(const Plan &plan, int bits) { return plan.opt.merge_bits > 0 ? std::min(bits, plan.opt.merge_bits) : bits; }
int table_bits(const Plan &plan) { return limited(plan, plan.dt == QS_C128 && plan.opt.arith == QS_ARITH_FP64 ? 10 : 5); }

// Product of finite numbers (operator* of std::complex also checks for NaN, several times slower).
inline cd mul(const cd &a, const cd &b)
{
    return cd(a.real() * b.real() - a.imag() * b.imag(), a.real() * b.imag() + a.imag() * b.real());
}

// the smallest pattern (lean_stage.cuh: 0 = all, or one value of one bit) that holds all of `elems`
uint32_t active_pattern(uint32_t elems, int RB, int first = 0)
{
    static const uint32_t ones[5] = {0xaaaaaaaau, 0xccccccccu, 0xf0f0f0f0u, 0xff00ff00u, 0xffff0000u};
    for (int j = first; j < RB; ++j) {
        if (!(elems & ones[j])) return 1 + 2 * j;
        if (!(elems & ~ones[j])) return 2 + 2 * j;
    }
    return 0;
}

struct Builder {
    const Plan &plan;
    const int RB, E;
    std::vector<LeanItem> items;
    std::vector<char> small;         // items[i] is a phase that may still join a table
    const bool unit;                 // complex128: unit-entry matrices instead of shears
    uint32_t F = 0;
    double d[6][2];
    bool bad = false;

    Builder(const Plan &p, int rb) : plan(p), RB(rb), E(1 << rb), unit(p.dt == QS_C128)
    {
        items.reserve(32);
        small.reserve(32);
        for (auto &v : d) v[0] = v[1] = 1.0;
    }

    void push(LeanItem it, bool is_small = false)
    {
        items.push_back(std::move(it));
        small.push_back(is_small);
    }
    bool carried() const
    {
        for (int j = 0; j < RB; ++j)
            if (d[j][0] != 1.0 || d[j][1] != 1.0) return true;
        return false;
    }
    double carry(int s) const
    {
        double f = 1.0;
        for (int j = 0; j < RB; ++j) f *= d[j][s >> j & 1];
        return f;
    }
    void reset_carry()
    {
        for (auto &v : d) v[0] = v[1] = 1.0;
    }
    // register bits that tell elements of the set m32 from elements outside it
    uint32_t set_reads(uint32_t m32) const
    {
        static const uint32_t low[5] = {0x55555555u, 0x33333333u, 0x0f0f0f0fu, 0x00ff00ffu, 0x0000ffffu};
        const uint32_t all = E == 32 ? ~0u : (1u << E) - 1u;
        uint32_t r = 0;
        for (int j = 0; j < RB; ++j)
            if ((m32 ^ (m32 >> (1 << j))) & low[j] & all) r |= 1u << j;
        return r;
    }
    uint32_t table_reads(const std::vector<cd> &tab) const
    {
        uint32_t r = 0;
        for (int j = 0; j < RB; ++j)
            for (size_t i = 0; i < tab.size() && !(r >> j & 1); ++i)
                if (tab[i] != tab[i ^ (size_t(1) << j)]) r |= 1u << j;
        return r;
    }
    uint32_t carry_reads() const
    {
        uint32_t r = 0;
        for (int j = 0; j < RB; ++j)
            if (d[j][0] != d[j][1]) r |= 1u << j;
        return r;
    }
    // the carried factors are a separable real diagonal
    void apply_carry_sep(LeanItem &t) const
    {
        std::vector<cd> &tab = t.sep[0].tab;
        for (size_t h = 0; h < tab.size(); h += RB + 1)
            for (int j = 0; j < RB; ++j) {
                tab[h] *= d[j][0];
                tab[h + 1 + j] *= d[j][1] / d[j][0];
            }
        t.rd |= carry_reads();
    }
    // groups in logical indices
    void add_sep(std::vector<SepGroup> groups, uint32_t rd)
    {
        LeanItem t;
        t.op = L_SEP;
        t.rd = rd;
        for (SepGroup &g : groups)
            for (size_t h = 0; h < g.tab.size(); h += RB + 1)
                for (int j = 0; j < RB; ++j)
                    if (F >> j & 1) {  // e_j = 1 - s_j
                        g.tab[h] *= g.tab[h + 1 + j];
                        g.tab[h + 1 + j] = 1.0 / g.tab[h + 1 + j];
                    }
        t.sep = std::move(groups);
        if (carry_reads() || (!unit && carried())) {
            t.lift = lift();
            apply_carry_sep(t);
            reset_carry();
        }
        // single-bit phases and scalars without conditions that can meet it join it
        for (size_t k = items.size(); k-- > 0;) {
            if (!small[k] || items[k].lcm || items[k].ocm) continue;
            bool free = true;
            for (size_t i = k + 1; free && i < items.size(); ++i) free = commutes(items[k].rd, items[i]);
            if (!free || !join_sep(t, items[k])) continue;
            items.erase(items.begin() + k);
            small.erase(small.begin() + k);
        }
        push(std::move(t));
    }
    // Only phases of modulus 1: on a flipped bit the record needs 1 / p, which a projector (p = 0) or a
    // small p does not have; such a diagonal stays a record of its own or goes into a table.
    bool join_sep(LeanItem &t, const LeanItem &ph) const
    {
        if (ph.lcm || ph.ocm || __builtin_popcount(ph.rd) > 1 || !(std::abs(std::norm(ph.p) - 1.0) <= 1e-12)) return false;
        std::vector<cd> &tab = t.sep[0].tab;
        const bool e0 = ph.m32 & 1u;
        for (size_t h = 0; h < tab.size(); h += RB + 1) {
            if (e0) tab[h] *= ph.p;
            if (ph.rd) tab[h + 1 + __builtin_ctz(ph.rd)] *= e0 ? 1.0 / ph.p : ph.p;
        }
        t.rd |= ph.rd;
        return true;
    }
    // a diagonal reading the bits `rd` commutes with the item
    bool commutes(uint32_t rd, const LeanItem &it) const
    {
        if (it.op == L_ROTA) return !(it.mask & rd);
        if (it.op == L_CX) return !(rd >> it.j & 1);
        return true;
    }
    std::vector<uint8_t> conditions(const LeanItem &ph) const
    {
        std::vector<uint8_t> c;
        for (int l = 0; l < 32; ++l)
            if (ph.lcm >> l & 1) c.push_back((uint8_t)l);
        for (int q = 0; q < 64; ++q)
            if (ph.ocm >> q & 1) c.push_back((uint8_t)(0x80 | q));
        return c;
    }
    // the table over more conditions (`dl` begins with those that it has)
    void grow(LeanItem &t, const std::vector<uint8_t> &dl) const
    {
        const size_t n = t.tab.size();
        t.tab.resize(size_t(E) << dl.size());
        for (size_t at = n; at < t.tab.size(); at += n) std::copy_n(t.tab.begin(), n, t.tab.begin() + at);
        t.dl = dl;
    }
    // multiply the phase into the table if its conditions are, or can become, table conditions
    bool join(LeanItem &t, const LeanItem &ph) const
    {
        const std::vector<uint8_t> c = conditions(ph);
        std::vector<uint8_t> dl = t.dl;
        for (uint8_t b : c)
            if (std::find(dl.begin(), dl.end(), b) == dl.end()) dl.push_back(b);
        if (dl.size() > t.dl.size() && (int)dl.size() > table_bits(plan)) return false;
        uint32_t need = 0;
        for (uint8_t b : c) need |= 1u << (std::find(dl.begin(), dl.end(), b) - dl.begin());
        grow(t, dl);
        for (size_t h = need; h < (size_t(1) << dl.size()); h = (h + 1) | need)
            for (int e = 0; e < E; ++e)
                if (ph.m32 >> e & 1) t.tab[(h << RB) | e] = mul(t.tab[(h << RB) | e], ph.p);
        t.rd |= ph.rd;
        return true;
    }
    void add_table(LeanItem t)
    {
        // (a carry that is the same for all elements waits for the stage's end)
        if (carry_reads() || (!unit && carried())) {
            t.lift = lift();
            apply_carry(t);
            reset_carry();
        }
        // phases before it that can move up to here
        for (size_t k = items.size(); k-- > 0;) {
            if (!small[k]) continue;
            const uint32_t rd = items[k].rd;
            bool free = true;
            for (size_t i = k + 1; free && i < items.size(); ++i) free = commutes(rd, items[i]);
            if (free && join(t, items[k])) {
                items.erase(items.begin() + k);
                small.erase(small.begin() + k);
            }
        }
        // a table that it can be moved back to takes it in
        for (size_t k = items.size(); k-- > 0;) {
            if (items[k].op == L_TABLE && merge(items[k], t)) return;
            if (!commutes(t.rd, items[k])) break;
        }
        push(std::move(t));
    }
    // a *= b if their conditions together are few enough
    bool merge(LeanItem &a, const LeanItem &b) const
    {
        std::vector<uint8_t> dl = a.dl;
        for (uint8_t c : b.dl)
            if (std::find(dl.begin(), dl.end(), c) == dl.end()) dl.push_back(c);
        if (dl.size() > std::max(a.dl.size(), b.dl.size()) && (int)dl.size() > table_bits(plan)) return false;
        Lift both = a.lift;
        if (!in_range(both += b.lift)) return false;
        std::vector<int> at(b.dl.size());
        for (size_t j = 0; j < b.dl.size(); ++j) at[j] = int(std::find(dl.begin(), dl.end(), b.dl[j]) - dl.begin());
        grow(a, dl);
        for (size_t h = 0; h < (size_t(1) << dl.size()); ++h) {
            size_t hb = 0;
            for (size_t j = 0; j < at.size(); ++j) hb |= ((h >> at[j]) & 1) << j;
            for (int e = 0; e < E; ++e) a.tab[(h << RB) | e] = mul(a.tab[(h << RB) | e], b.tab[(hb << RB) | e]);
        }
        a.rd |= b.rd;
        a.lift = both;
        return true;
    }
    void apply_carry(LeanItem &t) const
    {
        double f[32];
        for (int s = 0; s < E; ++s) f[s] = carry(s);
        for (size_t i = 0; i < t.tab.size(); ++i) t.tab[i] *= f[i & (E - 1)];
        t.rd |= carry_reads();
    }
    void add_phase(LeanItem ph)
    {
        const uint32_t rd = ph.rd = set_reads(ph.m32);
        for (size_t k = items.size(); k-- > 0;) {
            if (items[k].op == L_TABLE && join(items[k], ph)) return;
            if (items[k].op == L_SEP && join_sep(items[k], ph)) return;
            if (!commutes(rd, items[k])) break;
        }
        push(std::move(ph), true);
    }
    // real 2x2 matrix (logical) on register bit j
    void add_real(int j, double m00, double m01, double m10, double m11)
    {
        double s00 = m00, s01 = m01, s10 = m10, s11 = m11;
        if (F >> j & 1) {
            std::swap(s00, s11);
            std::swap(s01, s10);
        }
        if (std::abs(s11) < std::abs(s10)) {  // hold the result flipped: rows exchanged
            std::swap(s00, s10);
            std::swap(s01, s11);
            F ^= 1u << j;
            if (std::abs(s11) < std::abs(s10)) {
                bad = true;  // both rows have |first| > |second|: not orthogonal
                return;
            }
        }
        if (unit) {
            // (double-float numbers have the range of FP32)
            const double most = plan.opt.arith == QS_ARITH_DF ? 1e18 : 1e100;
            const double r = s00 != 0.0 ? s11 / s00 : 0.0;
            if (!(std::abs(std::abs(r) - 1.0) <= 1e-13)) {
                bad = true;
                return;
            }
            LeanItem it;
            it.op = L_ROTA;
            it.mask = 1u << j;
            it.neg = r < 0 ? 1u << j : 0;
            it.y[j] = s10 / s00;
            it.x[j] = s01 / s00;
            d[j][0] *= s00;
            d[j][1] *= s00;
            push(std::move(it));
            if (!(std::abs(d[j][0]) < most && std::abs(d[j][0]) > 1.0 / most)) flush_carry();
            return;
        }
        const double det = s00 * s11 - s01 * s10;
        auto moderate = [](double v) { return std::abs(v) > 0x1p-30 && std::abs(v) < 0x1p30; };
        if (!moderate(s11) || !moderate(det / s11) || !(std::abs(det) > 1e-6 * s11 * s11)) {
            bad = true;
            return;
        }
        double y = s10 / s11, x = s01 * s11 / det;
        const double r = d[j][0] / d[j][1];
        y *= r;
        x /= r;
        d[j][0] *= det / s11;
        d[j][1] *= s11;
        LeanItem it;
        it.op = L_ROTA;
        it.mask = 1u << j;
        it.y[j] = y;
        it.x[j] = x;
        push(std::move(it));
        // a run of rotations without a table: keep the carried factors near 1
        for (int k = 0; k < 2; ++k)
            if (!(std::abs(d[j][k]) < 4096.0 && std::abs(d[j][k]) > 1.0 / 4096.0)) {
                flush_carry();
                break;
            }
    }
    Lift lift() const
    {
        Lift r;
        r.e[0] = std::ilogb(carry(0));
        for (int j = 0; j < RB; ++j)
            if (d[j][1] != d[j][0]) r.e[1 + j] = std::ilogb(d[j][1] / d[j][0]);
        return r;
    }
    // whether all factors of an item that took these in, and what later records hold instead, stay within FP32 (double-float: also
    // 2^-48 of them, the last bits of a product)
    bool in_range(const Lift &t) const
    {
        int sum = 0;
        for (int v : t.e) sum += std::abs(v);
        return sum < (plan.opt.arith == QS_ARITH_DF ? 40 : 90);
    }
    // The carried diagonal joins the last table it can be moved back to, or becomes a scaling: also where a table
    // that many of them have joined would leave the range of FP32.
    void flush_carry()
    {
        if (!carried()) return;
        size_t t = items.size();
        bool found = false;
        while (t-- > 0) {
            const LeanItem &it = items[t];
            if (it.op == L_TABLE || it.op == L_SEP) {
                found = true;
                break;
            }
            if (it.op == L_CX && d[it.j][0] != d[it.j][1]) break;
        }
        Lift after = lift();
        if (!found || !in_range(after += items[t].lift)) {
            LeanItem sc;
            sc.op = L_SCALE;
            sc.scale.resize(E);
            for (int s = 0; s < E; ++s) sc.scale[s] = carry(s);
            sc.rd = carry_reads();
            reset_carry();
            push(std::move(sc));
            return;
        }
        for (size_t i = t + 1; i < items.size(); ++i)
            if (items[i].op == L_ROTA)
                for (int j = 0; j < RB; ++j)
                    if (items[i].mask >> j & 1) {
                        const double r = d[j][0] / d[j][1];
                        items[i].y[j] /= r;  // D L = (D L D^-1) D
                        items[i].x[j] *= r;
                    }
        items[t].lift = after;
        if (items[t].op == L_SEP) apply_carry_sep(items[t]);
        else apply_carry(items[t]);
        reset_carry();
    }
    // X on register bit j where the conditions hold
    void add_x(int j, int ctrl, uint32_t lcm, uint64_t ocm)
    {
        if (d[j][0] != d[j][1]) flush_carry();
        LeanItem it;
        it.op = L_CX;
        it.j = j;
        it.ctrl = ctrl;
        it.lcm = lcm;
        it.ocm = ocm;
        push(it);
    }
    void add_sub(const DevSub &sb)
    {
        const cd *M = plan.coef.data() + sb.mat;
        const bool ctl = (sb.scm | sb.lcm | sb.ocm) != 0;
        switch (sb.type) {
        case SB_G1N: add_real(sb.j0, 1.0, M[0].real(), M[1].real(), 1.0); break;
        case SB_G1NM: add_real(sb.j0, 1.0, M[0].real(), M[1].real(), -1.0); break;
        case SB_G1A: add_real(sb.j0, M[0].real(), 1.0, 1.0, M[1].real()); break;
        case SB_G1AM: add_real(sb.j0, M[0].real(), 1.0, -1.0, M[1].real()); break;
        case SB_G1R:  // (factor = 1 keeps full matrices, euler = 1 complex ones: the general engine's)
            if (ctl || plan.opt.factor == 1) bad = true;
            else add_real(sb.j0, M[0].real(), M[1].real(), M[2].real(), M[3].real());
            break;
        case SB_G1: {
            // complex 2x2: phase, real rotation, phase (the planner's Z-Y-Z form)
            const double c = std::abs(M[0]), s = std::abs(M[2]);
            if (ctl || plan.opt.factor == 1 || plan.opt.euler == 1 || c < 1e-6 || s < 1e-6) {
                bad = true;
                break;
            }
            const cd g = M[0] / c, eb = M[2] / (g * s), ed = -M[1] / (g * s);
            const double tol = split_tolerance(plan.dt);
            const bool unitary = std::abs(std::abs(eb) - 1.0) <= tol && std::abs(std::abs(ed) - 1.0) <= tol;
            if (!unitary || std::abs(M[3] - g * eb * ed * c) > tol * c || std::abs(c * c + s * s - 1.0) > 1e-12) {
                bad = true;
                break;
            }
            add_bit_phase(sb.j0, ed);
            add_real(sb.j0, c, -s, s, c);
            add_bit_phase(sb.j0, eb);
            LeanItem ph;  // the scalar g
            ph.op = L_PHASE;
            ph.m32 = E == 32 ? ~0u : (1u << E) - 1u;
            ph.p = g;
            add_phase(ph);
            break;
        }
        case SB_X: {
            if (!ctl) {
                F ^= 1u << sb.j0;  // slots keep their values (and the carried diagonal)
                break;
            }
            const int nreg = __builtin_popcount(sb.scm);
            if (nreg > 1) {
                bad = true;
                break;
            }
            const int c = nreg ? __builtin_ctz(sb.scm) : -1;
            add_x(sb.j0, c, sb.lcm, sb.ocm);
            if (c >= 0 && (F >> c & 1)) {
                // the control's slot value is 0: X where the other conditions hold, undone at 1
                if (sb.lcm | sb.ocm) add_x(sb.j0, -1, sb.lcm, sb.ocm);
                else F ^= 1u << sb.j0;
            }
            break;
        }
        case SB_PHASE: {
            const cd p = M[0];
            if (!ctl && p.imag() == 0.0) {
                // (rotations alone stay just beyond 2^-64; matrices scaled further keep their order of factors)
                if (!(std::abs(p.real()) > 0x1p-68 && std::abs(p.real()) < 0x1p68)) {
                    bad = true;
                    break;
                }
                d[0][0] *= p.real();
                d[0][1] *= p.real();
                break;
            }
            LeanItem ph;
            ph.op = L_PHASE;
            for (int s = 0; s < E; ++s)
                if (((uint32_t(s) ^ F) & sb.scm) == sb.scm) ph.m32 |= 1u << s;
            ph.p = p;
            ph.lcm = sb.lcm;
            ph.ocm = sb.ocm;
            add_phase(ph);
            break;
        }
        case SB_DIAG: {
            LeanItem t;
            t.op = L_TABLE;
            t.dl.assign(sb.dl, sb.dl + sb.ndl);
            t.tab.resize(size_t(E) << sb.ndl);
            for (size_t h = 0; h < (size_t(1) << sb.ndl); ++h)
                for (int s = 0; s < E; ++s) t.tab[(h << RB) | s] = M[(h << RB) | (uint32_t(s) ^ F)];
            t.rd = table_reads(t.tab);
            add_table(std::move(t));
            break;
        }
        default: bad = true; break;
        }
    }
    // factors of the logical register elements
    void add_factors(const std::vector<cd> &q)
    {
        LeanItem t;
        t.op = L_TABLE;
        t.tab.resize(E);
        for (int s = 0; s < E; ++s) t.tab[s] = q[uint32_t(s) ^ F];
        t.rd = table_reads(t.tab);
        add_table(std::move(t));
    }
    void add_bit_phase(int j, cd p)
    {
        LeanItem ph;
        ph.op = L_PHASE;
        for (int s = 0; s < E; ++s)
            if ((uint32_t(s) ^ F) >> j & 1) ph.m32 |= 1u << s;
        ph.p = p;
        add_phase(ph);
    }
    bool commute_between(uint32_t rd, size_t i, size_t j) const
    {
        for (; i < j; ++i)
            if (!commutes(rd, items[i])) return false;
        return true;
    }
    // Phases that found no table: those that can meet in one place become a table where that is
    // cheaper.  complex64 runs any complex phase as a table (it takes about as long as one phase of
    // 16 elements, 270 ns); otherwise the multiplies decide (a pattern: half of the elements).
    void gather_phases()
    {
        auto cost = [&](uint32_t elems) { return active_pattern(elems, RB) ? 1 : 2; };
        for (size_t k = 0; k < items.size(); ++k) {
            if (!small[k] || items[k].p == cd(-1.0)) continue;
            LeanItem t;
            t.op = L_TABLE;
            t.tab.assign(E, cd(1.0));
            if (!join(t, items[k])) continue;
            std::vector<size_t> in;
            uint32_t elems = items[k].m32;
            int apart = cost(elems);
            for (size_t j = 0; j < items.size(); ++j) {
                if (j == k || !small[j]) continue;
                const uint32_t rd = items[j].rd;
                const bool sign = items[j].p == cd(-1.0);
                if (!(j > k ? commute_between(rd, k + 1, j) : commute_between(rd, j + 1, k))) continue;
                if (plan.dt != QS_C64 && cost(elems | items[j].m32) > cost(elems) + (sign ? 0 : cost(items[j].m32))) continue;
                if (!join(t, items[j])) continue;
                in.push_back(j);
                elems |= items[j].m32;
                if (!sign) apart += cost(items[j].m32);
            }
            if (plan.dt != QS_C64 && apart <= cost(elems)) continue;
            items[k] = std::move(t);
            small[k] = 0;
            for (size_t i = in.size(); i-- > 0;) {
                items.erase(items.begin() + in[i]);
                small.erase(small.begin() + in[i]);
                if (in[i] < k) --k;
            }
        }
    }
    // tables that can meet become one (shears gathered in front of them may have brought them together)
    void merge_tables()
    {
        for (size_t i = 1; i < items.size(); ++i) {
            if (items[i].op != L_TABLE) continue;
            for (size_t k = i; k-- > 0;) {
                if (items[k].op == L_TABLE && merge(items[k], items[i])) {
                    items.erase(items.begin() + i);
                    --i;
                    break;
                }
                if (!commutes(items[i].rd, items[k])) break;
            }
        }
    }
    // shear pairs on distinct bits that commute with what lies between them form one record
    void group_shears()
    {
        std::vector<LeanItem> out;
        std::vector<char> used(items.size(), 0);
        for (size_t i = 0; i < items.size(); ++i) {
            if (used[i]) continue;
            LeanItem cur = std::move(items[i]);
            if (cur.op == L_ROTA) {
                uint32_t blocked = 0;
                for (size_t k = i + 1; k < items.size(); ++k) {
                    if (used[k]) continue;
                    const LeanItem &it = items[k];
                    if (it.op == L_ROTA) {
                        if (it.mask & (cur.mask | blocked)) {
                            blocked |= it.mask;
                            continue;
                        }
                        const int j = __builtin_ctz(it.mask);
                        cur.mask |= it.mask;
                        cur.y[j] = it.y[j];
                        cur.x[j] = it.x[j];
                        cur.neg |= it.neg;
                        used[k] = 1;
                    } else if (it.op == L_CX) {
                        blocked |= 1u << it.j;
                        if (it.ctrl >= 0) blocked |= 1u << it.ctrl;
                    } else {
                        blocked |= it.rd;
                    }
                }
            }
            out.push_back(std::move(cur));
        }
        items = std::move(out);
    }
};

// ------------------------------------------------------------------ device encoding

template <typename T>
void put(unsigned char *p, size_t off, const T &v)
{
    std::memcpy(p + off, &v, sizeof v);
}

// one real number in the state precision; returns its size in bytes
size_t put_real(unsigned char *p, size_t off, double v, qs_dtype dt, bool df)
{
    if (dt == QS_C64) {
        put(p, off, (float)v);
        return 4;
    }
    if (df) {  // h = fl32(v), l = fl32(v - h)
        const float h = (float)v;
        put(p, off, h);
        put(p, off + 4, (float)(v - (double)h));
    } else {
        put(p, off, v);
    }
    return 8;
}

}  // namespace

namespace {

// A diagonal sub-op as q(e) s(h) prod_j phi_j(h)^(e_j), h its condition bits (logical indices).
struct Separable {
    std::vector<cd> q;        // 2^RB, empty if 1 throughout
    std::vector<uint8_t> dl;
    std::vector<cd> tab;      // (RB + 1) per h
    uint32_t rd = 0;          // register bits the conditional part reads
    bool scalar = false;      // s differs from 1 for some h
    size_t need = 0;          // the factors differ from 1 only where these condition bits hold
};

bool near(const cd &a, const cd &b) { return std::abs(a.real() - b.real()) <= 4e-15 && std::abs(a.imag() - b.imag()) <= 4e-15; }

// (The conjugate would double what a product of many phases is off the unit circle, once per factor.)
cd inverse(const cd &a)
{
    const double n = std::norm(a);
    return cd(a.real() / n, -a.imag() / n);
}

// false: not conditional, not of unit modulus, or not separable
bool separable(const Plan &plan, const DevSub &sb, int RB, Separable &o)
{
    const int E = 1 << RB;
    const cd *M = plan.coef.data() + sb.mat;
    if (sb.type == SB_PHASE) {
        for (int l = 0; l < 32; ++l)
            if (sb.lcm >> l & 1) o.dl.push_back((uint8_t)l);
        for (int x = 0; x < 64; ++x)
            if (sb.ocm >> x & 1) o.dl.push_back((uint8_t)(0x80 | x));
        if (o.dl.empty() || o.dl.size() > 4 || __builtin_popcount(sb.scm) > 1 || std::abs(std::abs(M[0]) - 1.0) > 1e-12) return false;
        const size_t H = size_t(1) << o.dl.size();
        o.tab.assign(H * (RB + 1), cd(1.0));
        o.tab[(H - 1) * (RB + 1) + (sb.scm ? 1 + __builtin_ctz(sb.scm) : 0)] = M[0];
        o.rd = sb.scm;
        o.scalar = sb.scm == 0;
        o.need = H - 1;
        return true;
    }
    if (sb.type != SB_DIAG || sb.ndl == 0) return false;
    const size_t H = size_t(1) << sb.ndl;
    o.dl.assign(sb.dl, sb.dl + sb.ndl);
    o.tab.resize(H * (RB + 1));
    for (size_t i = 0; i < H * E; ++i)
        if (std::abs(std::norm(M[i]) - 1.0) > 1e-12) return false;
    // relative to h = 0, which q takes whole
    bool unit_q = true;
    for (int e = 0; e < E; ++e) unit_q = unit_q && M[e] == cd(1.0);
    if (!unit_q) o.q.assign(M, M + E);
    cd inv[6];
    inv[0] = inverse(M[0]);
    for (int j = 0; j < RB; ++j) inv[1 + j] = inverse(M[1 << j]);
    for (size_t h = 0; h < H; ++h) {
        cd *t = o.tab.data() + h * (RB + 1);
        const cd *m = M + (h << RB);
        t[0] = mul(m[0], inv[0]);
        if (near(t[0], cd(1.0))) t[0] = 1.0;
        else o.scalar = true;
        const cd is = inverse(t[0]);
        for (int j = 0; j < RB; ++j) {
            t[1 + j] = mul(mul(m[1 << j], inv[1 + j]), is);
            if (!near(t[1 + j], cd(1.0))) o.rd |= 1u << j;
            else t[1 + j] = 1.0;
        }
        cd f[32];
        for (int e = 0; e < E; ++e) {
            f[e] = e == 0 ? t[0] : mul(f[e & (e - 1)], t[1 + __builtin_ctz(e)]);
            const cd d = mul(f[e], M[e]) - m[e];
            if (std::norm(d) > 3.6e-29) return false;  // 6e-15: the rounding noise of products of 45 phases stays below
        }
    }
    return true;
}

uint32_t sub_targets(const DevSub &s)
{
    switch (s.type) {
    case SB_PHASE: case SB_DIAG: return 0;
    case SB_G2: case SB_SWAP: return (1u << s.j0) | (1u << s.j1);
    default: return 1u << s.j0;
    }
}

constexpr int kSepBits = 8;      // condition bits per group, at most merge_bits
constexpr size_t kSepGroups = 24;

// The stage with its separable conditional diagonals collected at as few places as possible; each place
// becomes one L_SEP.  Returns false if there is nothing to collect.
bool lower_regrouped(const Plan &plan, const DevSub *sub, int ns, int RB, Builder &b)
{
    struct Cond {
        Separable f;
        int lo, hi, point = -1;
    };
    std::vector<Cond> conds;
    std::vector<int> of_sub(ns, -1), order;
    // a diagonal lies between the non-diagonal subs lo - 1 and hi: the nearest ones on a bit that it reads
    int m = 0, last[6] = {0, 0, 0, 0, 0, 0}, next[6];
    for (int i = 0; i < ns; ++i) {
        if (const uint32_t tg = sub_targets(sub[i])) {
            ++m;
            for (int j = 0; j < RB; ++j)
                if (tg >> j & 1) last[j] = m;
            continue;
        }
        Cond c;
        if (separable(plan, sub[i], RB, c.f)) {
            c.lo = 0;
            for (int j = 0; j < RB; ++j)
                if (c.f.rd >> j & 1) c.lo = std::max(c.lo, last[j]);
            of_sub[i] = (int)conds.size();
            order.push_back(of_sub[i]);
            conds.push_back(std::move(c));
        }
    }
    if (conds.size() < 4) return false;
    for (int &x : next) x = m;
    for (int i = ns, k = m; i-- > 0;) {
        if (const uint32_t tg = sub_targets(sub[i])) {
            --k;
            for (int j = 0; j < RB; ++j)
                if (tg >> j & 1) next[j] = k;
        } else if (of_sub[i] >= 0) {
            Cond &c = conds[of_sub[i]];
            c.hi = m;
            for (int j = 0; j < RB; ++j)
                if (c.f.rd >> j & 1) c.hi = std::min(c.hi, next[j]);
        }
    }
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return conds[x].hi < conds[y].hi; });
    const int most = limited(plan, kSepBits);
    std::vector<std::vector<SepGroup>> at(m + 1);
    std::vector<uint32_t> at_rd(m + 1, 0);
    for (int i : order) {
        if (conds[i].point >= 0) continue;
        const int p = conds[i].hi;
        std::vector<int> in;
        for (int k : order)
            if (conds[k].point < 0 && conds[k].lo <= p && p <= conds[k].hi) {
                conds[k].point = p;
                in.push_back(k);
            }
        // groups of at most `most` conditions: the most widely used orders first, by condition code
        std::stable_sort(in.begin(), in.end(), [&](int x, int y) {
            const auto &a = conds[x].f.dl, &c = conds[y].f.dl;
            return std::lexicographical_compare(a.begin(), a.end(), c.begin(), c.end());
        });
        std::vector<SepGroup> &groups = at[p];
        std::vector<std::vector<int>> members;
        for (int k : in) {
            const std::vector<uint8_t> &dl = conds[k].f.dl;
            size_t best = groups.size();
            int fewest = most + 1;
            for (size_t g = 0; g < groups.size(); ++g) {
                int extra = 0;
                for (uint8_t c : dl) extra += std::find(groups[g].dl.begin(), groups[g].dl.end(), c) == groups[g].dl.end();
                if (extra < fewest && (int)groups[g].dl.size() + extra <= std::max<int>(most, (int)dl.size())) {
                    fewest = extra;
                    best = g;
                }
            }
            if (best == groups.size()) {
                groups.emplace_back();
                members.emplace_back();
            }
            for (uint8_t c : dl)
                if (std::find(groups[best].dl.begin(), groups[best].dl.end(), c) == groups[best].dl.end()) groups[best].dl.push_back(c);
            members[best].push_back(k);
            at_rd[p] |= conds[k].f.rd;
        }
        if (groups.size() > kSepGroups) return false;
        for (size_t g = 0; g < groups.size(); ++g) {
            SepGroup &G = groups[g];
            const size_t H = size_t(1) << G.dl.size();
            G.tab.assign(H * (RB + 1), cd(1.0));
            for (int k : members[g]) {
                const Separable &f = conds[k].f;
                std::vector<int> pos;
                for (uint8_t c : f.dl) pos.push_back(int(std::find(G.dl.begin(), G.dl.end(), c) - G.dl.begin()));
                size_t need = 0;
                for (size_t j = 0; j < pos.size(); ++j) need |= ((f.need >> j) & 1) << pos[j];
                for (size_t h = need; h < H; h = (h + 1) | need) {
                    size_t hk = 0;
                    for (size_t j = 0; j < pos.size(); ++j) hk |= ((h >> pos[j]) & 1) << j;
                    cd *to = G.tab.data() + h * (RB + 1);
                    const cd *from = f.tab.data() + hk * (RB + 1);
                    if (f.scalar) to[0] = mul(to[0], from[0]);
                    for (int j = 0; j < RB; ++j)
                        if (f.rd >> j & 1) to[1 + j] = mul(to[1 + j], from[1 + j]);
                }
            }
        }
    }
    int k = 0;
    auto emit = [&](int p) {
        if (!at[p].empty()) b.add_sep(std::move(at[p]), at_rd[p]);
    };
    for (int i = 0; i < ns && !b.bad; ++i) {
        if (of_sub[i] >= 0) {
            const Separable &f = conds[of_sub[i]].f;
            if (!f.q.empty()) b.add_factors(f.q);
            continue;
        }
        if (sub_targets(sub[i])) {
            emit(k);
            ++k;
        }
        b.add_sub(sub[i]);
    }
    if (!b.bad) emit(k);
    return true;
}

// Estimated time of a stage's diagonals: complex64 in ns per slab and SM, else in FP multiplies per amplitude.
double diagonal_cost(const Plan &plan, int RB, const std::vector<LeanItem> &items)
{
    const int E = 1 << RB;
    double c = 0.0;
    for (const LeanItem &it : items) {
        const double frac = __builtin_popcount(it.m32) / double(E);
        uint32_t active = 0;
        for (size_t i = 0; i < it.tab.size(); ++i)
            if (it.tab[i] != cd(1.0)) active |= 1u << (i & (E - 1));
        if (plan.dt == QS_C64) {
            if (it.op == L_TABLE) c += (it.dl.empty() ? 300.0 : 380.0) * (active_pattern(active, RB, 1) ? 0.6 : 1.0);
            else if (it.op == L_SEP) c += 450.0 + 60.0 * it.sep.size();
            else if (it.op == L_PHASE) c += 270.0;
            else if (it.op == L_SCALE) c += 100.0;
        } else {
            if (it.op == L_TABLE) c += active_pattern(active, RB) ? 2.0 : 4.0;
            else if (it.op == L_SEP) c += 4.0 * (2.0 * E - 6.0) / E + 4.0 * (RB + 0.5) / E * (it.sep.size() - 1.0);
            else if (it.op == L_PHASE && it.p != cd(-1.0)) c += 4.0 * std::max(0.5, frac);
            else if (it.op == L_SCALE) c += 2.0;
        }
    }
    return c;
}

}  // namespace

void lower_stage(const Plan &plan, const DevStage &st, int RB, LeanStage &out)
{
    auto finish = [](Builder &b) {
        b.flush_carry();
        b.gather_phases();
        b.group_shears();
        b.merge_tables();
    };
    // The same stage with its conditional diagonals in separable form, where that is clearly cheaper (in
    // complex64 and double-float it also takes the larger kernel).  If it is even against a low
    // estimate of the merged tables, those are not built.
    LeanStage alt;
    double alt_cost = 0.0;
    const size_t index = size_t(&st - plan.stages.data());
    double most = 0.0;  // what its merged conditional diagonals cost, against one separable table of one group
    for (int i = st.sub_begin; i < st.sub_end; ++i) {
        const DevSub &sb = plan.subs[i];
        if (sb.type == SB_DIAG && sb.ndl) most += plan.dt == QS_C64 ? 380.0 : 4.0;
        if (sb.type == SB_PHASE && (sb.lcm | sb.ocm))
            most += plan.dt == QS_C64 ? 270.0 : plan.coef[sb.mat] == cd(-1.0) ? 0.0 : 2.0;
    }
    if (index < plan.raw_range.size() && (plan.dt == QS_C64 ? 510.0 : 4.0 * (2.0 - 6.0 / (1 << RB))) < 0.8 * most) {
        const auto range = plan.raw_range[index];
        Builder r(plan, RB);
        if (lower_regrouped(plan, plan.raw_subs.data() + range.first, range.second - range.first, RB, r) && !r.bad) {
            finish(r);
            alt.ok = true;
            alt.flip = r.F;
            alt.items = std::move(r.items);
            alt_cost = diagonal_cost(plan, RB, alt.items);
            double low = 0.0;
            for (int i = st.sub_begin; i < st.sub_end; ++i)
                if (plan.subs[i].type == SB_DIAG) low += plan.dt == QS_C64 ? 300.0 : 2.0;
            if (alt_cost < 0.8 * low) {
                out = std::move(alt);
                return;
            }
        }
    }
    Builder b(plan, RB);
    for (int i = st.sub_begin; i < st.sub_end && !b.bad; ++i) b.add_sub(plan.subs[i]);
    out = LeanStage{};
    if (b.bad) return;
    finish(b);
    if (alt.ok && alt_cost < 0.8 * diagonal_cost(plan, RB, b.items)) {
        out = std::move(alt);
        return;
    }
    out.ok = true;
    out.flip = b.F;
    out.items = std::move(b.items);
}

void lower_stages(const Plan &plan, qs_dtype dt, bool df, std::vector<DevStage> &stages, LeanImage &img)
{
    const int RB = plan.stage_bits > 0 ? plan.stage_bits : (dt == QS_C64 ? kStageBitsC64 : kStageBitsC128);
    const int E = 1 << RB;
    const int pl = lean_pair_log(dt);
    const size_t real = dt == QS_C64 ? 4 : 8;
    std::vector<unsigned char> &W = img.words;
    auto word = [&]() {  // a new zero word; its byte offset
        W.resize(W.size() + 16, 0);
        return W.size() - 16;
    };
    auto conditions = [&](const LeanItem &it) {
        const size_t c = word();
        put(W.data(), c, it.lcm);
        put(W.data(), c + 8, it.ocm);
    };
    // factor of element e at word w + (e >> pl) of `buf`
    auto put_factor = [&](unsigned char *buf, size_t w, int e, const cd &v) {
        unsigned char *p = buf + 16 * (w + (size_t(e) >> pl));
        if (pl) {  // [re, re, im, im]
            put_real(p, 4 * (e & 1), v.real(), dt, df);
            put_real(p, 8 + 4 * (e & 1), v.imag(), dt, df);
        } else {
            put_real(p, 0, v.real(), dt, df);
            put_real(p, real, v.imag(), dt, df);
        }
    };
    auto pattern = [&](uint32_t elems) { return active_pattern(elems, RB, pl); };  // complex64: not of bit 0
    for (DevStage &st : stages) {
        LeanStage ls;
        lower_stage(plan, plan.stages[&st - stages.data()], RB, ls);
        st.lean_begin = -1;
        st.lean_words = st.lean_full = 0;
        if (!ls.ok) continue;
        const size_t head = word();
        st.lean_begin = int(head / 16);
        for (int j = 0; j < RB; ++j) W[head + j] = st.sbits[j];
        put(W.data(), head + 8, uint32_t(st.nrest) | ls.flip << 8);
        for (const LeanItem &it : ls.items) {
            if (it.op == L_ROTA) {
                // complex64: from 4 of 5 bits on, one record for all bits (missing ones are the
                // identity) is cheaper than a record per bit: 413 against 114 ns each per slab of
                // 2^13 and SM.  FP64 and double-float arithmetic costs too much to run for nothing.
                const bool all = dt == QS_C64 && __builtin_popcount(it.mask) >= RB - 1;
                size_t at = 0;
                if (all) {
                    at = word();
                    W[at] = (unsigned char)L_ROTA;
                }
                int k = 0;
                for (int j = 0; j < RB; ++j) {
                    if (!all && !(it.mask >> j & 1)) continue;
                    if (!all) {
                        at = word();
                        W[at] = (unsigned char)(((it.neg >> j & 1) ? L_ROTM0 : L_ROT0) + j);
                    }
                    size_t off;
                    if (dt != QS_C64) off = word();
                    else if (!all || k == 0) off = at + 8;
                    else off = (k & 1) ? word() : W.size() - 8;
                    put_real(W.data(), off, it.y[j], dt, df);
                    put_real(W.data(), off + real, it.x[j], dt, df);
                    ++k;
                }
                continue;
            }
            const size_t at = word();
            W[at] = (unsigned char)it.op;
            if (it.op == L_SEP || it.op == L_CX || (it.op == L_PHASE && it.p != cd(-1.0) && dt == QS_C64)) st.lean_full = 1;
            switch (it.op) {
            case L_CX:
                W[at + 1] = (unsigned char)it.j;
                W[at + 2] = (unsigned char)(it.ctrl < 0 ? 0xff : it.ctrl);
                conditions(it);
                break;
            case L_PHASE:
                put(W.data(), at + 4, it.m32);
                put(W.data(), at + 8, pattern(it.m32));
                conditions(it);
                if (it.p == cd(-1.0)) {
                    W[at] = (unsigned char)L_SIGN;
                } else {
                    const size_t f = word();
                    put_real(W.data(), f, it.p.real(), dt, df);
                    put_real(W.data(), f + real, it.p.imag(), dt, df);
                }
                break;
            case L_SEP: {
                bool scalar = false;
                for (const SepGroup &g : it.sep)
                    for (size_t i = 0; i < g.tab.size(); i += RB + 1) scalar = scalar || g.tab[i] != cd(1.0);
                W[at] = (unsigned char)(scalar ? L_SEP : L_SEP1);
                W[at + 1] = (unsigned char)it.sep.size();
                for (const SepGroup &g : it.sep) {
                    const int ndl = int(g.dl.size());
                    std::vector<int> order(ndl);
                    for (int j = 0; j < ndl; ++j) order[j] = j;
                    std::sort(order.begin(), order.end(), [&](int a, int b) { return g.dl[a] < g.dl[b]; });
                    int nl = 0;
                    while (nl < ndl && !(g.dl[order[nl]] & 0x80)) ++nl;
                    const size_t off = img.pool.size() / 16, per = size_t(RB + 1 + pl) >> pl;  // words per setting
                    const size_t gw = word(), codes = word();
                    put(W.data(), gw, uint32_t(off));
                    W[gw + 4] = (unsigned char)nl;
                    W[gw + 5] = (unsigned char)ndl;
                    for (int j = 0; j < ndl; ++j) W[codes + j] = g.dl[order[j]];
                    img.pool.resize(img.pool.size() + (per << ndl) * 16, 0);
                    for (size_t h = 0; h < (size_t(1) << ndl); ++h) {
                        size_t src = 0;
                        for (int j = 0; j < ndl; ++j) src |= ((h >> j) & 1) << order[j];
                        const size_t hl = h & ((size_t(1) << nl) - 1), ho = h >> nl;
                        for (int t = 0; t <= RB; ++t) {
                            const cd v = g.tab[src * (RB + 1) + t];
                            unsigned char *p = img.pool.data() + 16 * (off + (((ho * per + (t >> pl)) << nl) | hl)) + (pl ? 8 * (t & 1) : 0);
                            put_real(p, 0, v.real(), dt, df);
                            put_real(p, real, v.imag(), dt, df);
                        }
                    }
                }
                break;
            }
            case L_SCALE: {
                const size_t per = dt == QS_C64 ? 4 : 1;  // factors per word
                const size_t f = W.size();
                for (size_t w = 0; w < E / per; ++w) word();
                for (int e = 0; e < E; ++e) put_real(W.data(), f + e * (16 / per), it.scale[e], dt, df);
                break;
            }
            default: {  // L_TABLE
                const int ndl = int(it.dl.size());
                uint32_t active = 0;  // elements with a factor other than 1
                const uint32_t every = E == 32 ? ~0u : (1u << E) - 1u;
                for (size_t i = 0; i < it.tab.size() && active != every; ++i)
                    if (it.tab[i] != cd(1.0)) active |= 1u << (i & (E - 1));
                put(W.data(), at + 8, pattern(active));
                if (dt != QS_C64 && !df && pattern(active)) st.lean_full = 1;
                if (ndl == 0) {
                    W[at] = (unsigned char)L_CONST;
                    const size_t f = W.size() / 16;
                    for (int w = 0; w < E >> pl; ++w) word();
                    for (int e = 0; e < E; ++e) put_factor(W.data(), f, e, it.tab[e]);
                    break;
                }
                // conditions inside the slab first, ascending (they differ between a warp's lanes), then
                // those outside it, which are the same for a whole slab
                std::vector<int> order(ndl);
                for (int j = 0; j < ndl; ++j) order[j] = j;
                std::sort(order.begin(), order.end(), [&](int a, int b) { return it.dl[a] < it.dl[b]; });
                int nl = 0;
                while (nl < ndl && !(it.dl[order[nl]] & 0x80)) ++nl;
                W[at + 2] = (unsigned char)nl;
                W[at + 3] = (unsigned char)ndl;
                const size_t off = img.pool.size() / 16;
                put(W.data(), at + 4, uint32_t(off));
                const size_t codes = word();
                for (int j = 0; j < ndl; ++j) W[codes + j] = it.dl[order[j]];
                img.pool.resize(img.pool.size() + ((size_t(E) << ndl) >> pl) * 16, 0);
                for (size_t h = 0; h < (size_t(1) << ndl); ++h) {
                    size_t src = 0;
                    for (int j = 0; j < ndl; ++j) src |= ((h >> j) & 1) << order[j];
                    const size_t hl = h & ((size_t(1) << nl) - 1), ho = h >> nl;
                    for (int e = 0; e < E; ++e) {
                        const size_t row = (ho << (RB - pl)) | (size_t(e) >> pl);
                        const cd &v = it.tab[(src << RB) | e];
                        unsigned char *p = img.pool.data() + 16 * (off + ((row << nl) | hl));
                        if (dt != QS_C64 && !df) std::memcpy(p, &v, 16);
                        else put_factor(p, 0, e & ((1 << pl) - 1), v);
                    }
                }
                break;
            }
            }
        }
        st.lean_words = int(W.size() / 16) - st.lean_begin;
        put(W.data(), head + 12, uint32_t(st.lean_words - 1));
    }
}

}  // namespace qs

// lower.cpp -- register stages rewritten for the in-place stage engine (lean_stage.cuh).
//
// A plan describes a stage by its sub-ops (DevSub): real 2x2 matrices with two unit entries,
// diagonal tables, controlled phases, X.  The engine wants few kinds of records, each a straight
// run of in-place updates, so the stage is rewritten here, in FP64, without changing what it
// computes (Eq. 2-3 reassociated):
//
//  * FP32 and double-float: a real 2x2 matrix S with s11 != 0 is D L, L two shears and D a real diagonal:
//      v1 += y v0;  v0 += x v1;   y = s10 / s11,  x = s01 s11 / det,  D = diag(det / s11, s11),
//    two FMAs per pair that overwrite their inputs -- no copy through a temporary, which the
//    unit-entry forms need when both results use both old values.  |s11| >= |s10| is had by
//    exchanging the rows first where it does not hold, and the exchange (an X on that bit) is
//    not executed: from there on the bit is held "flipped" (slot s of the registers holds
//    logical index s ^ F), later sub-ops are written for slots, and the stage stores through
//    addresses XORed with F.  Uncontrolled X gates become such flips too.
//  * FP64: S = s00 [[1, x], [y, +-1]], with the same exchange of rows, two
//    FMAs per pair as well.  The copies through a temporary are free beside FP64 arithmetic, and the
//    factor is the same for both values of the bit, so it needs no multiply of its own.
//  * The factors D are carried along: past a shear pair on the same bit by D^-1 L D (real again,
//    and x y stays the same, so the relative rounding of each update does not change), past
//    everything else freely, until the next diagonal table takes them in.  A stage without a
//    table gets one real scaling at its end.
//  * Phases that can reach a table without crossing a record that does not commute with them
//    join it.
//  * Shear pairs on distinct register bits that can be brought together form one record.
#include "lower.h"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace qs {

namespace {

// Condition bits up to which a table grows to take in a conditional phase.  A sign costs three
// integer instructions per element as a record of its own; FP32 tables double in size per bit.
int table_bits(const Plan &plan) { return plan.dt == QS_C128 && plan.opt.arith == QS_ARITH_FP64 ? 10 : 5; }

struct Builder {
    const Plan &plan;
    const int RB, E;
    std::vector<LeanItem> items;
    std::vector<char> small;         // items[i] is a phase that may still join a table
    const bool unit;                 // FP64: unit-entry matrices instead of shears
    uint32_t F = 0;
    double d[6][2];
    bool bad = false;

    Builder(const Plan &p, int rb) : plan(p), RB(rb), E(1 << rb), unit(p.dt == QS_C128 && p.opt.arith == QS_ARITH_FP64)
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
    // a diagonal reading the bits `rd` commutes with item k
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
    // multiply the phase into the table if its conditions are, or can become, table conditions
    bool join(LeanItem &t, const LeanItem &ph) const
    {
        const std::vector<uint8_t> c = conditions(ph);
        std::vector<uint8_t> dl = t.dl;
        for (uint8_t b : c)
            if (std::find(dl.begin(), dl.end(), b) == dl.end()) dl.push_back(b);
        if (dl.size() > t.dl.size() && (int)dl.size() > table_bits(plan)) return false;
        std::vector<cd> tab(size_t(E) << dl.size());
        uint32_t need = 0;
        for (uint8_t b : c) need |= 1u << (std::find(dl.begin(), dl.end(), b) - dl.begin());
        const size_t old = (size_t(1) << t.dl.size()) - 1;
        for (size_t h = 0; h < (size_t(1) << dl.size()); ++h)
            for (int e = 0; e < E; ++e) {
                cd v = t.tab[((h & old) << RB) | e];
                if ((h & need) == need && (ph.m32 >> e & 1)) v *= ph.p;
                tab[(h << RB) | e] = v;
            }
        t.tab = std::move(tab);
        t.dl = std::move(dl);
        t.rd |= ph.rd;
        return true;
    }
    void add_table(LeanItem t)
    {
        // (a carry that is the same for all elements waits for the stage's end)
        if (carry_reads() || (!unit && carried())) {
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
        push(std::move(t));
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
            if (!(std::abs(d[j][0]) < 1e100 && std::abs(d[j][0]) > 1e-100)) flush_carry();
            return;
        }
        const double det = s00 * s11 - s01 * s10;
        if (!(std::abs(s11) > 0.0) || !(std::abs(det) > 1e-6 * s11 * s11)) {
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
    // The carried diagonal joins the last table it can be moved back to, or becomes a scaling.
    void flush_carry()
    {
        if (!carried()) return;
        size_t t = items.size();
        bool found = false;
        while (t-- > 0) {
            const LeanItem &it = items[t];
            if (it.op == L_TABLE) {
                found = true;
                break;
            }
            if (it.op == L_CX && d[it.j][0] != d[it.j][1]) break;
        }
        if (!found) {
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
        apply_carry(items[t]);
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
        case SB_G1R:
            if (ctl) bad = true;
            else add_real(sb.j0, M[0].real(), M[1].real(), M[2].real(), M[3].real());
            break;
        case SB_G1: {
            // complex 2x2: phase, real rotation, phase (the planner's Z-Y-Z form)
            const double c = std::abs(M[0]), s = std::abs(M[2]);
            if (ctl || c < 1e-6 || s < 1e-6) {
                bad = true;
                break;
            }
            const cd g = M[0] / c, eb = M[2] / (g * s), ed = -M[1] / (g * s);
            const bool unitary = std::abs(std::abs(eb) - 1.0) <= 1e-12 && std::abs(std::abs(ed) - 1.0) <= 1e-12;
            if (!unitary || std::abs(M[3] - g * eb * ed * c) > 1e-12 * c || std::abs(c * c + s * s - 1.0) > 1e-12) {
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
    // cheaper.  complex64 runs any complex phase as a table (it
    // takes about as long as one phase of 16 elements, 270 ns); otherwise the multiplies decide, E against the phases' elements.
    void gather_phases()
    {
        for (size_t k = 0; k < items.size(); ++k) {
            if (!small[k] || items[k].p == cd(-1.0)) continue;
            LeanItem t;
            t.op = L_TABLE;
            t.tab.assign(E, cd(1.0));
            if (!join(t, items[k])) continue;
            std::vector<size_t> in;
            int elems = __builtin_popcount(items[k].m32);
            for (size_t j = 0; j < items.size(); ++j) {
                if (j == k || !small[j]) continue;
                const uint32_t rd = items[j].rd;
                if (!(j > k ? commute_between(rd, k + 1, j) : commute_between(rd, j + 1, k))) continue;
                if (!join(t, items[j])) continue;
                in.push_back(j);
                if (items[j].p != cd(-1.0)) elems += __builtin_popcount(items[j].m32);
            }
            if (plan.dt != QS_C64 && elems <= E) continue;
            items[k] = std::move(t);
            small[k] = 0;
            for (size_t i = in.size(); i-- > 0;) {
                items.erase(items.begin() + in[i]);
                small.erase(small.begin() + in[i]);
                if (in[i] < k) --k;
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

void lower_stage(const Plan &plan, const DevStage &st, int RB, LeanStage &out)
{
    Builder b(plan, RB);
    for (int i = st.sub_begin; i < st.sub_end && !b.bad; ++i) b.add_sub(plan.subs[i]);
    out = LeanStage{};
    if (b.bad) return;
    b.flush_carry();
    b.gather_phases();
    b.group_shears();
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
    // the smallest pattern (lean_stage.cuh: all, or one value of one bit) that holds all `elems`
    auto pattern = [&](uint32_t elems) -> uint32_t {
        static const uint32_t ones[4] = {0xaaaaaaaau, 0xccccccccu, 0xf0f0f0f0u, 0xff00ff00u};
        for (int j = 0; j < RB && j < 4; ++j) {
            if (!(elems & ones[j])) return 1 + 2 * j;
            if (!(elems & ~ones[j])) return 2 + 2 * j;
        }
        return 0;
    };
    for (DevStage &st : stages) {
        LeanStage ls;
        lower_stage(plan, st, RB, ls);
        st.lean_begin = -1;
        st.lean_words = 0;
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
                for (size_t i = 0; i < it.tab.size(); ++i)
                    if (it.tab[i] != cd(1.0)) active |= 1u << (i & (E - 1));
                put(W.data(), at + 8, pattern(active));
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
                        put_factor(img.pool.data(), off + ((row << nl) | hl), e & ((1 << pl) - 1), it.tab[(src << RB) | e]);
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

// lowered_stages.cpp -- executes the register stages of a plan twice on the host, once by the sub-ops that
// the general engine runs and once by the records of the in-place engine (lower.h), and compares.
// Built by test_lowered_stages_cpu.py against the library's host code; no GPU.
#include <algorithm>
#include <cmath>
#include <complex>
#include <random>
#include <string>
#include <vector>

#include "lower.h"

using namespace qs;

namespace {

using Regs = std::vector<cd>;

// Value of condition bits (DevSub::dl codes) of a group at slab-local index `base` in slab `cta`.
size_t setting(const uint8_t *dl, size_t n, uint32_t base, uint64_t cta)
{
    size_t h = 0;
    for (size_t j = 0; j < n; ++j) {
        const uint32_t b = dl[j] & 0x7f;
        h |= size_t((dl[j] & 0x80) ? (cta >> b) & 1 : (base >> b) & 1) << j;
    }
    return h;
}

bool run_sub(const Plan &p, const DevSub &s, int RB, uint32_t base, uint64_t cta, Regs &v)
{
    if ((base & s.lcm) != s.lcm || (cta & s.ocm) != s.ocm) return true;
    const cd *M = p.coef.data() + s.mat;
    const uint32_t E = 1u << RB, t = 1u << s.j0;
    auto pair = [&](cd a, cd b, cd c, cd d) {
        for (uint32_t e = 0; e < E; ++e)
            if (!(e & t) && (e & s.scm) == s.scm) {
                const cd x = v[e], y = v[e | t];
                v[e] = a * x + b * y;
                v[e | t] = c * x + d * y;
            }
        return true;
    };
    switch (s.type) {
    case SB_G1: case SB_G1R: return pair(M[0], M[1], M[2], M[3]);
    case SB_G1N: return pair(1, M[0], M[1], 1);
    case SB_G1NM: return pair(1, M[0], M[1], -1);
    case SB_G1A: return pair(M[0], 1, 1, M[1]);
    case SB_G1AM: return pair(M[0], 1, -1, M[1]);
    case SB_X: return pair(0, 1, 1, 0);
    case SB_PHASE:
        for (uint32_t e = 0; e < E; ++e)
            if ((e & s.scm) == s.scm) v[e] *= M[0];
        return true;
    case SB_DIAG: {
        const size_t h = setting(s.dl, s.ndl, base, cta);
        for (uint32_t e = 0; e < E; ++e) v[e] *= M[(h << RB) | e];
        return true;
    }
    default: return false;
    }
}

// x as the device holds it: FP64, FP32, or the sum of two FP32 numbers.
double held(double x, qs_dtype dt, bool df)
{
    if (dt == QS_C64) return (float)x;
    if (!df) return x;
    const float h = (float)x;
    return (double)h + (double)(float)(x - (double)h);
}

// The plan of a circuit, or false.
bool plan_of(const qs_gate *g, size_t ng, int n, const qs_options *opt, Plan &p)
{
    std::vector<CGate> cg;
    std::string err;
    return !canonicalize(g, ng, n, cg, err) && !build_plan(cg, n, (qs_dtype)opt->dtype, *opt, p, err);
}

}  // namespace

// most: condition bits of a lowered table, of a separable group, of a sub-op of the plan (before and after the
// planner's merges); lowered stages with a 2x2 matrix; stages with one.
extern "C" int lowered_widths(const qs_gate *g, size_t ng, int n, const qs_options *opt, int64_t *most)
{
    Plan p;
    if (!plan_of(g, ng, n, opt, p)) return -1;
    auto conditions = [](const DevSub &s) -> int64_t {
        if (s.type == SB_DIAG) return s.ndl;
        return s.type == SB_PHASE ? __builtin_popcount(s.lcm) + __builtin_popcountll(s.ocm) : 0;
    };
    for (const DevSub &s : p.raw_subs) most[2] = std::max(most[2], conditions(s));
    for (const DevSub &s : p.subs) most[2] = std::max(most[2], conditions(s));
    for (const DevStage &st : p.stages) {
        LeanStage ls;
        lower_stage(p, st, p.stage_bits, ls);
        bool matrix = false;
        for (int i = st.sub_begin; i < st.sub_end; ++i) {
            const int t = p.subs[i].type;
            matrix |= t != SB_PHASE && t != SB_DIAG && t != SB_X && t != SB_SWAP;
        }
        most[4] += matrix;
        if (!ls.ok) continue;
        most[3] += matrix;
        for (const LeanItem &it : ls.items) {
            if (it.op == L_TABLE) most[0] = std::max<int64_t>(most[0], it.dl.size());
            for (const SepGroup &q : it.sep) most[1] = std::max<int64_t>(most[1], q.dl.size());
        }
    }
    return 0;
}

// count: stages, lowered stages, separable records, records in all.  Returns the largest difference of an
// amplitude relative to the largest amplitude of its group (inf for a NaN), or -1 on a bad circuit.
extern "C" double lowered_difference(const qs_gate *g, size_t ng, int n, const qs_options *opt, int64_t *count)
{
    const qs_dtype dt = (qs_dtype)opt->dtype;
    const bool df = dt == QS_C128 && opt->arith == QS_ARITH_DF;
    Plan p;
    if (!plan_of(g, ng, n, opt, p)) return -1.0;
    const int RB = p.stage_bits;
    const uint32_t E = 1u << RB;
    std::mt19937_64 rng(1);
    std::normal_distribution<double> normal;
    auto C = [&](const cd &x) { return cd(held(x.real(), dt, df), held(x.imag(), dt, df)); };
    auto D = [&](double x) { return held(x, dt, df); };
    double worst = 0.0;
    for (const DevStage &st : p.stages) {
        LeanStage ls;
        lower_stage(p, st, RB, ls);
        ++count[0];
        if (!ls.ok) continue;
        ++count[1];
        count[3] += (int64_t)ls.items.size();
        for (const LeanItem &it : ls.items) count[2] += it.op == L_SEP;
        for (int rep = 0; rep < 4; ++rep) {
            const uint64_t cta = rep ? rng() : ~0ull;
            uint32_t base = rep ? uint32_t(rng()) & 0xffffu : 0xffffu;
            for (int j = 0; j < RB; ++j) base &= ~(1u << st.sbits[j]);
            Regs w(E);
            for (cd &x : w) x = cd(normal(rng), normal(rng));
            Regs u = w;
            for (int i = st.sub_begin; i < st.sub_end; ++i)
                if (!run_sub(p, p.subs[i], RB, base, cta, w)) return -1.0;
            for (const LeanItem &it : ls.items) {
                const bool on = (base & it.lcm) == it.lcm && (cta & it.ocm) == it.ocm;
                switch (it.op) {
                case L_ROTA:
                    for (int j = 0; j < RB; ++j)
                        for (uint32_t e = 0; e < E; ++e) {
                            if (!(it.mask >> j & 1) || (e >> j & 1)) continue;
                            cd &a = u[e], &b = u[e | 1u << j];
                            if (dt == QS_C128) {
                                const cd a0 = a;
                                a = a0 + D(it.x[j]) * b;
                                b = D(it.y[j]) * a0 + ((it.neg >> j & 1) ? -b : b);
                            } else {
                                b += D(it.y[j]) * a;
                                a += D(it.x[j]) * b;
                            }
                        }
                    break;
                case L_TABLE: {
                    const size_t h = setting(it.dl.data(), it.dl.size(), base, cta);
                    for (uint32_t e = 0; e < E; ++e) u[e] *= C(it.tab[(h << RB) | e]);
                    break;
                }
                case L_SEP:
                    for (uint32_t e = 0; e < E; ++e) {
                        cd f = 1.0;
                        for (const SepGroup &q : it.sep) {
                            const cd *t = q.tab.data() + setting(q.dl.data(), q.dl.size(), base, cta) * (RB + 1);
                            f *= C(t[0]);
                            for (int j = 0; j < RB; ++j)
                                if (e >> j & 1) f *= C(t[1 + j]);
                        }
                        u[e] *= f;
                    }
                    break;
                case L_SCALE:
                    for (uint32_t e = 0; e < E; ++e) u[e] *= D(it.scale[e]);
                    break;
                case L_PHASE:
                    for (uint32_t e = 0; on && e < E; ++e)
                        if (it.m32 >> e & 1) u[e] *= C(it.p);
                    break;
                case L_CX:
                    for (uint32_t e = 0; on && e < E; ++e)
                        if (!(e >> it.j & 1) && (it.ctrl < 0 || (e >> it.ctrl & 1))) std::swap(u[e], u[e | 1u << it.j]);
                    break;
                default: return -1.0;
                }
            }
            double most = 0.0, diff = 0.0;
            for (uint32_t e = 0; e < E; ++e) {
                most = std::max(most, std::abs(w[e]));
                const double d = std::abs(u[e] - w[e ^ ls.flip]);
                if (!(d <= diff)) diff = std::isnan(d) ? INFINITY : d;
            }
            if (diff > 0.0) worst = std::max(worst, most > 0.0 ? diff / most : INFINITY);
        }
    }
    return worst;
}

// lower.h -- register stages of a plan rewritten for the in-place stage engine (lean_stage.cuh).
#pragma once

#include <cstdint>
#include <vector>

#include "planner.h"

namespace qs {

// One group of a separable table: factor(e) = s prod_j phi_j^(e_j), with s and phi looked up by the
// condition bits dl: entry h (RB + 1) + 0 is s, + 1 + j is phi_j.
struct SepGroup {
    std::vector<uint8_t> dl;
    std::vector<cd> tab;
};

// Exponents of carried factors: that of slot 0, then of each register bit's ratio.
struct Lift {
    int e[7] = {};
    Lift &operator+=(const Lift &o)
    {
        for (int j = 0; j < 7; ++j) e[j] += o.e[j];
        return *this;
    }
};

// One record of a lowered stage, in FP64; lower_stages() writes it in the state precision.
struct LeanItem {
    LeanOp op = L_ROTA;
    int j = 0, ctrl = -1;           // L_CX: target and control register bit (-1: none)
    uint32_t mask = 0;              // L_ROTA: register bits with a shear pair
    // L_ROTA, per register bit: v1 += y v0, then v0 += x v1; complex128 (from both old values): v0 + x v1,
    // y v0 +- v1 (minus where neg has the bit)
    double y[6] = {}, x[6] = {};
    uint32_t neg = 0;
    std::vector<cd> tab;            // L_TABLE: 2^(RB + ndl) factors, index (hi << RB) | e
    std::vector<uint8_t> dl;        // L_TABLE: condition bits (DevSub::dl codes)
    std::vector<SepGroup> sep;      // L_SEP
    std::vector<double> scale;      // L_SCALE: 2^RB real factors
    Lift lift;                      // L_TABLE, L_SEP: the carried factors that they took in
    uint32_t rd = 0;                // diagonals: register bits the factors may depend on
    uint32_t m32 = 0;               // L_PHASE: register elements the phase p acts on
    cd p = 1.0;
    uint32_t lcm = 0;               // L_PHASE, L_CX: bits that must all be 1
    uint64_t ocm = 0;
};

struct LeanStage {
    bool ok = false;      // the stage runs on the in-place engine
    uint32_t flip = 0;    // register bits whose two values are exchanged when the stage stores
    std::vector<LeanItem> items;
};

// Rewrite one register stage; out.ok is false if it holds a sub-op the engine does not run
// (4x4 matrices, controlled matrices, controlled swaps, X with two or more register controls).
void lower_stage(const Plan &plan, const DevStage &st, int RB, LeanStage &out);

// Lowered stages of one or more plans as device bytes: 16-byte words (qs_internal.h) and the pool of
// conditional tables, in the state precision (df: double-float quadruples).
struct LeanImage {
    std::vector<unsigned char> words, pool;
};

// Lower every stage of a plan, appending to img; stages (a copy of plan.stages) gets lean_begin and
// lean_words, or lean_begin = -1 where the general engine has to run the stage.
void lower_stages(const Plan &plan, qs_dtype dt, bool df, std::vector<DevStage> &stages, LeanImage &img);

}  // namespace qs

// Tile and K split of the FP64 GEMM in kernels.cu: plain host arithmetic.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstddef>

namespace ctm {

constexpr int GK = 16;                  // K step of the kernel
constexpr int GMAX_TM = 4, GMAX_TN = 9;  // largest tile: (32 TM) x (8 TN)
// Most columns of a product (64 times the grid's limit in y).
constexpr long long DGEMM_MAX_N = 64ll * 65535;

struct GemmPlan {
    int tm = 1, tn = 1, splits = 1;
    int kchunk = GK;  // K range of a split, whole steps; meaningless for one split
};
// The tile and K split with the least work on the fullest SM: TM TN multiply-
// adds per thread and k, at ~150 cycles each (8 warps on 4 quarters, measured
// 153), an estimated 3000 cycles of launch, fill and drain per CTA, 600 per 16
// of K for loads that a small tile does not cover, and for a split its
// partials' pass.  K = 0 (C = beta C) is planned as K = 1.
inline GemmPlan dgemm_plan(int M, int N, int K, size_t ws_doubles) {
    GemmPlan best;
    double best_cost = -1.0;
    const long long k = std::max(K, 1);
    for (int tm = 1; tm <= GMAX_TM; tm *= 2)
        for (int tn = 1; tn <= GMAX_TN; ++tn) {
            const double tiles = std::ceil(M / (32.0 * tm)) * std::ceil(N / (8.0 * tn));
            if (tn < GMAX_TN && N > 8 * tn * 65535) continue;  // grid.y
            for (int sp = 1; sp <= 256; sp *= 2) {
                const long long kc = ((k + sp - 1) / sp + GK - 1) / GK * GK, s = (k + kc - 1) / kc;
                if (sp > 1 && (s != sp || (size_t)s * M * N > ws_doubles)) break;
                const double steps = std::ceil(kc / (double)GK), per = (double)tm * tn * std::min(kc, k) * 150.0;
                const double cta = std::max(per, 600.0 * steps) + 300.0 * steps + 3000.0;
                const double cost = std::ceil(tiles * s / 152.0) * cta + (s > 1 ? 6000.0 + 40.0 * s * M * N / 152.0 / 32.0 : 0.0);
                if (best_cost < 0.0 || cost < best_cost) {
                    best_cost = cost;
                    best.tm = tm;
                    best.tn = tn;
                    best.splits = (int)s;
                    best.kchunk = s > 1 ? (int)kc : GK;
                }
            }
        }
    return best;
}

}  // namespace ctm

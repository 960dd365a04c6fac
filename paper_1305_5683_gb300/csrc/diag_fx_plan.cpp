// diag_fx_plan.cpp -- see diag_fx_plan.h
#include "diag_fx_plan.h"

#include <algorithm>

namespace spi {

void build_diag_fx(const Symbolic& S, DiagFxHost& h) {
    h = DiagFxHost();
    h.pptr.assign(S.ns, -1);
    h.tptr.assign(S.ns, -1);
    for (int32_t s = 0; s < S.ns; ++s) {
        const int32_t k = S.k_of(s), m = S.m_of(s);
        h.pptr[s] = h.npieces;
        h.tptr[s] = h.ntiles;
        h.xptr.push_back(h.ndt);
        for (int32_t g = 0; g * kFxRows < k; ++g) {
            const int32_t w = std::min(kFxRows, k - g * kFxRows), base = std::min(kFxRows * (g + 1), k);
            const int32_t np = (w + kFxSub - 1) / kFxSub, nt = 1 + (m - base + kFxRows - 1) / kFxRows;
            h.xoff.push_back(h.nx);
            h.nx += (int64_t)w * w;
            for (int32_t c = 0; c < w; c += kFxInvCols) h.dtiles.insert(h.dtiles.end(), {s, g, h.ndt, c});
            for (int32_t i = 0; i < nt; ++i) {
                h.tiles.insert(h.tiles.end(), {s, g, i, (int32_t)h.npieces});
                h.tdiag.push_back(i == 0 ? h.ndt : -1);
                h.npieces += np;
                ++h.ntiles;
            }
            ++h.ndt;
        }
    }
}

void diag_fx_used(const Symbolic& S, const DiagFxHost& h, const DiagPlan& dp, std::vector<int32_t>& tiles) {
    std::vector<uint8_t> used(S.ns, 0);
    for (int32_t s : dp.us) used[s] = 1;
    tiles.clear();
    for (size_t t = 0; 4 * t < h.tiles.size(); ++t)
        if (used[h.tiles[4 * t]]) tiles.push_back((int32_t)t);
}

void diag_fx_used_inverses(const Symbolic& S, const DiagFxHost& h, const DiagPlan& dp, std::vector<int32_t>& dtiles) {
    std::vector<uint8_t> used(S.ns, 0);
    for (int32_t s : dp.us) used[s] = 1;
    dtiles.clear();
    for (size_t t = 0; t < h.dtiles.size(); t += 4)
        if (used[h.dtiles[t]]) dtiles.insert(dtiles.end(), h.dtiles.begin() + t, h.dtiles.begin() + t + 4);
}

namespace {
constexpr double kMhz = 2070.0, kSms = 152.0;
// Cycles of a CTA for block b.
double block_cycles(const Symbolic& S, const DiagPlan& dp, int32_t b) {
    double w = 0.0;
    for (int32_t u = dp.uptr[b]; u < dp.uptr[b + 1]; ++u) {
        const int32_t s = dp.us[u], k = S.k_of(s), m = S.m_of(s);
        const double N = (double)((dp.uhi[u] - (dp.ulo[u] & ~7) + 15) & ~15) / 64.0;
        for (int32_t c = 0; c < k; c += kFxRows) {
            const int32_t cw = std::min(kFxRows, k - c), below = m - c - cw;
            const double tiles = 1.0 + (below + kFxRows - 1) / kFxRows;
            w += tiles * (3000.0 + N * (2200.0 + 900.0 * ((cw + kFxSub - 1) / kFxSub))) + 3000.0;
        }
    }
    return w;
}
}  // namespace

void diag_fx_order(const Symbolic& S, const DiagPlan& dp, std::vector<int32_t>& order) {
    std::vector<double> w((size_t)dp.nblocks, 0.0);
    order.resize((size_t)dp.nblocks);
    for (int32_t b = 0; b < dp.nblocks; ++b) {
        order[(size_t)b] = b;
        w[(size_t)b] = block_cycles(S, dp, b);
    }
    std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return w[x] > w[y]; });
}

bool diag_fx_pays(const Symbolic& S, const DiagPlan& dp, int bands, double extra) {
    double sum = 0.0, most = 0.0, nodes = 0.0, most_nodes = 0.0, cols = 0.0, active = 0.0, rows = 0.0;
    for (int32_t b = 0; b < dp.nblocks; ++b) {
        const double w = block_cycles(S, dp, b), nd = dp.uptr[b + 1] - dp.uptr[b];
        double cl = 0.0, ac = 0.0, rw = 0.0;
        for (int32_t u = dp.uptr[b]; u < dp.uptr[b + 1]; ++u) {
            const int32_t k = S.k_of(dp.us[u]), below = S.m_of(dp.us[u]) - k;
            cl += k;
            ac += (double)k * (dp.uhi[u] - dp.ulo[u]);
            rw += (double)k * ((below + 63) / 64);
        }
        sum += w, most = std::max(most, w), nodes += nd, most_nodes = std::max(most_nodes, nd);
        cols = std::max(cols, cl), active = std::max(active, ac), rows = std::max(rows, rw);
    }
    constexpr double kFp64 = 1.13e6;  // flops per us of the FP64 pipe
    const double fx = extra + 58.0 + 1.1 * most_nodes + 2.4 * most / kMhz +
                      bands / kSms * (0.75 * sum / kMhz + 7.4 * nodes);
    const double simt = 42.0 + 0.58 * cols + 0.48 * active / dp.B + 0.23 * rows + 0.69 * bands * dp.work_flops / kFp64;
    return fx <= simt;
}

double tile_inverse_us(const Symbolic& S, const std::vector<int32_t>& dtiles, int bands) {
    double instr = 0.0, chain = 0.0;  // FP64 warp instructions; us of the widest tile
    for (size_t t = 0; t < dtiles.size(); t += 4) {
        const int32_t k = S.k_of(dtiles[t]), w = std::min(kFxRows, k - dtiles[t + 1] * kFxRows), q0 = dtiles[t + 3];
        const int32_t warps = std::min(4, (w - q0 + 1) / 2);
        for (int32_t i = q0 / 32; 32 * i < w; ++i)
            instr += warps * 2.0 * (32 * (i - q0 / 32) + std::min(32, w - 32 * i));
        chain = std::max(chain, 6.0 + 46.0 * (w / 128.0) * (w / 128.0));
    }
    return std::max(chain, 1.45 * bands * instr * 16.0 / (kSms * kMhz));
}

bool wide_solve_pays(const Symbolic& S, const DiagFxHost& h, int bands) {
    int32_t saved = 0;
    for (int32_t l = 0; l < S.nlevels; ++l) {
        int32_t kmax = 0;
        for (int32_t p = S.level_ptr[l]; p < S.level_ptr[l + 1]; ++p) kmax = std::max(kmax, S.k_of(S.level_list[p]));
        saved += (kmax + 31) / 32 - (kmax + 63) / 64;
    }
    return tile_inverse_us(S, h.dtiles, bands) <= 12.0 * saved + 9.0;
}

}  // namespace spi

// diag_fx_plan.h -- host plan of the FP64 variance kernel on the tensor cores
// (diag_fx.cu): the packed left-operand tiles of every supernode.
#pragma once
#include <cstdint>
#include <vector>

#include "analysis.h"

namespace spi {

constexpr int kFxRows = 128;    // rows of a tile (the MMA's M) and columns of a K chunk
constexpr int kFxSub = 16;      // columns of one packed piece of a tile (the MMA's K)
constexpr int kFxInvCols = 8;   // columns of a diagonal tile's inverse per CTA
constexpr int kFxMaxBlock = 64; // right-hand sides of a block the kernel takes

struct DiagFxHost {
    int64_t npieces = 0;          // packed 128 x 16 pieces (per band)
    int32_t ntiles = 0, ndt = 0;  // 128 x 128 tiles, inverted diagonal tiles (per band)
    std::vector<int64_t> pptr;    // [ns] first packed piece of the supernode
    std::vector<int32_t> tptr;    // [ns] first tile of the supernode
    std::vector<int32_t> tiles;   // [ntiles][4]: supernode, chunk g, tile i of the chunk (0: its
                                  //   diagonal tile's inverse, i > 0: rows base + 128 (i - 1) ..), first piece
    std::vector<int32_t> dtiles;  // [][4]: supernode, chunk, number of the diagonal tile, first of 8 columns
    std::vector<int32_t> tdiag;   // [ntiles]: the diagonal tile's number (i = 0), else -1
    std::vector<int64_t> xoff;    // [ndt] offset of the diagonal tile's inverse (w x w, column-major)
    std::vector<int32_t> xptr;    // [ns] first diagonal tile of the supernode
    int64_t nx = 0;               // doubles of all inverses (per band)
};

// Every supernode; per 128-column chunk g of a supernode (k pivots, m rows): the inverse of its
// unit-lower diagonal tile, then the rows from min(128 (g + 1), k) to m in
// tiles of 128, each tile in ceil(w / 16) pieces (w the chunk's columns).
void build_diag_fx(const Symbolic& S, DiagFxHost& h);
// the tiles (positions in h.tiles / 4) of the supernodes that plan dp walks
void diag_fx_used(const Symbolic& S, const DiagFxHost& h, const DiagPlan& dp, std::vector<int32_t>& tiles);
// The diagonal tiles' columns (positions in h.dtiles / 4) of the supernodes that plan dp walks
void diag_fx_used_inverses(const Symbolic& S, const DiagFxHost& h, const DiagPlan& dp, std::vector<int32_t>& dtiles);
// Whether the inverses of all diagonal tiles are made by every factorization, for the solve's wide
// steps: where they shorten the solve by at least what they take.  us of each: a solve gains 6 per
// step saved in each sweep (and about 9 at any size), measured over the problems of diag_fx_pays; the
// inverses take tile_inverse_us.  P = 20,000: 175 us against 863 a solve; 48 trees of 50-2,000
// pointings 147 against 85; 400 problems of order 60 98 against 16 (factorization 127 us with
// the inverses left out, 213 with them), 32 bands of P = 800 107 against 24.  Where they are not
// made, the solve takes 32-column steps and the tensor-core variances make those they need.
bool wide_solve_pays(const Symbolic& S, const DiagFxHost& h, int bands);
// us of k_fx_tinv for `bands` bands of the listed column groups ([][4] as DiagFxHost::dtiles): its
// FP64 instructions at 1.45 times their share of the pipe, and at least the chain of the widest tile
// (measured: 104 us for 400 tiles of order 60, 194 for 60 fronts of order 300, 52 for one tile of 128)
double tile_inverse_us(const Symbolic& S, const std::vector<int32_t>& dtiles, int bands);
// The blocks of plan dp in the order in which they start: the costliest first, in cycles of a
// CTA: per tile 900 a piece and 2,200 for the read-out of 64 right-hand sides and 3,000
// whatever their number, 3,000 a chunk.  With about four CTAs per SM the last ones to start set
// the launch's end: by flops, which the many small supernodes of a long path hardly
// show in, 6.45 ms, so 5.67 (variances of P = 20,000).
void diag_fx_order(const Symbolic& S, const DiagPlan& dp, std::vector<int32_t>& order);

// Whether k_diag_fx serves plan dp of `bands` bands faster than the SIMT kernel in blocks of 16.  It
// costs about 7 us of an SM per supernode of a block whatever its width, and so loses where the
// supernodes are narrow and the blocks many: 8 bands of P = 800 0.70 against 0.41 ms, 3,000
// problems of order 8 0.35 against 0.10 ms, one unknown of P = 300 137 against 109 us; it wins from a
// few thousand pointings, a few dozen columns per supernode or one band on (P = 1,500 215 us against
// 350, 400 problems of order 60 182 against 258 us, P = 20,000 5.7 ms against 70).  Both times in us
// are fits (relative least squares, coefficients >= 0) to 120 calls measured with either kernel: 26
// problems of order 8 to 41,000, 1 to 32 bands, 1 to all unknowns.  They are right within 30 % (fx)
// and a factor 2 (SIMT), and the sides differ by more nearly everywhere: the choice was the slower one
// in three calls, by 5 to 25 %.
// extra: us of further work that only k_diag_fx needs.
bool diag_fx_pays(const Symbolic& S, const DiagPlan& dp, int bands, double extra);

}  // namespace spi

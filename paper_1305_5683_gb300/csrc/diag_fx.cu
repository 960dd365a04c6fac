// diag_fx.cu -- the FP64 form's variances on the 5th-generation tensor cores
// (paper Sec. 3.3.1 and Sec. 4.3: the pruned forward solves z = L^-1 e_i,
// right-hand sides in blocks, (N^-1)_ii = sum_k z_k^2 / d_k).
//
// An SM issues 1.7 FP64 multiply-adds per cycle but thousands of FP16 ones
// through tcgen05.mma, so the products of the forward solves are formed from
// exact integer pieces (the error-free splitting of Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59, 2012).  Every operand row (of L) or column (of z)
// is put on a fixed-point grid of 56 bits below its largest entry over 128 K
// columns, and cut into seven signed digits of 8 bits; digits are integers in
// [-128, 128], exact in FP16.  A product of digit i of one operand and digit
// j of the other is an integer of at most 2^14; for each level l = i + j <= 6
// the products of a 128-column chunk are accumulated in one FP32 accumulator:
// at most 7 x 128 x 2^14 < 2^24, so every sum is exact, whatever its order.
// The seven level sums are put together in 64-bit integers and rounded once to
// FP64.  What is dropped is bounded by the product of the row's and the column's largest
// entries, not by the product itself: at most 24 x 2^-56 of it for the levels > 6 and 4 x
// 2^-56 for the operands' rounding to their grids, about 2^-56 to 2^-54 rms.  The sums of
// squares taken here are served by that (an entry far below its column's largest adds as
// little to the variance); entries of N^-1 off the diagonal, which can be far smaller than
// the products they are summed from, are not, so covariances take the SIMT kernel's FP64
// solves (diag.cu).  To keep "largest entry" meaningful the kernel works with S^-1 L S and y = S^-1 z, S the
// powers of two next to D^1/2 (no rounding), so that the scale of an unknown cancels:
// the rows have the scale of N's entries over the square roots of their diagonal ones, y
// that of the variances' square roots, and (N^-1)_ii = sum_k y_k^2 f_k with f = S^2 / D
// between 1/2 and 2.
//
// Per block of B <= 64 right-hand sides one CTA walks the supernodes of the
// block's paths.  Per supernode and 128-column chunk g: the incoming values of the chunk's rows are cut into digits in
// shared memory and multiplied by the inverse of the chunk's 128 x 128
// diagonal tile (k_fx_tinv, FP64, at the end of the factorization), which gives the chunk's y; y is cut into
// digits, its squares are added to the variances in FP64, and the front's
// remaining rows are updated 128 at a time, Z_rows -= S^-1 L S y
// (Z, the block's workspace, holds S^-1 times the solves' vectors throughout).  The
// left operands arrive already cut, packed by k_fx_pack in the layout the MMA
// reads, by asynchronous bulk copies.
//
// Measured (one GB300, all variances, against the SIMT kernel on the FP64 pipe): P =
// 20,000 (n = 39,465) 70.4 -> 5.7 ms, of which the packing 0.14 and the walk 5.5 (the
// inverses, 0.18, come with the factorization); 48 problems as a forest (n = 51,264) 3.27 ->
// 1.25 ms; P = 300 (n = 467) 260 -> 118 us.  Largest error against 64-bit dense algebra the same for both (5e-14, rms
// 2.7e-15 at P = 20,000: the factorization's own).  The walk's 73,840 tiles of 128 x 64
// take 22,000 cycles of an SM each where the products need 7,900: what bounds it is
// the workers' chain of latencies -- tensor-memory reads, conversions, the read-modify-
// write of Z, one FP64 addition per element at 64 cycles a warp.
#include <cuda_runtime.h>

#include <algorithm>

#include "fx.cuh"
#include "spi_internal.cuh"

namespace spi {
namespace {

constexpr int kSlice = kFxRows * kFxSub * 2;       // bytes of one digit plane of a piece (4 KB)
constexpr int kPiece = kDig * kSlice;              // bytes of a packed piece

// Columns q0 .. q0 + 7 of the inverse X of the unit-lower diagonal tile of chunk g of
// supernode s (w <= 128 columns), one CTA per (tile, q0): forward substitution of unit
// vectors down the 32-row blocks, lane = row, two columns per warp.  Bound by the FP64
// pipe (64 cycles per warp instruction) and the chain of columns, so a tile is spread
// over w / 8 CTAs, every step is two independent multiply-adds per warp, and the values
// passed between steps are shuffled or read from shared memory.  X's transpose is stored too (xinvt
// not null).  (One column per warp
// was quicker for one small front, 21 against 27 us, but 354 against 193 us for all of
// P = 20,000.)
__global__ void __launch_bounds__(128) k_fx_tinv(DevSym d, const int32_t* __restrict__ dtiles,
                                                 const int64_t* __restrict__ xoff, int64_t nx,
                                                 const double* __restrict__ L, double* __restrict__ xinv,
                                                 double* __restrict__ xinvt, int64_t bsL) {
    static_assert(kFxInvCols == 8, "two columns for each of the four warps");
    L += blockIdx.y * bsL;
    const int32_t* dt = dtiles + 4 * (int64_t)blockIdx.x;
    const int s = dt[0], g = dt[1], q0 = dt[3];
    const int64_t t = dt[2];
    const int k = d.sfirst[s + 1] - d.sfirst[s];
    const int64_t m = d.srowptr[s + 1] - d.srowptr[s];
    const int c0 = g * kFxRows, w = min(kFxRows, k - c0);
    const double* P = L + d.lptr[s] + c0 + (int64_t)c0 * m;  // the tile, leading dimension m
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int col = q0 + 2 * warp;
    double* X = xinv + (int64_t)blockIdx.y * nx + xoff[t];  // column-major, leading dimension w
    double* Xt = xinvt ? xinvt + (int64_t)blockIdx.y * nx + xoff[t] : nullptr;  // its transpose, for the solve
    auto put = [&](int i, int j, double v) {
        X[i + j * w] = v;
        if (Xt) Xt[j + i * w] = v;
    };
    __shared__ double xs[4][kFxRows][2];
    double (*x)[2] = xs[warp];
    if (col >= w) return;
    const bool two = col + 1 < w;
    const int jb = col / 32;
    for (int r = lane; r < 32 * jb; r += 32) {  // above the columns' own block
        put(r, col, 0.0);
        if (two) put(r, col + 1, 0.0);
    }
    for (int i = jb; 32 * i < w; ++i) {
        const int r = 32 * i + lane;
        const bool on = r < w;
        double a0 = r == col ? 1.0 : 0.0, a1 = r == col + 1 ? 1.0 : 0.0;
        for (int kb = jb; kb < i; ++kb) {
            const double* Lk = P + r + (int64_t)(32 * kb) * m;
#pragma unroll 16
            for (int c = 0; c < 32; ++c) {
                const double l = on ? Lk[(int64_t)c * m] : 0.0;
                a0 = fma(-l, x[32 * kb + c][0], a0);
                a1 = fma(-l, x[32 * kb + c][1], a1);
            }
        }
        const double* Ld = P + r + (int64_t)(32 * i) * m;
        const int nc = min(32, w - 32 * i);
        for (int c8 = 0; c8 < nc; c8 += 8) {
            double l[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) l[q] = (on && c8 + q < lane) ? Ld[(int64_t)(c8 + q) * m] : 0.0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const double y0 = __shfl_sync(0xffffffffu, a0, c8 + q), y1 = __shfl_sync(0xffffffffu, a1, c8 + q);
                a0 = fma(-l[q], y0, a0);
                a1 = fma(-l[q], y1, a1);
            }
        }
        x[r][0] = a0;
        x[r][1] = a1;
        __syncwarp();
        if (on) put(r, col, a0);
        if (on && two) put(r, col + 1, a1);
    }
}

// One 128 x 128 tile of a left operand (of S^-1 X S, X the inverse of a diagonal tile,
// or of S^-1 L S), cut into digits: per row the exponent of its largest entry,
// then the seven digit planes of each 16-column piece in the K-major core-matrix layout
// (8 rows x 16 bytes; 128 bytes between K neighbours, 256 between row groups).
// One thread per row, 32 columns in flight (read again for the digits when there are
// more); the scales are added to the exponents, no FP64 arithmetic.  The tile of a chunk's inverse also writes
// f = s^2 / d of its pivots.
__global__ void __launch_bounds__(kFxRows) k_fx_pack(DevSym d, const int32_t* __restrict__ tiles,
                                                     const int32_t* __restrict__ tdiag,
                                                     const int32_t* __restrict__ list, int64_t ntiles, int64_t npieces,
                                                     const int64_t* __restrict__ xoff, int64_t nx,
                                                     const double* __restrict__ L,
                                                     const double* __restrict__ D, const double* __restrict__ xinv,
                                                     unsigned char* __restrict__ pack, int32_t* __restrict__ rexp,
                                                     double* __restrict__ fr, int64_t bsL, int64_t bsn) {
    const int64_t t = list[blockIdx.x];
    const int band = blockIdx.y, tid = threadIdx.x;
    L += band * bsL;
    D += band * bsn;
    const int s = tiles[4 * t], g = tiles[4 * t + 1], i = tiles[4 * t + 2], piece = tiles[4 * t + 3];
    const int f = d.sfirst[s], k = d.sfirst[s + 1] - f;
    const int64_t m = d.srowptr[s + 1] - d.srowptr[s];
    const int c0 = g * kFxRows, w = min(kFxRows, k - c0);
    const double* src;
    int64_t ld;
    bool on;
    int pivot;  // of this row
    if (i == 0) {
        on = tid < w;
        src = xinv + (int64_t)band * nx + xoff[tdiag[t]] + (on ? tid : 0);
        ld = w;
        pivot = f + c0 + tid;
    } else {
        const int64_t row = min(c0 + kFxRows, k) + (int64_t)(i - 1) * kFxRows + tid;
        on = row < m;
        src = L + d.lptr[s] + (on ? row : 0) + (int64_t)c0 * m;
        ld = m;
        pivot = on ? d.srows[d.srowptr[s] + row] : 0;
    }
    __shared__ int cs[kFxRows];
    double v[32];
    auto load = [&](int c0v) {
#pragma unroll
        for (int c = 0; c < 32; ++c) v[c] = (on && c0v + c < w) ? src[(c0v + c) * ld] : 0.0;
    };
    load(0);
    const double dv = on ? D[pivot] : 1.0;
    const int rs = -fx_scale_exp(dv);
    cs[tid] = tid < w ? fx_scale_exp(D[f + c0 + tid]) : 0;
    __syncthreads();
    int E = -16384;
    for (int cb = 0; cb < w; cb += 32) {
        if (cb > 0) load(cb);
#pragma unroll
        for (int c = 0; c < 32; ++c) E = max(E, fx_scaled_exp(v[c]) + cs[cb + c] + rs);
    }
    rexp[((int64_t)band * ntiles + t) * kFxRows + tid] = E - 1022;
    unsigned char* dst = pack + ((int64_t)band * npieces + piece) * kPiece + (tid >> 3) * kFxSub * 16 + (tid & 7) * 16;
    const int wp = (w + kFxSub - 1) / kFxSub * kFxSub;
    for (int cb = 0; cb < w; cb += 32) {
        if (w > 32) load(cb);
#pragma unroll
        for (int c8 = 0; c8 < 32; c8 += 8) {
            const int c = cb + c8;
            if (c < wp) {
                unsigned long long x[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) x[q] = fx_fix(v[c8 + q], fx_scaled_exp(v[c8 + q]) + cs[c + q] + rs, E);
                fx_store_planes<0>(dst + (size_t)(c / kFxSub) * kPiece + (c % kFxSub) / 8 * 128, kSlice, x);
            }
        }
    }
    if (i == 0 && on) fr[band * bsn + pivot] = fx_pow2(-2 * rs) / dv;
}

struct FxArgs {
    int32_t B;
    const int32_t *order, *blk_ptr, *uptr, *us, *ulo, *uhi, *uzoff, *rel, *rhs_out, *rhs_zrow, *rhs_col;
    const int64_t *urel, *zbase;
    double* Z;
    const int64_t* pptr;          // [ns] first packed piece
    const int32_t* tptr;          // [ns] first tile
    int64_t npieces, ntiles;      // per band
    const unsigned char* pack;
    const int32_t* rexp;
    const double *D, *fr;
    uint32_t wait_limit;          // polls of each wait, then the kernel gives up
};

// Roles: warps 0-15 cut z into digits, read the products out of tensor memory and
// update Z; lane 0 of warp 16 copies the packed pieces of L, lane 0 of warp 17
// issues the MMAs.  For digit plane i of L one MMA takes the planes 0 .. 6 - i of z
// side by side (N up to 256 columns per instruction): plane pair (i, j) lands in the
// accumulator columns of level i + j, and a plane of L is read from shared memory once
// or twice for all its partners.  The B = 64 right operand and the ring of left operands
// fill the SM's shared memory and the levels 448 columns of tensor memory, so a CTA
// has an SM to itself.  The workers first bring a tile's level sums into registers as
// 64-bit integers, free tensor memory for the next tile's products, and convert, subtract
// and store while those run (one FP64 addition per element: its pipe needs 4,100 cycles
// for a 128 x 64 tile, the products 7,200).
constexpr int kFxWork = 512;
constexpr int kFxThreads = kFxWork + 64;
enum : int { kFAF = 0, kFAE = 6, kFBF = 12, kFCF = 13, kFCE = 14, kFxBars = 15 };  // A full/empty, B full, acc full/empty
__host__ __device__ constexpr int fx_stages(int B) { return B > 32 ? 4 : 6; }
constexpr size_t fx_smem(int B) {
    return (size_t)fx_stages(B) * kPiece + (size_t)kDig * B * kFxRows * 2 + 128 * sizeof(int) +
           kFxBars * sizeof(uint64_t) + 16 + 2 * kFxRows * (sizeof(int) + sizeof(short));
}

__device__ __forceinline__ void fx_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(tc_smem_u32(bar)) : "memory");
}
// Bounded wait that also gives up when another role has.
__device__ __forceinline__ bool fx_wait(uint64_t* bar, uint32_t parity, volatile int* abort, uint32_t limit) {
    uint32_t done = 0;
    for (uint32_t it = 0; it < limit && !done; ++it) {
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done) : "r"(tc_smem_u32(bar)), "r"(parity) : "memory");
        if (!done && *abort) return false;
    }
    return done != 0;
}
// Barrier among the worker warps (every one of them meets every barrier, also after a wait ran out).
__device__ __forceinline__ void fx_bar() { asm volatile("barrier.cta.sync 1, %0;" :: "n"(kFxWork) : "memory"); }

// The block's supernodes in walk order and the shape of each; the right-hand sides
// from the multiple of 8 at or below the first active one (the extra columns of Z are
// zero on these rows), N of them rounded up to the MMA's 16.
struct FxNode {
    int s, lo, N, zo, f, k, m, G;
    int64_t urel;
};
__device__ __forceinline__ bool fx_next(const DevSym& d, const FxArgs& p, int& u, int u1, FxNode& x) {
    if (++u < u1) {
        const int s = p.us[u];
        x.s = s;
        x.lo = p.ulo[u] & ~7;
        x.N = (p.uhi[u] - x.lo + 15) & ~15;
        if (x.lo + x.N > p.B) x.lo = p.B - x.N;
        x.zo = p.uzoff[u];
        x.f = d.sfirst[s];
        x.k = d.sfirst[s + 1] - x.f;
        x.m = (int)(d.srowptr[s + 1] - d.srowptr[s]);
        x.G = (x.k + kFxRows - 1) / kFxRows;
        x.urel = p.urel[u];
        return true;
    }
    return false;
}
// Rows below chunk g start at `base`; tiles of the chunk: the diagonal one and those below.
__device__ __forceinline__ int fx_base(const FxNode& x, int g) { return min(kFxRows * (g + 1), x.k); }
__device__ __forceinline__ int fx_tiles(const FxNode& x, int g) {
    return 1 + (x.m - fx_base(x, g) + kFxRows - 1) / kFxRows;
}

// (kLimit: p.wait_limit polls per wait; a limit that is not a constant costs 2 to 4 % of the kernel.
// 576 threads put five warps on one of the four schedulers, 96 registers each: ptxas spills 196
// bytes of stores and 292 of loads.)
template <bool kLimit>
__global__ void __launch_bounds__(kFxThreads, 1)
    k_diag_fx(DevSym d, FxArgs p, double* __restrict__ out, Strides bs, DevStatus* status) {
    const uint32_t limit = kLimit ? p.wait_limit : kTcWaitLimit;
    const int band = blockIdx.y;
    out += band * bs.out;
    const int B = p.B, nst = fx_stages(B);
    extern __shared__ __align__(1024) unsigned char fsm[];
    unsigned char* Ar = fsm;
    unsigned char* Bs = fsm + (size_t)nst * kPiece;
    int* emax = reinterpret_cast<int*>(Bs + (size_t)kDig * B * kFxRows * 2);  // [2][64]
    uint64_t* bar = reinterpret_cast<uint64_t*>(emax + 128);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar + kFxBars);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* s_row = reinterpret_cast<int*>(tmem_slot + 4);           // [2][128] Z row of each row of a tile, -1: none
    short* s_exp = reinterpret_cast<short*>(s_row + 2 * kFxRows);  // [2][128] its exponent
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b = p.order[blockIdx.x];
    double* Z = p.Z + band * bs.Z + p.zbase[b];
    const int r0b = p.blk_ptr[b], nr = p.blk_ptr[b + 1] - r0b;
    const int u0 = p.uptr[b], u1 = p.uptr[b + 1];
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(tc_smem_u32(tmem_slot)),
                     "r"(kTcCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == kFxWork) {
        for (int q = 0; q < kFxBars; ++q)  // one arrival per worker warp, or one copy / commit
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(tc_smem_u32(bar + q)),
                         "r"(q == kFBF || q == kFCE ? kFxWork / 32 : 1));
        asm volatile("fence.mbarrier_init.release.cluster;");
        *abort = 0;
    }
    const int64_t zsz = p.zbase[b + 1] - p.zbase[b];
    for (int64_t i = 2 * tid; i < zsz; i += 2 * kFxThreads) *reinterpret_cast<double2*>(Z + i) = make_double2(0.0, 0.0);
    if (tid < 128) emax[tid] = 0;
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (tid < nr) Z[(int64_t)p.rhs_zrow[r0b + tid] * B + tid] =
        fx_pow2(-fx_scale_exp(p.D[band * bs.n + p.rhs_col[r0b + tid]]));
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tmem_slot;
    __syncthreads();
    uint32_t a_issued = 0;  // copies and finished tiles, for the drain below
    uint32_t tiles_issued = 0;
    bool partial = false;   // MMAs issued since the last commit to kFCF
    if (warp == kFxWork / 32) {
        if (lane == 0) {
            int u = u0 - 1;
            FxNode x;
            bool ok = true;
            while (ok && fx_next(d, p, u, u1, x)) {
                const unsigned char* src = p.pack + ((int64_t)band * p.npieces + p.pptr[x.s]) * kPiece;
                int np = 0;
                for (int g = 0; g < x.G; ++g)
                    np += fx_tiles(x, g) * ((min(kFxRows, x.k - g * kFxRows) + kFxSub - 1) / kFxSub);
                for (int t = 0; t < np && ok; ++t) {
                    const uint32_t st = a_issued % nst;
                    if (a_issued >= (uint32_t)nst && !fx_wait(bar + kFAE + st, (a_issued / nst - 1) & 1u, abort, limit)) {
                        ok = false;
                        break;
                    }
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                                 :: "r"(tc_smem_u32(bar + kFAF + st)), "r"(kPiece) : "memory");
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 :: "r"(tc_smem_u32(Ar + st * kPiece)), "l"(src + (size_t)t * kPiece), "r"(kPiece),
                                    "r"(tc_smem_u32(bar + kFAF + st)) : "memory");
                    ++a_issued;
                }
            }
            if (!ok) *abort = 1;
        }
    } else if (warp == kFxWork / 32 + 1) {
        if (lane == 0) {
            int u = u0 - 1;
            FxNode x;
            bool ok = true;
            uint32_t piece = 0, bfull = 0;
            const uint32_t bb = tc_smem_u32(Bs);
            while (ok && fx_next(d, p, u, u1, x)) {
                const uint32_t id0 = (1u << 4) | ((uint32_t)(kFxRows >> 4) << 24);
                const int most = 256 / x.N;  // planes of z in one MMA
                for (int g = 0; g < x.G && ok; ++g) {
                    const int w = min(kFxRows, x.k - g * kFxRows), nt = fx_tiles(x, g);
                    for (int i = 0; i < nt && ok; ++i) {
                        if (tiles_issued > 0 && !fx_wait(bar + kFCE, (tiles_issued - 1) & 1u, abort, limit)) { ok = false; break; }
                        if (i < 2 && !fx_wait(bar + kFBF, bfull++ & 1u, abort, limit)) { ok = false; break; }
                        for (int sub = 0; sub * kFxSub < w; ++sub) {
                            const uint32_t st = piece % nst;
                            if (!fx_wait(bar + kFAF + st, (piece / nst) & 1u, abort, limit)) { ok = false; break; }
                            asm volatile("tcgen05.fence::after_thread_sync;");
                            const uint32_t ab = tc_smem_u32(Ar + st * kPiece);
#pragma unroll
                            for (int q = 0; q < kDig; ++q) {
                                const uint64_t da = fx_desc(ab + q * kSlice, kFxSub * 16);
                                const uint32_t acc = (sub > 0 || q > 0) ? 1u : 0u;
                                const int nq = kDig - q, n0 = min(nq, most);
                                const uint32_t bo = bb + sub * 256;
                                fx_mma(tmem + q * x.N, da, fx_desc(bo, 2048), id0 | ((uint32_t)(n0 * x.N >> 3) << 17), acc);
                                if (nq > n0)
                                    fx_mma(tmem + (q + n0) * x.N, da, fx_desc(bo + n0 * x.N * 256, 2048),
                                           id0 | ((uint32_t)((nq - n0) * x.N >> 3) << 17), acc);
                            }
                            partial = true;
                            fx_commit(bar + kFAE + st);
                            ++piece;
                        }
                        if (!ok) break;
                        fx_commit(bar + kFCF);
                        partial = false;
                        ++tiles_issued;
                    }
                }
            }
            if (!ok) *abort = 1;
        }
    } else {
        int u = u0 - 1;
        FxNode x;
        bool ok = true;
        uint32_t ndone = 0, nslice = 0;
        const int quad = warp & 3, part = warp >> 2;  // read-out: rows 32 quad .., column groups part, part + 4
        // cutting: right-hand side n, groups of 8 rows r8 and r8 + rstep; its share of the
        // variance stays in a register until the end (summed in a fixed order)
        const int n = tid & (B - 1), r8 = tid / B, rstep = kFxWork / B;
        double va = 0.0;
        while (fx_next(d, p, u, u1, x)) {
            const int32_t* rel = p.rel + x.urel;
            const int32_t* rexp = p.rexp + ((int64_t)band * p.ntiles + p.tptr[x.s]) * kFxRows;
            const double* fr = p.fr + band * bs.n + x.f;
            // Rows c0 .. c0 + w of Z, columns lo .. lo + N, into the digit planes of Bs (hand_over),
            // and their squares times f into the variance (z_final).
            auto cut = [&](int c0, int w, bool z_final, bool hand_over) {
                const int cur = (int)(nslice & 1u) * 64;
                const int nl = n - x.lo;
                const bool on = nl >= 0 && nl < x.N;
                const double* src = Z + (int64_t)(x.zo + c0) * B + n;
                double v[2][8];
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int r = 8 * (r8 + h * rstep) + q;
                        v[h][q] = (on && r < w) ? __ldcg(src + (int64_t)r * B) : 0.0;
                    }
                if (hand_over) {
                    int em = -1000000;
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int q = 0; q < 8; ++q) em = max(em, fx_scaled_exp(v[h][q]));
                    // exponents are kept with an offset so that 0 means "no entry"
                    if (em > -1000000) atomicMax(&emax[cur + n], em + 65536);
                    fx_bar();
                    const int E = on ? emax[cur + n] - 65536 : 0;
                    if (tid < 64) emax[(cur ^ 64) + tid] = 0;
                    const int wp = (w + 15) & ~15;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int row = 8 * (r8 + h * rstep);
                        if (on && row < wp) {
                            unsigned long long xv[8];
#pragma unroll
                            for (int q = 0; q < 8; ++q) xv[q] = fx_fix(v[h][q], fx_scaled_exp(v[h][q]), E);
                            fx_store_planes<0>(Bs + (nl >> 3) * 2048 + (row >> 3) * 128 + (nl & 7) * 16,
                                               (size_t)(x.N >> 3) * 2048, xv);
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) fx_arrive(bar + kFBF);
                    ++nslice;
                }
                if (z_final && on) {  // while the first tile below is multiplied
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            if (8 * (r8 + h * rstep) + q < w)
                                va = fma(v[h][q] * fr[c0 + 8 * (r8 + h * rstep) + q], v[h][q], va);
                }
            };
            int tile = 0;
            // The rows of tile i of chunk g into the tables' half `tile & 1`: thread r < 128 row r; its
            // part of the rows' Z (all threads: a 128-byte line each) is asked for.
            auto table = [&](int g, int i, int tl) {
                const int lr = tid & (kFxRows - 1);
                const int row0 = i == 0 ? g * kFxRows : fx_base(x, g) + (i - 1) * kFxRows;
                const int rows = min(kFxRows, (i == 0 ? x.k : x.m) - row0), row = row0 + lr;
                const int zr = lr < rows ? (row < x.k ? x.zo + row : rel[row - x.k]) : -1;
                if (i > 0 && zr >= 0 && 16 * (tid / kFxRows) < x.N)
                    asm volatile("prefetch.global.L2 [%0];" :: "l"(Z + (int64_t)zr * B + x.lo + 16 * (tid / kFxRows)));
                if (tid < kFxRows) {
                    s_row[(tl & 1) * kFxRows + lr] = zr;
                    s_exp[(tl & 1) * kFxRows + lr] = (short)rexp[tl * kFxRows + lr];
                }
            };
            for (int g = 0; g < x.G; ++g) {
                const int c0 = g * kFxRows, w = min(kFxRows, x.k - c0), nt = fx_tiles(x, g);
                fx_bar();  // Z rows written by the other warps
                table(g, 0, tile);  // before the digits are handed over: read once their product is done
                cut(c0, w, false, true);
                for (int i = 0; i < nt; ++i, ++tile) {
                    // a warp whose wait ran out does no further work but meets every barrier
                    if (ok && !__all_sync(0xffffffffu, fx_wait(bar + kFCF, ndone & 1u, abort, limit))) {
                        ok = false;
                        *abort = 1;
                    }
                    ++ndone;
                    if (ok) {
                        asm volatile("tcgen05.fence::after_thread_sync;");
                        if (i + 1 < nt) table(g, i + 1, tile + 1);
                        // this thread's four rows of the tile: 32 quad + lane / 4 + 8 q
                        int zrow[4], re[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int lr = (tile & 1) * kFxRows + 32 * quad + (lane >> 2) + 8 * q;
                            zrow[q] = s_row[lr];
                            re[q] = s_exp[lr] - 65536 - 1022;
                        }
                        long long vi[2][2][4];  // [column group][16 rows][register]
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int cg = part + 4 * h;
                            if (cg * 8 < x.N) {
#pragma unroll
                                for (int r16 = 0; r16 < 2; ++r16) {
                                    const uint32_t ta = tmem + ((uint32_t)(32 * quad + 16 * r16) << 16) + cg * 8;
                                    uint32_t t[kDig][4];
#pragma unroll
                                    for (int l = 0; l < kDig; ++l) fx_ld16x8(ta + l * x.N, t[l]);
                                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                                    for (int j = 0; j < 4; ++j) {
                                        const uint32_t a[kDig] = {t[0][j], t[1][j], t[2][j], t[3][j], t[4][j], t[5][j], t[6][j]};
                                        vi[h][r16][j] = fx_join(a);
                                    }
                                }
                            }
                        }
                        asm volatile("tcgen05.fence::before_thread_sync;");
                        __syncwarp();
                        if (lane == 0) fx_arrive(bar + kFCE);
                        const int* be = emax + ((nslice - 1) & 1u) * 64 + x.lo;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int cc = 8 * (part + 4 * h) + 2 * (lane & 3);
                            if (8 * (part + 4 * h) < x.N) {
                                const int b0 = be[cc], b1 = be[cc + 1];
                                double2* zp = reinterpret_cast<double2*>(Z + x.lo + cc);
                                double2 o[4];
#pragma unroll
                                for (int q = 0; q < 4; ++q)
                                    o[q] = (i > 0 && zrow[q] >= 0) ? __ldcg(zp + (int64_t)zrow[q] * (B / 2)) : make_double2(0.0, 0.0);
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    const double a = fx_value(vi[h][q >> 1][2 * (q & 1)], re[q] + b0);
                                    const double c = fx_value(vi[h][q >> 1][2 * (q & 1) + 1], re[q] + b1);
                                    const double2 z = i > 0 ? make_double2(o[q].x - a, o[q].y - c) : make_double2(a, c);
                                    if (zrow[q] >= 0) __stcg(zp + (int64_t)zrow[q] * (B / 2), z);
                                }
                            }
                        }
                    }
                    if (i == 0) {
                        fx_bar();  // the chunk's y is complete
                        cut(c0, w, true, nt > 1);
                    }
                }
            }
        }
        // every product has been read: the digit planes' space takes the partial sums
        double* part_sum = reinterpret_cast<double*>(Bs);
        fx_bar();
        if (ok) part_sum[tid] = va;
        fx_bar();
        if (ok && tid < nr) {
            double a = 0.0;
            for (int q = 0; q < rstep; ++q) a += part_sum[q * B + tid];
            va = a;
        }
        if (!ok) *abort = 1;
        else if (tid < nr) out[p.rhs_out[r0b + tid]] = va;
    }
    // ---- a wait ran out somewhere: let the copies and products in flight finish (bounded),
    // report it and leave the variances; tensor memory is released either way
    __syncthreads();
    const bool failed = *abort != 0;
    if (failed) {
        if (tid == kFxWork) {
            atomicOr(&status->flags, FLAG_TIMEOUT);
            for (uint32_t q = a_issued > (uint32_t)nst ? a_issued - nst : 0; q < a_issued; ++q)
                tc_wait(bar + kFAF + q % nst, (q / nst) & 1u);
        }
        if (tid == kFxWork + 32 && (partial || tiles_issued > 0)) {
            if (partial) fx_commit(bar + kFCF);  // tracks every MMA issued so far
            tc_wait(bar + kFCF, (partial ? tiles_issued : tiles_issued - 1) & 1u);
        }
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(kTcCols));
}

}  // namespace

size_t diag_fx_pack_bytes(int64_t npieces) { return (size_t)npieces * kPiece; }

cudaError_t diag_fx_setup() {
    const cudaError_t e =
        cudaFuncSetAttribute(k_diag_fx<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fx_smem(kFxMaxBlock));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_diag_fx<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fx_smem(kFxMaxBlock));
}

void launch_tile_inverses(const DevSym& d, const DevTileInv& x, const double* L, int nb, const Strides& bs,
                          cudaStream_t st) {
    if (x.ncta == 0 || nb == 0) return;
    k_fx_tinv<<<dim3((unsigned)x.ncta, nb), 128, 0, st>>>(d, x.dtiles, x.xoff, x.nx, L, x.xinv, x.xinvt, bs.L);
}

void launch_diag_fx(const DevSym& d, const DevDiagPlan& dp, const DevDiagFx& p, const DevTileInv& x, const double* L, const double* D,
                    double* out, int nb, const Strides& bs, DevStatus* status, int wait_limit, cudaStream_t st) {
    if (dp.nblocks == 0 || nb == 0) return;
    if (dp.fx_ninv > 0) {  // (the factorization did not make them)
        DevTileInv part = x;
        part.dtiles = dp.fx_inv;
        part.ncta = dp.fx_ninv;
        launch_tile_inverses(d, part, L, nb, bs, st);
    }
    k_fx_pack<<<dim3((unsigned)dp.fx_ntiles, nb), kFxRows, 0, st>>>(d, p.tiles, p.tdiag, dp.fx_tiles, p.ntiles, p.npieces,
                                                                    x.xoff, x.nx, L, D, x.xinv, p.pack, p.rexp, p.fr,
                                                                    bs.L, bs.n);
    FxArgs a{dp.B, dp.order_tc, dp.blk_ptr, dp.uptr, dp.us, dp.ulo, dp.uhi, dp.uzoff, dp.rel, dp.rhs_out,
             dp.rhs_zrow, dp.rhs_col, dp.urel, dp.zbase, dp.Z, p.pptr, p.tptr, p.npieces, p.ntiles, p.pack, p.rexp,
             D, p.fr, wait_limit > 0 ? (uint32_t)wait_limit : wait_limit < 0 ? 0u : kTcWaitLimit};
    const dim3 g(dp.nblocks, nb);
    if (wait_limit == 0) k_diag_fx<false><<<g, kFxThreads, fx_smem(dp.B), st>>>(d, a, out, bs, status);
    else k_diag_fx<true><<<g, kFxThreads, fx_smem(dp.B), st>>>(d, a, out, bs, status);
}

}  // namespace spi

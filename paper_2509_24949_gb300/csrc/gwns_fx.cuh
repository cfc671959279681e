// gwns_fx.cuh -- the FP64 form's bin arithmetic off the FP64 pipe. GB300 issues
// one FP64 warp instruction per 64 cycles per SM sub-partition (measured; FP32
// one per cycle, a 32 x 32 -> 64-bit integer multiply-add one per four), so a
// bin's 8 phase terms, its sines and cosines and its complex products cost
// thousands of cycles in FP64 and a few hundred in the split arithmetic here:
//
//  * the phase in turns as a fixed-point sum of products, modulo one turn. The
//    grid is cut into blocks of frequency where the phases have fallen far enough
//    (FxBlocks). In a block the basis and the frequency are 59-bit integers scaled
//    to their largest value there, a point's coefficients 60-bit integers on one
//    scale per point and block: the unit is 2^-59 of the power of two above the
//    point's largest term in the block, where FP64 rounds that term at 2^-53, so
//    that also a block's last bins are rounded below FP64's sums (0.01 to 0.5 of
//    their rms, by octave). One scale for a whole grid would give every bin the
//    rounding of the lowest frequency's terms: rms error of the phases at 50 to 400 Hz, chirp
//    mass 1.2, grid from 20 / 5 / 1 / 0.1 Hz, FP64 1.3e-13 rad, one scale with
//    58-bit coefficients and floored halves 5e-13 / 7e-12 / 1.2e-10 / 3.9e-9, blocks
//    1.0e-13 (the tabulated basis' own rounding).
//    Both factors are split at 2^30 into a high half and a signed low half, so that
//    the high and the cross products add up in two 64-bit accumulators without
//    carries: three multiply-adds per term; the dropped low products average to
//    nothing (with low halves that are never negative they would shift every
//    bin's phase the same way).
//  * exp(2 pi i phase): the top 10 fraction bits pick cos and sin of k 2 pi/1024
//    from a table (double-float, half a turn, the other half by sign), the rest
//    r, |r| < 0.0031 rad, enters through sin r and cos r - 1 by their Taylor
//    polynomials and one complex product, all in double-float (absolute error
//    about 1e-15).
//  * the products with the weighted data and their sums in double-float
//    (48 bits), the data scaled by a power of two per detector. With the phases'
//    finer rounding the sums as a whole are no further from the exact ones than
//    an FP64 loop's (rms error over the weights' norm, FP64 -> here, 512 bins
//    1.6e-14 -> 1.3e-14, 4017 1.4e-14 -> 0.9e-14, low masses on 64,897 bins
//    1.6e-12 -> 1.0e-12).
//
// Plain C++ besides the qualifiers, so the same code compiles for the host
// (where a CPU test checks it against 60-digit references) and for sm_103a.
#pragma once
#include "gwns_df.cuh"

namespace gwns {

constexpr int FX_NB = 8;            // phase basis functions
constexpr int FX_DET = 4;           // detectors at most
constexpr int FX_ABITS = 60;        // coefficients: |A| <= 2^60
constexpr int FX_BBITS = 59;        // tables: |b| <= 2^59
constexpr int FX_SC = 512;          // table points over half a turn
constexpr int FX_NODES = 32;        // nodes of a tile (below)
constexpr int FX_LG0 = 6;           // log2 of the shortest tile's bins
constexpr int FX_LEV = 10;          // tile levels at most
constexpr int FX_SEG = 2 * FX_LEV + 1;
constexpr int FX_BLK = 6;           // blocks of frequency at most
constexpr int64_t FX_HALF = 1 << 29;    // the cross products' sum starts here: fx_phase rounds

// A signed integer of up to 61 bits as 2^30 h + l, -2^29 <= l < 2^29.
struct fx2 {
    int32_t h, l;
};

// Blocks of frequency: block b starts at bin (relative binning: at edge) bin[b],
// and e[b] are the binary exponents that bring its basis functions and
// frequencies below one.
struct FxBlocks {
    int32_t n;
    int32_t bin[FX_BLK];
    int32_t e[FX_BLK][FX_NB + 1];
};

// One point's fixed-point phase coefficients in a block (a: basis, t: detector
// delays) in units of 2^(E - 60) turns per full-scale table entry, 2^E the power
// of two above its largest term; c0 in the phase sum's unit 2^(E - 59) turns;
// sh = E + 5 lifts the sum's fraction to 64 bits; end: the running row that the
// block ends at.
struct FxCoef {
    fx2 a[FX_NB];
    fx2 t[FX_DET];
    int64_t c0;
    int32_t sh, end;
};
struct FxPoint {
    FxCoef blk[FX_BLK];
    int32_t bad;        // a coefficient is not finite: the sums are NaN
    // the rows to sum: running index r < rows lies in the first segment with
    // r < end and is table row r + off
    int32_t nseg, rows;
    struct { int32_t end, off; } seg[FX_SEG];
};

// Tiles of the long grids. Over a tile of 2^(FX_LG0 + l) bins (level l) the
// phase of any point of the prior differs from a reference phase by a few
// radians, so exp(i (Psi - Psi_ref)) is a polynomial of degree 31 there to 1e-15
// and the tile's sum over bins is exactly a sum over FX_NODES Chebyshev nodes,
// with the bins' weighted data gathered once into weights of the nodes. Level l
// covers the grid from bin first[l] on (where its bound holds) with rows from
// row[l] on; rows 0 .. N-1 are the bins themselves.
struct FxTiles {
    int32_t nlev;
    int32_t first[FX_LEV], row[FX_LEV];
};

struct fxe {
    float rh, rl, ih, il;       // double-float complex
};

DFI fx2 fx_split(int64_t v) {
    const int64_t h = (v + FX_HALF) >> 30;
    return fx2{(int32_t)h, (int32_t)(v - (h << 30))};
}

#if defined(__CUDA_ARCH__)
DFI uint64_t fx_mulhi(uint64_t a, uint64_t b) { return __umul64hi(a, b); }
DFI uint64_t fx_bits(double x) { return (uint64_t)__double_as_longlong(x); }
#else
DFI uint64_t fx_mulhi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
DFI uint64_t fx_bits(double x) { uint64_t b; memcpy(&b, &x, 8); return b; }
#endif

// |x| (or |x| / 2 pi, TURNS) = m 2^e with m a 64-bit integer of at least 62
// significant bits, from the double's bits alone; 0 (and anything below 2^-1022)
// gives m = 0. Not finite: *bad is set. Returns e.
template <bool TURNS>
DFI int fx_mantissa(double x, uint64_t *m, int32_t *bad) {
    const uint64_t b = fx_bits(x);
    const int ex = (int)(b >> 52) & 0x7ff;
    if (ex == 0x7ff) *bad = 1;
    if (ex == 0) { *m = 0; return -100000; }
    const uint64_t q = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 11;
    // 1/(2 pi) = 0xA2F9836E4E44152A 2^-66 (rounded)
    *m = TURNS ? fx_mulhi(q, 0xA2F9836E4E44152Aull) : q;
    return TURNS ? ex - 1088 : ex - 1086;
}
// m 2^-s rounded, with x's sign (s >= 1)
DFI int64_t fx_scaled(uint64_t m, int s, double x) {
    const uint64_t v = s > 64 ? 0 : ((m >> (s - 1)) + 1) >> 1;
    return (fx_bits(x) >> 63) ? -(int64_t)v : (int64_t)v;
}

// The shifts of a coefficient's mantissa (|x| < 2^ex) to the unit 2^(E - FX_ABITS), of
// the constant phase's (one more) and of the phase sum's fraction to 2^-64 turns.
DFI int fx_shift(int E, int ex) { return E - ex + 64 - FX_ABITS; }
DFI int fx_lift(int E) { return E + 65 - FX_ABITS; }

// Table entry of a double with |v| <= 2^eb.
#if defined(__CUDACC__)
__device__ __forceinline__ fx2 fx_table(double v, int eb) {
    return fx_split(__double2ll_rn(scalbn(v, FX_BBITS - eb)));
}
#else
DFI fx2 fx_table(double v, int eb) { return fx_split(llrint(scalbn(v, FX_BBITS - eb))); }
#endif

// Block of bin j.
DFI int fx_block(const FxBlocks &K, int j) {
    int b = 0;
    while (b + 1 < K.n && j >= K.bin[b + 1]) b++;
    return b;
}
// Ends of the blocks that a segment closes: bins [pos, e) by units of 2^lg bins
// with rpt rows each from running row `rows` on. A unit belongs to the block of its
// first bin.
DFI void fx_block_ends(const FxBlocks *K, FxPoint &o, int &b, int pos, int e, int lg, int rpt, int rows) {
    for (int it = 0; K && it < FX_BLK && b + 1 < K->n && K->bin[b + 1] < e; it++) {
        const int d = K->bin[b + 1] > pos ? K->bin[b + 1] - pos : 0;
        o.blk[b++].end = rows + ((d + (1 << lg) - 1) >> lg) * rpt;
    }
}

// The segments of the bins 0 .. n - 1: bins below the first tiled one, then tiles
// of growing length, each level up to the next one's first bin, then of
// shrinking length up to the cutoff and the last few bins one by one. With K also
// the running rows that the blocks end at.
DFI void fx_layout(const FxTiles &T, const FxBlocks *K, bool tiles, int n, FxPoint &o) {
    int ns = 0, rows = 0, pos = 0, b = 0;
    if (tiles && T.nlev > 0 && n > T.first[0]) {
        if (T.first[0] > 0) {
            fx_block_ends(K, o, b, 0, T.first[0], 0, 1, 0);
            pos = rows = T.first[0];
            o.seg[ns].end = rows;
            o.seg[ns++].off = 0;
        }
        int l = 0, step = 1;
        for (int it = 0; it < 2 * FX_LEV && l >= 0; it++) {
            const int lg = FX_LG0 + l;
            int e = n >> lg << lg;
            bool up = false;
            if (step > 0 && l + 1 < T.nlev && e >= T.first[l + 1]) {
                e = T.first[l + 1];
                up = true;
            }
            if (e > pos) {
                fx_block_ends(K, o, b, pos, e, lg, FX_NODES, rows);
                o.seg[ns].off = T.row[l] + ((pos - T.first[l]) >> lg) * FX_NODES - rows;
                rows += ((e - pos) >> lg) * FX_NODES;
                o.seg[ns++].end = rows;
                pos = e;
            }
            if (!up) step = -1;
            l += step;
        }
    }
    if (n > pos) {
        fx_block_ends(K, o, b, pos, n, 0, 1, rows);
        o.seg[ns].off = pos - rows;
        rows += n - pos;
        o.seg[ns++].end = rows;
    }
    if (K) o.blk[b].end = 0x7fffffff;
    o.nseg = ns;
    o.rows = rows;
}
DFI void fx_segments(const FxTiles &T, bool tiles, int n, FxPoint &o) { fx_layout(T, nullptr, tiles, n, o); }

// The blocks of a grid. FP64 rounds a bin's phase by its size there: the Newtonian
// term 3/128 (pi T_sun Mc f)^(-5/3) (at the prior's lowest chirp mass mc), twice
// 2 pi f tau (tau a typical delay: its product and its sum are rounded) and 20 rad
// for the rest; the split arithmetic rounds it by the block's largest term at 2^-5
// to 2^-6 of that. So a block ends where the phases have fallen to 1/40 of its first
// bin's Newtonian term (a larger fall only where FX_BLK blocks do not suffice, on
// more than five decades of frequency). From 20 Hz, chirp masses of 1.1 or more take
// one block.
// A block's largest values are taken over its bins and the tiles that start in it,
// whose nodes reach half a bin beyond the tile's bins. Every basis function is
// monotone between its ends but f^(1/3) ln f, whose minimum is -3/e at f = e^-3.
inline void fx_make_blocks(int N, double f0, double df, double mc, double tau, const FxTiles &T, FxBlocks &K) {
    const double f1 = f0 + (double)(N - 1) * df;
    auto newton = [&](double f) { return 0.0234375 * pow(3.141592653589793 * 4.925490947641267e-6 * mc * f, -5.0 / 3.0); };
    double fall = 40.0;
    for (int it = 0; it < 64; it++, fall *= 1.5) {
        K.n = 1;
        K.bin[0] = 0;
        int more = 0;
        double top = newton(f0);
        double f = f0;
        for (int s = 0; s < (1 << 14) && f < f1; s++, f *= 1.09) {      // (a subnormal f may not grow)
            if (!(top > fall * (newton(f) + 12.566370614359172 * f * tau + 20.0))) continue;
            const double j = ceil((f - f0) / df);
            if (!(j < (double)N)) break;
            top = newton(f);
            if ((int)j <= K.bin[K.n - 1]) continue;
            if (K.n == FX_BLK) { more = 1; break; }
            K.bin[K.n++] = (int)j;
        }
        if (!more) break;
    }
    for (int b = 0; b < K.n; b++) {
        const int last = (b + 1 < K.n ? K.bin[b + 1] : N) - 1;
        double lo = f0 + (double)K.bin[b] * df, hi = f0 + (double)last * df;
        for (int l = 0; l < T.nlev; l++) {
            const int lg = FX_LG0 + l;
            if (last < T.first[l]) continue;
            int end = ((((last - T.first[l]) >> lg) + 1) << lg) + T.first[l];
            if (end > N) end -= 1 << lg;
            hi = fmax(hi, f0 + ((double)end - 0.5) * df);
            if (lo > 8.0 * df) lo = fmin(lo, f0 + ((double)K.bin[b] - 0.5) * df);
        }
        double mx[FX_NB + 1] = {};
        for (int i = 0; i < 2; i++) {
            const double f = i == 0 ? lo : hi, r = cbrt(f), l = log(f);
            const double B[FX_NB + 1] = {1.0 / (f * r * r), 1.0 / f, 1.0 / (r * r), 1.0 / r, l, r, r * l, r * r, f};
            for (int m = 0; m <= FX_NB; m++) mx[m] = fmax(mx[m], fabs(B[m]));
        }
        if (lo < 0.05 && hi > 0.049) mx[6] = fmax(mx[6], 1.2);
        for (int m = 0; m <= FX_NB; m++) K.e[b][m] = ilogb(fmin(fmax(mx[m] * (1.0 + 1e-12), 1e-300), 1e300)) + 1;
    }
}

// A point's coefficients in block b from its basis coefficients a [rad], delays
// tau [s] and constant phase c0 [rad]; bad is set where one is not finite.
inline void fx_coef(const FxBlocks &K, int b, const double *a, const double *tau, int nt, double c0, FxCoef &o,
                    int32_t &bad) {
    uint64_t m[FX_NB + FX_DET + 1];
    int ex[FX_NB + FX_DET + 1], E = 0;
    for (int i = 0; i < FX_NB; i++) ex[i] = fx_mantissa<true>(a[i], &m[i], &bad) + K.e[b][i] + 64;
    for (int d = 0; d < nt; d++) ex[FX_NB + d] = fx_mantissa<false>(tau[d], &m[FX_NB + d], &bad) + K.e[b][FX_NB] + 64;
    uint64_t mc;
    const int ec = fx_mantissa<true>(c0, &mc, &bad) + 64;
    for (int i = 0; i < FX_NB + nt; i++) E = ex[i] > E ? ex[i] : E;
    E = ec > E ? ec : E;
    for (int i = 0; i < FX_NB; i++) o.a[i] = fx_split(fx_scaled(m[i], fx_shift(E, ex[i]), a[i]));
    for (int d = 0; d < nt; d++) o.t[d] = fx_split(fx_scaled(m[FX_NB + d], fx_shift(E, ex[FX_NB + d]), tau[d]));
    o.c0 = fx_scaled(mc, fx_shift(E, ec) + 1, c0);
    o.sh = fx_lift(E);
}

// One term's products: hi += a.h b.h, cr += a.h b.l + a.l b.h (the low product,
// within 1/4 of the unit either way, is dropped). |a.h| <= 2^30, |b.h| <= 2^29 and
// |l| <= 2^29: the nine terms of a phase stay below 2^63 in either sum.
DFI void fx_mac(int64_t &hi, int64_t &cr, fx2 a, fx2 b) {
    hi += (int64_t)a.h * b.h;
    cr += (int64_t)a.h * b.l;
    cr += (int64_t)a.l * b.h;
}
// The phase's fraction of a turn (2^-64 turns) from the sums.
DFI uint64_t fx_phase(int64_t hi, int64_t cr, int32_t sh) {
    const uint64_t p = (uint64_t)(hi + (cr >> 30));
    return sh > 63 ? 0 : p << sh;
}

// exp(2 pi i F 2^-64). tab: FX_SC points (cos h, cos l, sin h, sin l) of
// k 2 pi/1024.
#if defined(__CUDACC__)
typedef float4 fx_f4;
#else
struct fx_f4 { float x, y, z, w; };
#endif
DFI fxe fx_cis(uint64_t F, const fx_f4 *tab) {
    const uint32_t fh = (uint32_t)(F >> 32), fl = (uint32_t)F;
    const uint32_t g = fh + 0x200000u;                    // round to the nearest table point
    // rest in units of 2^-32 turns: r0 = g mod 2^22 - 2^21 (exact) + r1 2^-23
    const float r0 = f_sub(i_as_f((int32_t)(0x4b000000u | (g & 0x3fffffu))), 10485760.0f);
    const float r1 = f_sub(i_as_f((int32_t)(0x4b000000u | (fl >> 9))), 8388608.0f);
    const fx_f4 T = tab[(g >> 22) & (FX_SC - 1)];
    const uint32_t sgn = g & 0x80000000u;                 // second half turn: -T
    const float ch = i_as_f((int32_t)((uint32_t)f_as_i(T.x) ^ sgn)), cl = i_as_f((int32_t)((uint32_t)f_as_i(T.y) ^ sgn));
    const float sh = i_as_f((int32_t)((uint32_t)f_as_i(T.z) ^ sgn)), sl = i_as_f((int32_t)((uint32_t)f_as_i(T.w) ^ sgn));
    // r = p + e [rad]
    const float CH = (float)1.4629180792671596e-9, CL = (float)(1.4629180792671596e-9 - (double)CH);   // 2 pi 2^-32
    const float p = f_mul(r0, CH);
    float e = f_fma(r0, CH, -p);
    e = f_fma(r0, CL, e);
    e = f_fma(r1, (float)(1.4629180792671596e-9 / 8388608.0), e);
    // cos r - 1 = c1 + c2, sin r = p + s2
    const float r2 = f_mul(p, p), r2e = f_fma(p, p, -r2);
    const float c1 = f_mul(-0.5f, r2);
    const float c2 = f_fma(f_mul(c1, c1), 1.0f / 6.0f, f_fma(-p, e, f_mul(-0.5f, r2e)));
    const float s2 = f_fma(f_mul(r2, p), f_fma(r2, 1.0f / 120.0f, -1.0f / 6.0f), f_fma(c1, e, e));
    // T + T (c + i s): the products' sum b (below 0.0031) with the table's low part,
    // then T + b by size (the table's nonzero entries exceed 0.0061), then the low parts
    fxe E;
    {
        const float u = f_mul(sh, p), ue = f_fma(sh, p, -u);
        const float v = f_mul(ch, c1), ve = f_fma(ch, c1, -v);
        const dfl b = two_sum_f(-u, v), bc = two_sum_f(b.h, cl), x = fast_two_sum_f(ch, bc.h);
        float l = f_add(f_add(b.l, bc.l), f_sub(ve, ue));
        l = f_fma(ch, c2, l);
        l = f_fma(-sh, s2, l);
        l = f_fma(-sl, p, l);
        l = f_fma(cl, c1, l);
        E.rh = x.h;
        E.rl = f_add(x.l, l);
    }
    {
        const float u = f_mul(ch, p), ue = f_fma(ch, p, -u);
        const float v = f_mul(sh, c1), ve = f_fma(sh, c1, -v);
        const dfl b = two_sum_f(u, v), bc = two_sum_f(b.h, sl), x = fast_two_sum_f(sh, bc.h);
        float l = f_add(f_add(b.l, bc.l), f_add(ve, ue));
        l = f_fma(sh, c2, l);
        l = f_fma(ch, s2, l);
        l = f_fma(cl, p, l);
        l = f_fma(sl, c1, l);
        E.ih = x.h;
        E.il = f_add(x.l, l);
    }
    return E;
}

// zh + zl += w E for one real product of double-floats
DFI void fx_acc(float &zh, float &zl, float wh, float wl, float eh, float el) {
    const float p = f_mul(wh, eh);
    float e = f_fma(wh, eh, -p);
    e = f_fma(wh, el, e);
    e = f_fma(wl, eh, e);
    const dfl s = two_sum_f(zh, p);
    zh = s.h;
    zl = f_add(zl, f_add(s.l, e));
}
// Z += w E, w = (re h, re l, im h, im l), z = (re, im)
DFI void fx_cmac(float (&zh)[2], float (&zl)[2], fx_f4 w, fxe E) {
    fx_acc(zh[0], zl[0], w.x, w.y, E.rh, E.rl);
    fx_acc(zh[0], zl[0], -w.z, -w.w, E.ih, E.il);
    fx_acc(zh[1], zl[1], w.x, w.y, E.ih, E.il);
    fx_acc(zh[1], zl[1], w.z, w.w, E.rh, E.rl);
}

}  // namespace gwns

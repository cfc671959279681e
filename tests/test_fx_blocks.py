"""The split arithmetic's blocks of frequency: phases and bin sums no further from the
exact ones than FP64's, wherever the grid starts. The device header is compiled here
for the host, beside the same sums in FP64 (fused multiply-adds for the phase, a
rotation per detector, as a plain FP64 bin loop has them)."""
import math
import random
import shutil
import subprocess

import pytest

from test_df_math import CSRC

mp = pytest.importorskip("mpmath")

DRIVER = r"""
#include <stdio.h>
#include <stdlib.h>
#include "gwns_fx.cuh"
using namespace gwns;
static double rd() { double v; if (scanf("%lf", &v) != 1) exit(1); return v; }
static fx_f4 tab[FX_SC];
static const long double PIL = 3.14159265358979323846264338327950288L;

// phase in 2^-64 turns at a table row of block b
static uint64_t phase(const FxCoef &c, const int32_t *e, const double *B) {
    int64_t hi = c.c0, cr = FX_HALF;
    for (int m = 0; m < 8; m++) fx_mac(hi, cr, c.a[m], fx_table(B[m], e[m]));
    fx_mac(hi, cr, c.t[0], fx_table(B[8], e[8]));
    return fx_phase(hi, cr, c.sh);
}
static void basis(double f, double *B) {
    const double c = cbrt(f), l = log(f);
    const double b[9] = {1.0 / (f * c * c), 1.0 / f, 1.0 / (c * c), 1.0 / c, l, c, c * l, c * c, f};
    for (int m = 0; m < 9; m++) B[m] = b[m];
}

int main() {
    for (int i = 0; i < FX_SC; i++) {
        const double c = rd(), s = rd();
        tab[i] = fx_f4{(float)c, (float)(c - (double)(float)c), (float)s, (float)(s - (double)(float)s)};
    }
    char op[16];
    while (scanf("%15s", op) == 1) {
        const int N = (int)rd();
        const double f0 = rd(), df = rd();
        const double mc = rd(), tscale = rd();      // the prior's lowest chirp mass, a typical delay
        FxTiles T;
        T.nlev = 0;
        FxBlocks K;
        if (op[0] == 'b') {             // tile levels' first bins and rows: blocks, then for counts the blocks' ends
            T.nlev = (int)rd();
            for (int i = 0; i < T.nlev; i++) { T.first[i] = (int)rd(); T.row[i] = (int)rd(); }
            fx_make_blocks(N, f0, df, mc, tscale, T, K);
            printf("%d", K.n);
            for (int b = 0; b < K.n; b++) {
                printf(" %d", K.bin[b]);
                for (int m = 0; m < 9; m++) printf(" %d", K.e[b][m]);
            }
            for (int n = (int)rd(); n > 0; n--) {
                FxPoint o;
                fx_layout(T, &K, true, (int)rd(), o);
                printf(" %d", o.rows);
                int b = 0;
                do printf(" %d", o.blk[b].end);
                while (o.blk[b++].end != 0x7fffffff);
            }
            printf("\n");
            continue;
        }
        fx_make_blocks(N, f0, df, mc, tscale, T, K);
        double a[8], B[9];
        for (int m = 0; m < 8; m++) a[m] = rd();
        const double tau = rd(), c0 = rd();
        const double c0r = c0 - 2 * M_PI * rint(c0 / (2 * M_PI));
        FxCoef C[FX_BLK];
        int32_t bad = 0;
        for (int b = 0; b < K.n; b++) fx_coef(K, b, a, &tau, 1, c0, C[b], bad);
        if (op[0] == 'p') {             // phases at given bins: split (2^-64 turns), FP64 [rad], unit exponent, basis
            for (int n = (int)rd(); n > 0; n--) {
                const int j = (int)rd(), b = fx_block(K, j);
                basis(fma((double)j, df, f0), B);
                double psi = c0r;
                for (int m = 0; m < 8; m++) psi = fma(a[m], B[m], psi);
                psi += 2 * M_PI * B[8] * tau;
                printf("%llu %a %d", (unsigned long long)phase(C[b], K.e[b], B), psi, C[b].sh - 5);
                for (int m = 0; m < 9; m++) printf(" %a", B[m]);
                printf("\n");
            }
        } else {                        // Z = sum w exp(i phase) over n bins: errors of FP64's and the split sums
            const int n = (int)rd();
            float zh[32][2] = {}, zl[32][2] = {};
            double hr[32] = {}, hi[32] = {}, pr, pi_, fr = 0, fi = 0, sr = 0, si = 0;
            long double zr = 0, zi = 0, ww = 0;
            sincos(2 * M_PI * (32 * df) * tau, &pi_, &pr);
            double *w = (double *)malloc(sizeof(double) * 2 * n);
            for (int j = 0; j < 2 * n; j++) w[j] = rd();
            for (int j = 0; j < n; j++) {
                const int t = j & 31, b = fx_block(K, j);
                basis(fma((double)j, df, f0), B);
                const long double f = B[8], c = cbrtl(f), l = logl(f);
                const long double L[8] = {1 / (f * c * c), 1 / f, 1 / (c * c), 1 / c, l, c, c * l, c * c};
                long double ph = c0 + 2 * PIL * f * tau;
                for (int m = 0; m < 8; m++) ph += a[m] * L[m];
                zr += w[2 * j] * cosl(ph) - w[2 * j + 1] * sinl(ph);
                zi += w[2 * j] * sinl(ph) + w[2 * j + 1] * cosl(ph);
                ww += (long double)w[2 * j] * w[2 * j] + (long double)w[2 * j + 1] * w[2 * j + 1];
                const float v[4] = {(float)w[2 * j], (float)(w[2 * j] - (double)(float)w[2 * j]), (float)w[2 * j + 1],
                                    (float)(w[2 * j + 1] - (double)(float)w[2 * j + 1])};
                fx_cmac(zh[t], zl[t], fx_f4{v[0], v[1], v[2], v[3]}, fx_cis(phase(C[b], K.e[b], B), tab));
            }
            for (int j = n - 1; j >= 0; j--) {      // the detector's factor by Horner's rule over a lane's bins
                const int t = j & 31;
                basis(fma((double)j, df, f0), B);
                double psi = c0r, s, co;
                for (int m = 0; m < 8; m++) psi = fma(a[m], B[m], psi);
                sincos(psi, &s, &co);
                const double cr = fma(w[2 * j], co, -w[2 * j + 1] * s), ci = fma(w[2 * j], s, w[2 * j + 1] * co);
                const double r = fma(hr[t], pr, fma(-hi[t], pi_, cr));
                hi[t] = fma(hr[t], pi_, fma(hi[t], pr, ci));
                hr[t] = r;
            }
            for (int t = 0; t < 32; t++) {
                double rs, rc;
                sincos(2 * M_PI * (f0 + t * df) * tau, &rs, &rc);
                const double r = rc * hr[t] - rs * hi[t], i = rc * hi[t] + rs * hr[t];
                hr[t] = t < n ? r : 0;
                hi[t] = t < n ? i : 0;
            }
            for (int o = 16; o; o /= 2)
                for (int t = 0; t < o; t++) {
                    hr[t] += hr[t + o];
                    hi[t] += hi[t + o];
                    for (int k = 0; k < 2; k++) {
                        const dfl v = df_add(dfl{zh[t][k], zl[t][k]}, dfl{zh[t + o][k], zl[t + o][k]});
                        zh[t][k] = v.h;
                        zl[t][k] = v.l;
                    }
                }
            fr = hr[0]; fi = hi[0];
            sr = (double)zh[0][0] + (double)zl[0][0]; si = (double)zh[0][1] + (double)zl[0][1];
            printf("%Lg %Lg\n", hypotl(fr - zr, fi - zi) / sqrtl(ww), hypotl(sr - zr, si - zi) / sqrtl(ww));
            free(w);
        }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fxblocks")
    (d / "drv.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O1", "-std=gnu++17", "-ffp-contract=off", "-fno-fast-math", "-I", CSRC, str(d / "drv.cpp"),
                    "-o", str(d / "drv"), "-lm"], check=True)
    mp.mp.dps = 60
    head = "\n".join("%r %r" % (float(mp.cospi(mp.mpf(i) / 512)), float(mp.sinpi(mp.mpf(i) / 512))) for i in range(512))

    def run(lines):
        r = subprocess.run([str(d / "drv")], input=head + "\n" + "\n".join(lines) + "\n", capture_output=True,
                           text=True, check=True)
        return r.stdout.splitlines()
    return run


def point(rng, masses):
    """Phase coefficients of a draw of chirp mass and mass ratio (leading three orders and the
    logarithmic terms at their sizes), a delay within 0.12 s and a constant phase."""
    mc, eta = rng.uniform(*masses), rng.uniform(0.16, 0.25)
    x, k = (math.pi * mc * 4.925490947641267e-6 * eta ** -0.6) ** (1 / 3), 3 / (128 * eta)
    p = [1.0, 3715 / 756 + 55 / 9 * eta, -16 * math.pi + rng.uniform(-20, 20), 30 + 54 * eta, 160 - 65 * eta, 11000.0, -109.0, 700.0]
    e = [-5, -3, -2, -1, 0, 1, 1, 2]
    a = [k * v * x ** n for v, n in zip(p, e)]
    fisco = 1 / (6 ** 1.5 * math.pi * mc * 4.925490947641267e-6 * eta ** -0.6)
    return a + [rng.uniform(-0.12, 0.12), rng.uniform(-20, 20)], fisco


@pytest.mark.parametrize("f0", [20.0, 5.0, 1.0, 0.1, 0.01])
def test_phases_against_fp64(fx, f0):
    """Against the exact sums of the tabulated values, over every octave: the root mean square rounding no
    larger than that of FP64's fused multiply-adds; everywhere within the 12 units of 2^(E - 59) that nine
    coefficients' (1/2 each), table entries' (1/2 of the term's share of 2^E), dropped products' (1/4) and the
    final rounding allow, and without a common shift (mean within half a unit; each point's coefficients shift
    it by some 0.5 at random)."""
    rng = random.Random(2)
    N, f1 = 4097, 2048.0
    df = (f1 - f0) / (N - 1)
    lines, js, pts = [], [], []
    for _ in range(24):
        a, _ = point(rng, (1.1, 1.5))
        j = sorted(min(N - 1, int((f0 * (f1 / f0) ** rng.random() - f0) / df)) for _ in range(80))
        lines.append(f"p {N} {f0!r} {df!r} 1.1 0.06 " + " ".join(repr(v) for v in a) + f" {len(j)} " + " ".join(map(str, j)))
        js += j
        pts += [a] * len(j)
    fp64, split, units = {}, {}, []
    for j, a, o in zip(js, pts, fx(lines)):
        t = o.split()
        B = [mp.mpf(float.fromhex(v)) for v in t[3:]]
        f = B[8]
        want = sum(mp.mpf(u) * v for u, v in zip(a[:8], B)) + mp.mpf(a[9]) + 2 * mp.pi * f * mp.mpf(a[8])
        s = mp.mpf(int(t[0])) / mp.mpf(2) ** 64 * 2 * mp.pi

        def err(x):
            d = (x - want) / (2 * mp.pi)
            return float((d - mp.nint(d)) * 2 * mp.pi)
        octave = int(math.log2(float(f) / f0))
        fp64.setdefault(octave, []).append(err(mp.mpf(float.fromhex(t[1]))))
        split.setdefault(octave, []).append(err(s))
        units.append(err(s) / (2 * math.pi) / 2.0 ** (int(t[2]) - 59))
    rms = lambda v: math.sqrt(sum(x * x for x in v) / len(v))
    for o in fp64:
        assert rms(split[o]) <= rms(fp64[o]), (o, rms(split[o]), rms(fp64[o]))
    assert max(map(abs, units)) <= 12 and abs(sum(units) / len(units)) <= 0.5


@pytest.mark.parametrize("f1,N,masses,points", [(512.0, 512, (10.0, 40.0), 150), (1024.0, 4017, (10.0, 40.0), 60),
                                                (2048.0, 16225, (10.0, 40.0), 40), (2048.0, 8113, (1.1, 1.5), 40)])
def test_sums_against_fp64(fx, f1, N, masses, points):
    """Sums over the bins below f_ISCO from 20 Hz of weights that fall as f^(-7/6) over the noise: the
    root mean square error over draws, relative to the weights' norm, within 5% of the FP64 loop's."""
    rng = random.Random(4)
    df = (f1 - 20.0) / (N - 1)
    w = []
    for j in range(N):
        f = 20.0 + j * df
        s = f ** (-7 / 6) / math.sqrt((f / 30.0) ** -4 + 2.0 + 2.0 * (f / 200.0) ** 2)
        w += [32.0 * s * rng.gauss(0, 1), 32.0 * s * rng.gauss(0, 1)]
    lines = []
    while len(lines) < points:
        a, fisco = point(rng, masses)
        n = min(N, int((fisco - 20.0) / df) + 1)
        if n >= 32:
            lines.append(f"z {N} 20.0 {df!r} {masses[0]} 0.06 " + " ".join(repr(v) for v in a) + f" {n} " + " ".join(map(repr, w[:2 * n])))
    e = [list(map(float, o.split())) for o in fx(lines)]
    fp64, split = (math.sqrt(sum(v[k] ** 2 for v in e) / len(e)) for k in (0, 1))
    assert split <= 1.05 * fp64, (split, fp64)


@pytest.mark.parametrize("f0", [5e-324, 1e-310, 1e-200, 1e-60])
def test_blocks_of_the_smallest_frequencies(fx, f0):
    """Grids that start where the basis functions overflow are accepted too: the rule ends, with blocks
    that ascend from bin 0 and exponents of a double."""
    out = list(map(int, fx([f"b 300 {f0!r} 10.0 1.1 0.06 0 1 300"])[0].split()))
    nb = out[0]
    bins, e = [out[1 + 10 * b] for b in range(nb)], [out[2 + 10 * b:11 + 10 * b] for b in range(nb)]
    assert 1 <= nb <= 6 and bins[0] == 0 and all(a < b < 300 for a, b in zip(bins, bins[1:]))
    assert all(abs(k) <= 1074 for v in e for k in v)


@pytest.mark.parametrize("N,f0,df,mc,tau,first,blocks", [
    (9000, 20.0, 0.25, 10.0, 0.06, [], 1), (9000, 20.0, 0.25, 1.1, 0.06, [0], 1), (9000, 3.0, 0.25, 1.1, 0.06, [64, 256], 2),
    (70000, 20.0, 1 / 32, 1.1, 0.0, [192, 256, 512, 1024, 2048], 2), (1, 20.0, 1.0, 1.1, 0.06, [], 1), (2, 0.01, 100.0, 1.1, 0.06, [], 2),
    (5000, 0.01, 0.5, 1.1, 0.06, [], 5), (300, 1e-4, 10.0, 1.1, 0.06, [], 3), (3000000, 1e-6, 1e-4, 1.1, 0.06, [], 6),
    (40, 5.0, 1e-3, 1.1, 0.06, [], 1), (3000, 0.01, 1.0, 1e-4, 0.0, [], 5)])
def test_blocks_cover_the_grid(fx, N, f0, df, mc, tau, first, blocks):
    """Blocks start at bin 0 and ascend; every bin's and node's basis values stay below their block's
    power of two; a point's rows change block at the first bin, or the first tile, that starts in the next."""
    row, start = [], N
    for l, b in enumerate(first):
        row.append(start)
        start += ((N - b) >> (6 + l)) * 32
    rng = random.Random(1)
    counts = [0, 1, N] + [rng.randrange(N + 1) for _ in range(40)]
    out = list(map(int, fx([f"b {N} {f0!r} {df!r} {mc} {tau} {len(first)} " + " ".join(f"{a} {b}" for a, b in zip(first, row)) + " "
                            f"{len(counts)} " + " ".join(map(str, counts))])[0].split()))
    nb = out[0]
    bins, e = [out[1 + 10 * b] for b in range(nb)], [out[2 + 10 * b:11 + 10 * b] for b in range(nb)]
    assert bins[0] == 0 and all(a < b for a, b in zip(bins, bins[1:])) and bins[-1] < N and nb <= 6
    assert nb <= blocks

    def block(j):
        return max(b for b in range(nb) if bins[b] <= j)

    def fits(f, b):
        c, l = f ** (1 / 3), math.log(f)
        v = [1 / (f * c * c), 1 / f, 1 / (c * c), 1 / c, l, c, c * l, c * c, f]
        assert all(abs(x) <= 2.0 ** k for x, k in zip(v, e[b])), (f, b)
    for j in {0, N - 1} | set(bins) | {b - 1 for b in bins if b} | {rng.randrange(N) for _ in range(300)}:
        fits(f0 + j * df, block(j))
    for l, s0 in enumerate(first):
        n = 64 << l
        for s in range(s0, N - n + 1, n):
            for f in (f0 + (s - 0.5) * df, f0 + (s + n - 0.5) * df):
                if f > 8.0 * df:
                    fits(f, block(s))
    pos = 1 + 10 * nb
    for c in counts:
        rows, ends, pos = out[pos], [], pos + 1
        while not ends or ends[-1] != 0x7fffffff:
            ends.append(out[pos])
            pos += 1
        # the rows' first bins in order: bins, tiles of growing then shrinking length, bins
        at, j = [], 0
        if first and c > first[0]:
            at, j = list(range(first[0])), first[0]
            l, up = 0, True
            while l >= 0:
                n = 64 << l
                go = up and l + 1 < len(first) and c // n * n >= first[l + 1]
                to = first[l + 1] if go else c // n * n
                while j + n <= to:
                    at += [j] * 32
                    j += n
                up = go
                l += 1 if go else -1
        at += list(range(j, c))
        assert len(at) == rows
        for r in list(range(0, rows, 97)) + [x for x in ends + [x - 1 for x in ends] if 0 <= x < rows]:
            assert sum(r >= x for x in ends) == block(at[r]), (c, r)

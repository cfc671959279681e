"""The split arithmetic of the FP64 form's bin sums (fixed-point phases, table
cosine and sine, double-float products): the device header is plain C++ besides
its qualifiers, so it is compiled here for the host and checked against 60-digit
references."""
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
int main() {
    static fx_f4 tab[FX_SC];
    for (int i = 0; i < FX_SC; i++) {
        double c = rd(), s = rd();
        tab[i] = fx_f4{(float)c, (float)(c - (double)(float)c), (float)s, (float)(s - (double)(float)s)};
    }
    char op[16];
    while (scanf("%15s", op) == 1) {
        if (op[0] == 'c') {
            unsigned long long F;
            if (scanf("%llu", &F) != 1) return 1;
            fxe e = fx_cis(F, tab);
            printf("%a %a %a %a\n", (double)e.rh, (double)e.rl, (double)e.ih, (double)e.il);
        } else if (op[0] == 'p') {
            // 8 coefficients [rad], delay [s], constant [rad], 9 exponents, 8 basis values, frequency
            double a[9], c0, b[9];
            int eb[9], ex[9];
            uint64_t m[9], mc;
            int32_t bad = 0;
            for (int i = 0; i < 9; i++) a[i] = rd();
            c0 = rd();
            for (int i = 0; i < 9; i++) eb[i] = (int)rd();
            for (int i = 0; i < 9; i++) b[i] = rd();
            const int ec = fx_mantissa<true>(c0, &mc, &bad);
            int E = ec + 64 > 0 ? ec + 64 : 0;
            for (int i = 0; i < 9; i++) {
                ex[i] = (i < 8 ? fx_mantissa<true>(a[i], &m[i], &bad) : fx_mantissa<false>(a[i], &m[i], &bad)) + eb[i];
                E = ex[i] + 64 > E ? ex[i] + 64 : E;
            }
            int64_t hi = fx_scaled(mc, E - (ec + 64) + 7, c0), cr = 0;
            for (int i = 0; i < 9; i++)
                fx_mac(hi, cr, fx_split(fx_scaled(m[i], E - (ex[i] + 64) + 6, a[i])), fx_table(b[i], eb[i]));
            printf("%llu %d %d\n", (unsigned long long)fx_phase(hi, cr, E + 7), E, bad);
        } else if (op[0] == 's') {
            // levels, first bins, rows, bins to cover
            FxTiles T;
            FxPoint o;
            T.nlev = (int)rd();
            for (int i = 0; i < T.nlev; i++) { T.first[i] = (int)rd(); T.row[i] = (int)rd(); }
            fx_segments(T, true, (int)rd(), o);
            printf("%d %d", o.nseg, o.rows);
            for (int i = 0; i < o.nseg; i++) printf(" %d %d", o.seg[i].end, o.seg[i].off);
            printf("\n");
        } else {
            // n products w E summed
            float zh[2] = {0, 0}, zl[2] = {0, 0};
            const int n = (int)rd();
            for (int i = 0; i < n; i++) {
                float v[8];
                for (int k = 0; k < 4; k++) {
                    const double x = rd();
                    v[2 * k] = (float)x;
                    v[2 * k + 1] = (float)(x - (double)v[2 * k]);
                }
                fx_cmac(zh, zl, fx_f4{v[0], v[1], v[2], v[3]}, fxe{v[4], v[5], v[6], v[7]});
            }
            printf("%a %a %a %a\n", (double)zh[0], (double)zl[0], (double)zh[1], (double)zl[1]);
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
    d = tmp_path_factory.mktemp("fxmath")
    (d / "drv.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O1", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", "-I", CSRC, str(d / "drv.cpp"),
                    "-o", str(d / "drv"), "-lm"], check=True)
    mp.mp.dps = 60
    head = "\n".join("%r %r" % (float(mp.cospi(mp.mpf(i) / 512)), float(mp.sinpi(mp.mpf(i) / 512))) for i in range(512))

    def run(lines):
        r = subprocess.run([str(d / "drv")], input=head + "\n" + "\n".join(lines) + "\n", capture_output=True,
                           text=True, check=True)
        return r.stdout.splitlines()
    return run


def hexsum(t, i):
    return mp.mpf(float.fromhex(t[i])) + mp.mpf(float.fromhex(t[i + 1]))


def test_cis(fx):
    """Every table interval's ends and middle, both half turns, and random phases: the
    table's and the low parts' roundings (2^-49 each) and the Taylor tails stay below 4e-15."""
    rng = random.Random(3)
    F = [(i << 54) + o for i in range(1024) for o in (0, 1, (1 << 53) - 1, 1 << 53, (1 << 54) - 1)]
    F = [f % 2 ** 64 for f in F] + [rng.getrandbits(64) for _ in range(4000)]
    worst = mp.mpf(0)
    for f, o in zip(F, fx([f"c {f}" for f in F])):
        t = o.split()
        x = 2 * mp.mpf(f) / mp.mpf(2) ** 64
        worst = max(worst, abs(hexsum(t, 0) - mp.cospi(x)), abs(hexsum(t, 2) - mp.sinpi(x)))
    assert worst < 4e-15, worst


@pytest.mark.parametrize("f0,f1", [(20.0, 2048.0), (1e-3, 0.9), (0.2, 30.0), (1000.0, 1000.0)])
@pytest.mark.parametrize("size", [1e-30, 1.0, 3e4, 1e11])
def test_phase(fx, f0, f1, size):
    """The phase of random coefficients, largest term of about `size` radians, against the exact sum:
    within 16 units of 2^(E - 57) turns, 2^E the power of two above the largest term in turns."""
    rng = random.Random(5)

    def basis(f):
        c, l = f ** (1 / 3), math.log(f)
        return [c ** -5, 1 / f, c ** -2, 1 / c, l, c, c * l, c * c, f]

    top = [max(abs(basis(f)[m]) for f in (f0, f1, min(max(math.exp(-3), f0), f1))) for m in range(9)]
    eb = [math.frexp(x)[1] if x else -900 for x in top]
    lines, want = [], []
    for _ in range(200):
        a = [rng.choice([0.0, 1.0, 1.0, 1e-3]) * rng.uniform(-1, 1) * size / (x or 1.0) for x in top]
        a[8] /= 2 * math.pi
        c0 = rng.uniform(-math.pi, math.pi)
        f = rng.choice([f0, f1, rng.uniform(f0, f1)])
        b = basis(f)
        lines.append("p " + " ".join(repr(v) for v in a + [c0]) + " " + " ".join(map(str, eb)) + " " + " ".join(repr(v) for v in b))
        want.append((sum(mp.mpf(x) * mp.mpf(y) for x, y in zip(a[:8], b)) + mp.mpf(c0)) / (2 * mp.pi) + mp.mpf(a[8]) * mp.mpf(b[8]))
    for w, o in zip(want, fx(lines)):
        F, E, bad = map(int, o.split())
        d = mp.mpf(F) / mp.mpf(2) ** 64 - w
        d -= mp.nint(d)
        assert not bad and abs(d) <= 16 * mp.mpf(2) ** (E - 57), (F, E, d)


def test_phase_not_finite(fx):
    rest = " 0.5 " + " ".join(["1"] * 9) + " " + " ".join(["0.25"] * 9)
    for bad in ("nan", "inf", "-inf"):
        out = fx(["p " + " ".join([bad] + ["1.0"] * 8) + rest, "p " + " ".join(["1.0"] * 8 + [bad]) + rest])
        assert all(int(o.split()[2]) == 1 for o in out)


def test_products(fx):
    """Sums of n products against the exact ones: each product and addition within 2^-46 of its
    magnitude, the low accumulator's roundings (2^-24 of 2^-24 of the running sums) included."""
    rng = random.Random(7)
    for n in (1, 2, 33, 1000):
        v = [[rng.gauss(0, 1) * 2.0 ** rng.randint(-20, 0) for _ in range(2)] + [math.cos(p), math.sin(p)]
             for p in (rng.uniform(0, 7) for _ in range(n))]
        t = fx([f"z {n} " + " ".join(repr(x) for r in v for x in r)])[0].split()
        re = sum(mp.mpf(a) * mp.mpf(c) - mp.mpf(b) * mp.mpf(d) for a, b, c, d in v)
        im = sum(mp.mpf(a) * mp.mpf(d) + mp.mpf(b) * mp.mpf(c) for a, b, c, d in v)
        size = sum(abs(a) + abs(b) for a, b, _, _ in v)
        assert abs(hexsum(t, 0) - re) <= size * 2.0 ** -46 and abs(hexsum(t, 2) - im) <= size * 2.0 ** -46


@pytest.mark.parametrize("first", [[], [0], [128], [64, 256], [64, 128, 256, 1024], [0, 0, 0, 0, 0, 0, 0, 0, 0, 0],
                                   [192, 256, 256, 512, 1024, 2048, 4096, 8192, 16384, 32768]])
def test_segments(fx, first):
    """The segments of every bin count cover each bin once, in order, by whole tiles of a level past its first bin."""
    n = 70000 if len(first) == 10 else 9000
    row, start = [], n
    for l, f in enumerate(first):
        row.append(start)
        start += ((n - f) >> (6 + l)) * 32
    head = f"s {len(first)} " + " ".join(f"{a} {b}" for a, b in zip(first, row)) + " "
    rng = random.Random(1)
    counts = sorted({0, 1, 63, 64, 65, n} | {rng.randrange(n + 1) for _ in range(400)}
                    | {m + o for m in range(64, n, 64) for o in (0, 1) if rng.random() < 0.2})
    for c, o in zip(counts, fx([head + str(c) for c in counts])):
        v = list(map(int, o.split()))
        segs, pos, r = list(zip(v[2::2], v[3::2])), 0, 0
        assert v[0] == len(segs) <= 21
        for end, off in segs:
            lo = r + off
            if lo < n:              # bins
                assert lo == pos and lo + end - r <= n
                pos += end - r
            else:
                l = max(i for i in range(len(first)) if row[i] <= lo and (i + 1 == len(first) or lo < row[i + 1]))
                assert pos % (64 << l) == 0 and (lo - row[l]) == (pos - first[l]) // (64 << l) * 32 and pos >= first[l]
                assert (end - r) % 32 == 0
                pos += (end - r) // 32 * (64 << l)
            r = end
        assert pos == c and r == v[1]

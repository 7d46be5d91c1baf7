"""How the columns of a dense product are cut (no GPU needed): which shapes the tensor cores take and how much weight scratch a layer
needs may not depend on how fast a cut is."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KS = (16, 32, 64, 100, 128, 200, 256, 384, 600, 768, 1024, 2000)
MS = (1, 129, 9_000, 18_816, 18_817, 37_888, 131_072, 1_000_000)
SEGS = ((16, 0), (48, 48), (64, 0), (64, 64), (80, 0), (96, 0), (112, 0), (128, 0), (144, 0), (128, 128), (256, 0), (272, 0), (256, 256), (1024, 0),
        (1040, 0), (2048, 0), (4096, 0))
HEADS = ((1, 16), (1, 64), (1, 128), (1, 256), (2, 64), (2, 128), (4, 16), (4, 32), (8, 16), (4, 48))

PROGRAM = r"""
#include "common.cuh"
#include <cstdio>
int main() {
  int f32, k1, k2, n0, n1, hd; long long m;
  while (scanf("%d %lld %d %d %d %d %d", &f32, &m, &k1, &k2, &n0, &n1, &hd) == 7) {
    it_gemm_args a{};
    a.M = m; a.x_dtype = a.dt0 = a.dt1 = f32 ? IT_F32 : IT_BF16; a.X1 = &a; a.K1 = k1; a.X2 = k2 ? &a : nullptr; a.K2 = k2; a.n0 = n0; a.n1 = n1;
    it_tc_cols c{};
    const bool ok = it_tc_columns(a, hd ? hd : n0 + n1, hd > 0, &c);
    printf("%d %d %d %d %d\n", (int)ok, ok ? c.n_splits : 0, ok ? c.nbc : 0, ok ? c.NB : 0, ok ? c.stream : 0);
  }
}
"""


@pytest.fixture(scope="module")
def columns(tmp_path_factory):
    from paper_2307_00228_b200 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("columns")
    src, exe = d / "columns.cpp", d / "columns"
    src.write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-std=c++20", "-I", os.path.join(ROOT, "include"), "-I", build.CSRC, "-I", f"{cuda}/include", str(src), lib,
                           f"-Wl,-rpath,{os.path.dirname(lib)}", "-Wl,--allow-shlib-undefined", f"-L{cuda}/lib64", "-lcudart", f"-Wl,-rpath,{cuda}/lib64", "-o", str(exe)])

    def run(rows):
        text = subprocess.run([str(exe)], input="\n".join(" ".join(map(str, r)) for r in rows), text=True, capture_output=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in text.splitlines()]
    return run


def shapes():
    for k1 in KS:
        for k2 in (0, k1):
            for n0, n1 in SEGS:
                yield k1, k2, n0, n1, 0
        for heads, hd in HEADS:
            yield k1, 0, 0, heads * hd, hd


def narrow(k1, k2, n0, n1, hd):
    """fp32: as few splits of at most 64 columns as leave their weights (hi and lo, k-blocks of 32) resident; prepared columns, or None."""
    n = -(-n0 // 16) * 16 + -(-n1 // 16) * 16
    step = hd or 16
    if step % 16:
        return None
    kb = -(-k1 // 32) + -(-k2 // 32)
    budget = 227 * 1024 - 1024 - 320 - 1024 - 3 * 128 * 128 - 32 * 1024
    for s in range(1, 17):
        c = -(-(-(-n // s)) // step) * step
        if c <= 64 and 2 * kb * c * 128 <= budget and (not hd or c * s == n):
            return c * s
    return None


def test_fp32_products_are_taken_and_prepared_as_by_splits_of_64_columns(columns):
    """... for every number of rows: a layer keeps its arithmetic, and scratch that was enough stays enough."""
    rows = [(1, m, *s) for s in shapes() for m in MS]
    got = columns(rows)
    assert len(got) == len(rows)
    wide = 0
    for (_, m, *s), (ok, splits, nbc, nb, stream) in zip(rows, got):
        most = narrow(*s)
        assert ok == (most is not None), (m, s)
        if ok:
            n = sum(-(-x // 16) * 16 for x in s[2:4])
            assert nb <= most and n <= nb and nb == splits * nbc and nbc <= 128, (m, s, nb, most)
            assert not (s[4] and stream)
            wide += nbc > 64
    assert wide > 100


def test_short_fp32_products_keep_two_accumulators(columns):
    """One accumulator of 65 to 128 columns leaves nothing to hide a tile's epilogue behind: not for K of up to 64 (128 columns: up to 96)."""
    rows = [(1, m, k, 0, n, 0, 0) for k in (16, 32, 64, 96) for n in (96, 112, 128, 256) for m in MS if not (k == 96 and n == 96)]
    assert all(ok and nbc <= 64 for ok, _, nbc, _, _ in columns(rows))
    rows = [(1, m, k, 0, n, 0, 0) for k in (128, 192) for n in (96, 128) for m in MS[-3:] if not (k == 192 and n == 128)]
    assert all(ok and nbc == r[4] for r, (ok, _, nbc, _, _) in zip(rows, columns(rows)))

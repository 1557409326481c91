"""Host logic of the shared-operand tensor-core contraction, on CPU: the row
layouts (which products are rows of operand A and B, and the slot of every
item).  The C++ units are compiled with the host compiler into a small
driver; the checks are what the device code relies on: every item in one slot
of its own whose two rows hold exactly its bins, operand A within 64 rows, B
from a swizzle atom on within 256 rows, whole 16-row units."""
import itertools
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1705_06284_gb300", "csrc")

DRIVER = r'''
#include <cstdio>
#include "gram_rows.h"
#include "pair_cover.h"
int main() {
    char mode; int nb, n;
    if (scanf(" %c %d %d", &mode, &nb, &n) != 3) return 2;
    std::vector<std::array<int, 4>> it(n);
    std::vector<std::array<int, 3>> tr;
    for (auto &x : it) {
        if (scanf("%d %d %d %d", &x[0], &x[1], &x[2], &x[3]) != 4) return 2;
        if (x[3] < 0) tr.push_back({x[0], x[1], x[2]});
    }
    std::vector<fbs::GramRows> g(1);
    const bool ok = mode == 'S' ? fbs::gram_rows_shared(nb, it, g[0])
                  : mode == 'P' ? fbs::gram_rows_pairs(nb, tr, fbs::cover_triplet_pairs(nb, tr), g[0])
                                : fbs::gram_rows_wide(nb, tr, fbs::cover_triplet_pairs(nb, tr), g);
    printf("%d %zu\n", ok ? 1 : 0, ok ? g.size() : 0);
    if (ok) for (auto &r : g) {
        printf("%zu %d %d %zu\n", r.rows.size(), r.jb0, r.nbch, r.items.size());
        for (auto &x : r.rows) printf("%d %d\n", x[0], x[1]);
        for (auto &x : r.items) printf("%d %d %d\n", x[0], x[1], x[2]);
    }
    return 0;
}
'''


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("gram")
    src = d / "driver.cpp"
    src.write_text(DRIVER)
    exe = d / "driver"
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), os.path.join(CSRC, "gram_rows.cpp"),
                    os.path.join(CSRC, "pair_cover.cpp"), "-o", str(exe)], check=True, capture_output=True, text=True)
    return str(exe)


def _closing(nb, arity, width):
    """Ascending bin tuples whose edges (1 + width b) can close a polygon."""
    lo = [1 + width * b if width > 0 else (1 - width) ** b for b in range(nb)]
    hi = [1 + width * (b + 1) if width > 0 else (1 - width) ** (b + 1) for b in range(nb)]
    return [t for t in itertools.combinations_with_replacement(range(nb), arity)
            if lo[t[-1]] <= sum(hi[b] for b in t[:-1])]


def _layout(exe, mode, nb, items):
    text = "%s %d %d\n" % (mode, nb, len(items)) + "\n".join(" ".join(map(str, t + (-1,) * (4 - len(t)))) for t in items)
    r = subprocess.run([exe], input=text, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    v = iter(int(x) for x in r.stdout.split())
    ok, ngroups = next(v), next(v)
    groups = []
    for _ in range(ngroups):
        nrows, jb0, nbch, nitems = next(v), next(v), next(v), next(v)
        rows = [(next(v), next(v)) for _ in range(nrows)]
        groups.append((jb0, nbch, rows, [(next(v), next(v), next(v)) for _ in range(nitems)]))
    return bool(ok), groups


def _check(groups, items):
    seen = []
    for jb0, nbch, rows, slots in groups:
        assert jb0 % 4 == 0 and len(rows) % 16 == 0 and 1 <= nbch <= 32 and 8 * (jb0 + nbch) <= len(rows)
        assert slots == sorted(slots) and len({s[:2] for s in slots}) == len(slots)
        for a, b, i in slots:
            assert 0 <= a < 64 and 0 <= b < 8 * nbch
            bins = [x for x in rows[a] + rows[8 * jb0 + b] if x >= 0]
            assert sorted(bins) == list(items[i])
            seen.append(i)
    assert sorted(seen) == list(range(len(items)))


@pytest.mark.parametrize("nb,width", [(1, 2.0), (3, 2.0), (7, 1.5), (9, -0.6), (14, 1.0), (16, -0.35), (16, 1.5),
                                      (16, -0.2)])
def test_shared_rows_hold_every_item(driver, nb, width):
    """Triplets and quadruplets together; 16 bins (152 rows) need rows of
    operand A alone, or two tiles of B where those do not fit."""
    items = _closing(nb, 3, width) + _closing(nb, 4, width)
    ok, groups = _layout(driver, "S", nb, items)
    assert ok and len(groups) == 1
    _check(groups, items)


def test_shared_rows_refuse_what_does_not_fit(driver):
    nb = 24  # 300 pairs: past 256 rows
    assert not _layout(driver, "S", nb, _closing(nb, 3, 1.0) + _closing(nb, 4, 1.0))[0]


@pytest.mark.parametrize("nb,width", [(1, 2.0), (6, 1.3), (12, 1.3), (18, -0.3)])
def test_pair_rows_hold_every_triplet(driver, nb, width):
    items = _closing(nb, 3, width)
    ok, groups = _layout(driver, "P", nb, items)
    assert ok
    _check(groups, items)


@pytest.mark.parametrize("nb,width", [(5, 1.3), (24, 1.7), (29, 3.0), (33, 1.0), (48, 1.0), (64, -0.08)])
def test_wide_rows_hold_every_triplet(driver, nb, width):
    items = _closing(nb, 3, width)
    ok, groups = _layout(driver, "W", nb, items)
    assert ok
    _check(groups, items)
    assert not _layout(driver, "P", nb, items)[0] or nb <= 5


def test_wide_rows_refuse_more_than_64_bins(driver):
    assert not _layout(driver, "W", 70, _closing(70, 3, 1.0))[0]

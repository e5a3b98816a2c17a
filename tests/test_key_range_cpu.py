"""The allocator's selection on the host: the range arithmetic that the kernel includes (csrc/skim_key_range.h), driven by the
kernel's own loop, over keys of error tables with infinite, NaN and extreme entries.  The wanted key must stay inside the
range, the count of live keys must be the count inside it, and what is left must fit the list that is ranked directly."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LIST_CAP = 512

SOURCE = r"""
#include "skim_key_range.h"
#include <vector>
extern "C" int select_key(const uint64_t *keys, int64_t n, int64_t k, int64_t cap, uint64_t *lo, uint64_t *hi, int64_t *need, int64_t *live)
{
    SkimKeyRange r{~0ull, 0ull};
    for (int64_t i = 0; i < n; ++i) { r.lo = keys[i] < r.lo ? keys[i] : r.lo; r.hi = keys[i] > r.hi ? keys[i] : r.hi; }
    *need = k;
    *live = n;
    int splits = 0;
    while (*live > cap && r.lo < r.hi) {
        const int sh = r.shift();
        std::vector<int64_t> hist(1 << SkimKeyRange::PART_BITS, 0);
        for (int64_t i = 0; i < n; ++i)
            if (r.holds(keys[i])) {
                const unsigned p = r.part_of(keys[i], sh);
                if (p >= hist.size()) return -1;
                ++hist[p];
            }
        int64_t above = 0;
        int p = (int)hist.size() - 1;
        while (p >= 0 && above + hist[p] < *need) above += hist[p--];
        if (p < 0) return -2;
        *need -= above;
        *live = hist[p];
        r = r.part((unsigned)p, sh);
        if (++splits > 8) return -3;
    }
    *lo = r.lo;
    *hi = r.hi;
    return splits;
}
"""


@pytest.fixture(scope="module")
def select(tmp_path_factory):
    d = tmp_path_factory.mktemp("key_range")
    src, lib = d / "select.cpp", d / "select.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2412_04180_b200", "csrc"), "-o", str(lib), str(src)],
                   check=True)
    f = ctypes.CDLL(str(lib)).select_key
    f.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_int64, ctypes.c_int64] + [ctypes.c_void_p] * 4
    f.restype = ctypes.c_int
    return f


def _keys(err):
    """Order-preserving images of the running minimum of a row's gains, as the kernel forms them."""
    e = err.astype(np.float64)
    with np.errstate(invalid="ignore"):
        gain = e[:, :-1] - e[:, 1:]
    run = gain.copy()
    for t in range(1, run.shape[1]):
        run[:, t] = np.where(gain[:, t] < run[:, t - 1], gain[:, t], run[:, t - 1])
    run[run == 0.0] = 0.0
    u = run.view(np.uint64)
    return np.where(u >> np.uint64(63), ~u, u | np.uint64(1 << 63)).reshape(-1)


def _tables():
    rng = np.random.default_rng(3)
    n = 2000
    base = np.sort(rng.random((n, 4)), axis=1)[:, ::-1].astype(np.float32)
    forbidden = base.copy()
    forbidden[:, 0] = np.inf                       # width 1 ruled out for every row
    one_negative = forbidden.copy()
    one_negative[17] = [0.5, 0.501, 0.4, 0.3]      # and one row that a bit makes worse: the keys span nearly all of 64 bits
    some = base.copy()
    some[rng.random(n) < 0.4, 0] = np.inf
    some[rng.random(n) < 0.2, 3] = np.inf          # infinite losses as well
    nan = one_negative.copy()
    nan[::3, 1] = np.inf                           # inf - inf
    nan[5::7, 2] = np.nan
    return dict(base=base, forbidden=forbidden, one_negative=one_negative, some=some, nan=nan,
                huge=np.float32(3e38) * rng.choice([-1, 1], (n, 4)).astype(np.float32))


@pytest.mark.parametrize("name", list(_tables()))
def test_selection_stays_inside_its_list(select, name):
    keys = np.ascontiguousarray(_keys(_tables()[name]))
    _check(select, keys)


@pytest.mark.parametrize("nb", [2, 3, 4])
def test_optimal_walk(nb):
    """The dynamic programme's backward walk where choices carry no information (every way infinitely dear: all choices 0, or any
    other value a state can have): the state stays one that the rows before can have, and the walk ends at 0."""
    rng = np.random.default_rng(nb)
    for rows in (1, 2, 5, 40):
        for K in range(0, rows * (nb - 1) + 1, max(1, rows // 5)):
            for any_choice in (False, True):
                s = K
                for i in range(rows - 1, -1, -1):
                    assert 0 <= s <= min(K, (i + 1) * (nb - 1))          # the states whose choice the kernel writes
                    u = int(rng.integers(0, min(s, nb - 1) + 1)) if any_choice else 0
                    u = max(u, s - i * (nb - 1))
                    assert 0 <= u <= nb - 1
                    s -= u
                assert s == 0


@pytest.mark.parametrize("lo,hi", [(0, 2**64 - 1), (2**63 + 12345, 2**64 - 1), (2**64 - 4096, 2**64 - 1), (0, 4095), (7, 2**53 + 9)])
def test_selection_over_extreme_ranges(select, lo, hi):
    rng = np.random.default_rng(lo % 1000 + 1)
    keys = np.array([lo + int(x * (hi - lo)) for x in rng.random(3000)] + [lo, hi] * 400 + [hi - 1, hi - 2] * 300, dtype=np.uint64)
    _check(select, keys)


def _check(select, keys):
    n = keys.size
    order = np.sort(keys)[::-1]
    for k in (1, 2, n // 7, n // 3, n // 2, n - 600, n - 1, n):
        lo, hi, need, live = (ctypes.c_uint64(), ctypes.c_uint64(), ctypes.c_int64(), ctypes.c_int64())
        rc = select(keys.ctypes.data, n, k, LIST_CAP, *(ctypes.addressof(v) for v in (lo, hi, need, live)))
        assert rc >= 0, rc
        assert lo.value <= hi.value
        inside = (keys >= np.uint64(lo.value)) & (keys <= np.uint64(hi.value))
        assert int(inside.sum()) == live.value
        assert live.value <= LIST_CAP or lo.value == hi.value
        above = int((keys > np.uint64(hi.value)).sum())
        assert need.value == k - above and 1 <= need.value <= live.value
        assert lo.value <= int(order[k - 1]) <= hi.value

"""The one-launch sort of small sets (root cube, keys and sort by one cluster of
blocks) against the oracle's keys and stable order, bit for bit, at the edges
of its block and cluster sizes (1,024 or 2,048 positions a block, up
to 16 blocks) and just past its largest set, and against the general radix
passes (a named sort variant takes those)."""
import numpy as np
import pytest

import oracle
from synth import clustered_halos, plummer, uniform_cube

pytestmark = pytest.mark.gpu

from gpu_util import tb, to_np, torch  # noqa: E402

EDGES = [1, 2, 31, 33, 1023, 1024, 1025, 2049, 15361, 16384, 16385, 32768, 32769, 49153, 65535, 65536,
         65537]


def _positions(n, kind):
    if kind == "plummer":
        return plummer(n, 70 + n % 97)[0]
    rng = np.random.default_rng(n)
    if kind == "clumps":
        # two tight clumps and a far point: few distinct keys, in runs longer
        # than a tile of the run step
        pos = (rng.integers(0, 2, (n, 1)) * 0.25 + 1e-7 * rng.random((n, 3))).astype(np.float32)
        pos[0] = 1.0
        return pos
    # few distinct positions: long runs of identical keys beside short ones
    site = rng.random((max(1, n // 300), 3)).astype(np.float32)
    return np.ascontiguousarray(site[rng.integers(0, len(site), n)])


@pytest.mark.parametrize("kind", ["plummer", "clumps", "sites"])
@pytest.mark.parametrize("n", EDGES)
def test_keys_and_order_equal_the_oracle(n, kind):
    m = tb()
    pos = _positions(n, kind)
    keys, lo, side = oracle.keys(pos)
    okeys, operm = oracle.sort(keys)
    p = torch.from_numpy(pos).cuda()
    for kw in ({}, {"radix_bits": 8}):
        t = m.build(p, None, n_crit=16, **kw)
        assert t.sync() == 0
        assert np.array_equal(to_np(t.pkey), okeys), kw
        assert np.array_equal(to_np(t.perm), operm), kw
        assert t.side == side and list(t.lo) == list(lo)
    # the allocation-free entry point takes the same route
    if n <= m.NOALLOC_MAX_N:
        k = torch.empty(n, dtype=torch.uint64, device="cuda")
        q = torch.empty(n, dtype=torch.int32, device="cuda")
        st, root = m.keys_sorted_noalloc(p, k, q)
        assert st == 0 and root[3] == side
        assert np.array_equal(to_np(k), okeys) and np.array_equal(to_np(q), operm)


@pytest.mark.parametrize("hilbert", [False, True])
@pytest.mark.parametrize("n", [1500, 16_385, 32_768])
def test_long_runs_out_of_order_take_the_whole_key(n, hilbert):
    """Two cubes of width 2^-13, each within one depth-10 cell and of hundreds of
    distinct keys in random order: runs of more than 128 keys of equal upper 32
    bits that hold a descent, which the sort takes eight more passes for."""
    m = tb()
    rng = np.random.default_rng(n)
    pos = rng.integers(0, 2, (n, 1)) * 0.5 + 0.12515 + 2.0 ** -13 * rng.random((n, 3))
    pos[0], pos[1] = 0.0, 1.0
    pos = pos[rng.permutation(n)].astype(np.float32)
    keys = oracle.keys(pos, "hilbert" if hilbert else "morton")[0]
    assert len(np.unique(keys)) > n // 2
    k = keys[np.argsort(keys >> np.uint64(31), kind="stable")]
    same = (k[1:] >> np.uint64(31)) == (k[:-1] >> np.uint64(31))
    start = np.flatnonzero(np.r_[True, ~same])
    length = np.diff(np.r_[start, n])
    descents = np.add.reduceat(np.r_[0, (same & (k[1:] < k[:-1])).astype(int)], start)
    assert ((length > 128) & (descents > 0)).any()
    okeys, operm = oracle.sort(keys)
    t = m.build(torch.from_numpy(pos).cuda(), None, key_order=m.KEYS_HILBERT if hilbert else m.KEYS_MORTON)
    assert t.sync() == 0
    assert np.array_equal(to_np(t.pkey), okeys)
    assert np.array_equal(to_np(t.perm), operm)


@pytest.mark.parametrize("n", [1, 1500, 16_385, 32_768])
def test_options_equal_the_general_passes(n):
    """Hilbert keys, the power-of-two root, masses and positions that are not
    16-byte aligned: every array of the tree is the same either way."""
    m = tb()
    pos, _ = clustered_halos(n + 1, 5, n_halo=20) if n > 1 else uniform_cube(2, 5)
    p = torch.from_numpy(pos).cuda()[1:]
    w = torch.rand(n + 1, device="cuda")[1:]
    for kw in (dict(key_order=m.KEYS_HILBERT), dict(root_pow2=True), dict(reorder=True)):
        a = m.moments(m.build(p, w, n_crit=10, **kw), p, w)
        b = m.moments(m.build(p, w, n_crit=10, radix_bits=8, **kw), p, w)
        assert a.sync() == 0 and b.sync() == 0 and a.n_cells == b.n_cells
        for k in ("pkey", "perm", "ckey", "level", "parent", "child_first", "child_end", "pfirst",
                  "pend", "leaf_cell", "mass", "com", "com_lo", "quad", "aabb"):
            assert np.array_equal(to_np(getattr(a, k)), to_np(getattr(b, k))), (kw, k)


def test_bad_coordinate_is_reported():
    m = tb()
    pos = uniform_cube(5000, 9)[0]
    pos[4321, 1] = np.inf
    with pytest.raises(m.TbError) as e:
        m.build(torch.from_numpy(pos).cuda(), None)
    assert e.value.name == "TB_ENONFINITE"

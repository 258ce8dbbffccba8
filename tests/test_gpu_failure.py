"""Failure paths of the build, made without faulting the GPU.

- A radix-pass look-back wait that runs out: the wait limit is lowered so
  that a look-back which finds a predecessor tile not yet published gives up
  at once; the build reports TB_ETIMEOUT, every access stays in bounds, and
  the next build of the same tree with the default limit is exact.
- A wait of the moments' upward pass that runs out, in the same way.
- A device allocation that fails: the library's TB_FAULT_ALLOC=k hook makes
  its k-th cudaMalloc fail in a child process; the build reports TB_ENOMEM
  and releasing the half-made tree succeeds.
- A kernel of the allocation-free sort that cannot be loaded: TB_FAULT_LOAD=k
  makes the first k loads fail in a child process; each call that meets one
  reports TB_ENOMEM, and the next call tries again.
- A device that takes no cooperative launch: TB_FAULT_COOPERATIVE=1 in a child
  process; the same results come from one launch per level or phase.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from synth import uniform_cube

pytestmark = pytest.mark.gpu

from gpu_util import assert_structure_equal, tb, torch  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("gen", ["uniform", "clumps"])
def test_lookback_wait_runs_out_then_next_build_is_exact(gen):
    """(Clumps: runs of some thousand keys with equal upper bits, which are left
    alone when the passes before did not order them.)"""
    m = tb()
    # 2^21 particles: 512 tiles of 4096 keys in each of the five passes, with
    # hundreds of tiles in flight at once
    pos, mass = uniform_cube(1 << 21, 23)
    if gen == "clumps":
        rng = np.random.default_rng(24)
        pos = (rng.random((512, 3))[rng.integers(0, 512, len(pos))] + 5e-5 * (pos - 0.5)).astype(np.float32)
    p = torch.from_numpy(pos).cuda()
    w = torch.from_numpy(mass).cuda()
    t = m.Tree()
    cfg = (8, 512, 8)
    assert m.set_wait_limit(0) == 0
    m.set_wait_limit(1)
    try:
        with pytest.raises(m.TbError) as ei:
            m.build(p, w, n_crit=16, tree=t, sort_cfg=cfg)
            torch.cuda.synchronize()
            st = t.sync()
            if st != 0:
                raise m.TbError(st, "status")
        assert ei.value.name == "TB_ETIMEOUT"
    finally:
        m.set_wait_limit(0)
    assert m.set_wait_limit(-1) == 1          # TB_EINVAL
    m.build(p, w, n_crit=16, tree=t, sort_cfg=cfg)
    torch.cuda.synchronize()
    assert t.sync() == 0
    assert_structure_equal(t, oracle.build_tree(pos, 16))


@pytest.mark.parametrize("n,mode", [(20_000, 0), (400_000, 0), (400_000, 2)])
def test_moment_waits_run_out_then_next_build_is_exact(n, mode):
    """The moments under a limit of one poll: whichever of their waits give up
    (for staged copies, which are then waited for before the block leaves, or
    for other blocks), the call ends, reports TB_ETIMEOUT if any did, and the
    next build and moments are exact."""
    m = tb()
    pos, mass = uniform_cube(n, 29)
    p, w = torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda()
    t = m.moments(m.build(p, w, mom_mode=mode), p, w)
    assert t.sync() == 0
    keys = ("mass", "com", "com_lo", "quad", "aabb")
    want = {k: getattr(t, k).clone() for k in keys}
    ran_out = 0
    for _ in range(20):
        m.build(p, w, mom_mode=mode, tree=t)
        m.set_wait_limit(1)
        try:
            m.moments(t, p, w)
            st = t.sync()
        finally:
            m.set_wait_limit(0)
        assert m.STATUS[st] in ("TB_OK", "TB_ETIMEOUT")
        ran_out += m.STATUS[st] == "TB_ETIMEOUT"
    # hundreds of blocks do not all reach a barrier within one poll of each other
    # (20,000 particles have one level of several blocks only)
    assert ran_out > 0 or n == 20_000
    m.moments(m.build(p, w, mom_mode=mode, tree=t), p, w)
    assert t.sync() == 0
    for k in keys:
        assert torch.equal(getattr(t, k), want[k]), k


_CHILD = r"""
import sys, torch
sys.path.insert(0, sys.argv[1])
import paper_2312_06102_gb300 as tb
p = torch.rand(200000, 3, device="cuda")
t = tb.Tree()
try:
    tb.build(p, None, n_crit=16, tree=t, sort_cfg=(8, 512, 8))
    print("RESULT TB_OK")
except tb.TbError as e:
    print("RESULT", e.name)
t.free()
torch.cuda.synchronize()
print("FREED")
"""


@pytest.mark.parametrize("k", [1, 4, 9])
def test_allocation_failure_reports_enomem(k):
    env = dict(os.environ, TB_FAULT_ALLOC=str(k))
    r = subprocess.run([sys.executable, "-c", _CHILD, ROOT], env=env, capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    assert "RESULT TB_ENOMEM" in r.stdout, r.stdout
    assert "FREED" in r.stdout


_LOADS = r"""
import sys, torch
sys.path.insert(0, sys.argv[1])
import paper_2312_06102_gb300 as tb
p = torch.rand(100000, 3, device="cuda")
k = torch.empty(100000, dtype=torch.uint64, device="cuda")
q = torch.empty(100000, dtype=torch.int32, device="cuda")
for n in (2, 2, 2, 100000):
    st, _ = tb.keys_sorted_noalloc(p[:n], k[:n], q[:n])
    print("RESULT", tb.STATUS[st])
t = tb.build(p, None)
print("EQUAL", torch.equal(q, t.perm), torch.equal(k.view(torch.int64), t.pkey.view(torch.int64)))
"""


def test_noalloc_loads_again_after_a_failed_load():
    """Small sets launch one kernel and larger ones others, and all are loaded by
    the first call that can: after two calls in which a load failed, whatever
    their size, the third loads them all."""
    env = dict(os.environ, TB_FAULT_LOAD="2")
    r = subprocess.run([sys.executable, "-c", _LOADS, ROOT], env=env, capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    assert [v.split()[1] for v in r.stdout.splitlines() if v.startswith("RESULT")] == \
        ["TB_ENOMEM", "TB_ENOMEM", "TB_OK", "TB_OK"], r.stdout
    assert "EQUAL True True" in r.stdout


_SEPARATE = r"""
import sys
import numpy as np, torch
sys.path.insert(0, sys.argv[1])
import paper_2312_06102_gb300 as tb
from synth import clustered_halos
pos, mass = clustered_halos(50_000, 27, n_halo=40)
# a leaf of 3,000 (summed by a block) and one of 300 (by a warp) among the queued
pos = np.concatenate([pos, np.full((3000, 3), pos[5], np.float32), np.full((300, 3), pos[7], np.float32)])
mass = np.concatenate([mass, np.full(3300, mass[3], np.float32)])
p, w = torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda()
off = torch.tensor([0, 20_000, 20_000, 53_300], device="cuda")
out = {}
for mode in (0, 1, 2):
    t = tb.moments(tb.build(p, w, n_crit=8, mom_mode=mode), p, w)
    tb.moments(t, p, w)
    n0 = tb.kernel_launches()
    tb.moments(t, p, w)
    out[f"launches{mode}"] = tb.kernel_launches() - n0
    b = tb.build_batched(p, w, off, mom_mode=mode, cell_capacity=30_000, one_launch=True)
    for name, v in (("single", t), ("batched", b)):
        assert v.sync() == 0
        for k in ("mass", "com", "com_lo", "quad", "aabb") + (("mass64", "com64", "quad64") if mode == 2 else ()):
            out[f"{name}{mode}{k}"] = getattr(v, k)[:v.n_cells].cpu().numpy()
np.savez(sys.argv[2], **out)
"""


def test_without_cooperative_launches(tmp_path):
    got = []
    for i, extra in enumerate(({}, {"TB_FAULT_COOPERATIVE": "1"})):
        path = str(tmp_path / f"{i}.npz")
        r = subprocess.run([sys.executable, "-c", _SEPARATE, ROOT, path], env=dict(os.environ, **extra),
                           capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-2000:]
        got.append(dict(np.load(path)))
    a, b = got
    for mode in (0, 1, 2):
        # leaves and one upward launch; leaves, queued leaves and 21 levels
        assert (a.pop(f"launches{mode}"), b.pop(f"launches{mode}")) == (2, 23)
    for k in a:
        if k.startswith("batched"):
            # (leaves of more than 2048 are summed in another order)
            assert a[k].shape == b[k].shape and np.isfinite(b[k]).all()
        else:
            assert np.array_equal(a[k], b[k]), k

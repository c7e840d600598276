"""Warp-specialised narrow launches of the FP64 state: producer warps draw the FP64
Box-Muller normals ahead of the stepping warp.  Bitwise the work queue, whose blocks draw their own."""
import numpy as np
import pytest

from paper_1104_2499_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def abp():
    from paper_1104_2499_gb300 import abp as A
    from paper_1104_2499_gb300 import build as B

    B.build()
    A.lib()
    return A


def run(A, w, pieces=(-1,), **kw):
    with A.Ensemble(w, state_fp64=True, particles_per_thread=1, **kw) as ens:
        ens.set_params()
        for n in pieces:
            ens.integrate(n)
        res, st, tiles = ens.results(), ens.state(), ens.tiles()
        torch.cuda.synchronize()
        return res, st, tiles


# one lane; ragged sets; two blocks on an SM; windows and snapshots that end inside a slot
@pytest.mark.parametrize("n_traj", [[1], [33, 0, 257, 5], [9000]])
def test_fp64_narrow_launch_is_bitwise_the_work_queue(abp, n_traj):
    sets = [W.params(D=0.1 + 0.1 * i) for i in range(len(n_traj))]
    w = W.Workload(name="fp64", sets=sets, n_traj=n_traj, n_steps=[203, 150, 64, 203][: len(sets)], dt=1e-3, seed=9,
                   v0_mode=1, hist_x_bins=8, hist_v_bins=4, v_lo=-2.0, v_hi=2.0, snapshot_every=50)
    ra, sa, ta = run(abp, w, pieces=(1, 70, -1), schedule=1, steps_per_launch=77)
    rb, sb, _ = run(abp, w, schedule=2, steps_per_launch=1000)
    assert ta["narrow"] == 32 or n_traj == [9000]
    for k in sa:
        assert torch.equal(sa[k], sb[k]), k
    for k in ra:
        assert torch.equal(ra[k], rb[k]), k


def test_fp64_packed_items_and_timeout(abp):
    n = 70
    w = W.Workload(name="items", sets=[W.params(D=0.01 * (i + 1)) for i in range(n)], n_traj=[1] * n, n_steps=[130] * n,
                   dt=1e-3, seed=4)
    ra, sa, ta = run(abp, w, schedule=1, steps_per_launch=1000)
    rb, sb, _ = run(abp, w, schedule=2, steps_per_launch=1000)
    assert ta["packed"] == 1
    for k in sa:
        assert torch.equal(sa[k], sb[k]), k
    with abp.Ensemble(w, state_fp64=True, particles_per_thread=1, schedule=1, steps_per_launch=1000) as ens:
        ens.set_params()
        abp.abp_set_wait_limit(ens.ctx, 200_000_000)
        abp.abp_test_hold_tile(ens.ctx, 0)
        ens.integrate()
        with pytest.raises(abp.AbpError) as ei:
            ens.synchronize()
        assert ei.value.status == abp.ABP_ETIMEOUT
        abp.abp_test_hold_tile(ens.ctx, -1)
        ens.reset()
        ens.integrate()
        ens.synchronize()
        np.testing.assert_array_equal(ens.state(host=True)["x"].numpy(), sb["x"].cpu().numpy())


def test_fp64_positions_far_beyond_the_table_range(abp):
    # a free particle driven to 10^15 periods a step: the force's cosine stays bounded, so the
    # velocity is the driven one (the potential adds at most 3e-3 a step)
    w = W.Workload(name="far", sets=[W.params(D=0.0, d=0.0, gamma0=0.0, F0=1e18)], n_traj=[40], n_steps=[100], dt=1e-3,
                   seed=2)
    st = run(abp, w, schedule=1, steps_per_launch=1000)[1]
    np.testing.assert_allclose(st["v"].cpu().numpy(), 1e18 * 1e-3 * 100, rtol=1e-13)
    assert bool(torch.isfinite(st["x"]).all())

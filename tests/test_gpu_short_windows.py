"""Windows of one step and of a few take other kernels than long ones (packed tiles with one
trajectory per thread, the FP64 state without producer warps): the same bits as one launch and as
the work queue, which never packs or narrows."""
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


def run(A, w, pieces, **kw):
    with A.Ensemble(w, particles_per_thread=1, **kw) as ens:
        ens.set_params()
        for n in pieces:
            ens.integrate(n)
        res, st, tiles = ens.results(), ens.state(), ens.tiles()
        torch.cuda.synchronize()
        return res, st, tiles


# packed tiles with pairs (an even load of the schedulers) and a narrow FP64 batch, both with the
# last tile partly filled; windows that start and end anywhere in a counter block and across a fold
@pytest.mark.parametrize("sets,traj,mode", [(3000, 20, "em"), (3000, 20, "heun"), (3000, 20, "xorshift"),
                                            (1, 1000, "fp64"), (70, 1, "fp64")])
def test_windows_of_any_length(abp, sets, traj, mode):
    N = 75
    r = np.random.default_rng(3)
    w = W.Workload(name="win", sets=[W.params(D=float(d)) for d in r.uniform(0.05, 0.5, sets)], n_traj=[traj] * sets,
                   n_steps=[N] * sets, dt=1e-3, seed=17, v0_mode=1, hist_x_bins=8, snapshot_every=25,
                   scheme=int(mode == "heun"), noise=int(mode == "xorshift"))
    kw = dict(state_fp64=mode == "fp64")
    ref = run(abp, w, (-1,), schedule=2, steps_per_launch=N, **kw)
    whole = run(abp, w, (-1,), schedule=1, steps_per_launch=N, **kw)
    assert whole[2]["packed"] == (0 if sets == 1 else -(-sets * traj // 240) if traj == 20 else 1)
    for pieces in ([1] * N, [1, 2, 1, 3, 5, 1, 7, 60, -1]):
        out = run(abp, w, pieces, schedule=1, steps_per_launch=N, **kw)
        for a, b, c in zip(out[:2], ref[:2], whole[:2]):
            for k in a:
                assert torch.equal(a[k], b[k]) and torch.equal(a[k], c[k]), k

"""Packed tiles beyond narrow launches: one trajectory per thread in blocks of 64 threads or of a
whole tile, or two per thread, chosen by the load of an SM's schedulers.  Every form gives every
trajectory the bits of the unpacked work queue."""
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


def small_sets(n_tiles, steps, **kw):
    # two sets to a tile (their sizes add up to at most 256; the last tile holds 1 + 2 trajectories)
    r = np.random.default_rng(n_tiles)
    M = []
    for _ in range(n_tiles - 1):
        a = int(r.integers(1, 255))
        M += [a, int(r.integers(257 - a - min(a, 3), 257 - a))]
    M += [1, 2]
    sets = [W.params(D=float(D), F0=float(f)) for D, f in zip(r.uniform(0.01, 1.0, len(M)), r.uniform(-0.5, 0.5, len(M)))]
    return W.Workload(name="small", sets=sets, n_traj=M, n_steps=[steps] * len(M), dt=1e-3, seed=11, v0_mode=1, **kw)


def run(A, w, **kw):
    with A.Ensemble(w, particles_per_thread=1, **kw) as ens:
        ens.run()
        res, st, tiles = ens.results(), ens.state(), ens.tiles()
        torch.cuda.synchronize()
        return res, st, tiles


# a few tiles past one per SM (64-thread blocks), an even load (pairs; whole tiles with xorshift
# noise), a larger odd and a larger even one
@pytest.mark.parametrize("tiles", [155, 260, 330, 700])
@pytest.mark.parametrize("mode", ["em", "heun", "xorshift", "fp64"])
def test_wide_packed_forms_match_the_work_queue(abp, tiles, mode):
    if mode == "fp64" and tiles > 260:
        pytest.skip("the FP64 state takes the same blocks")
    w = small_sets(tiles, 131, hist_x_bins=16, hist_v_bins=8, v_lo=-2.0, v_hi=2.0, snapshot_every=50,
                   scheme=int(mode == "heun"), noise=int(mode == "xorshift"))
    kw = dict(state_fp64=mode == "fp64")
    ra, sa, ta = run(abp, w, schedule=1, steps_per_launch=70, **kw)
    rb, sb, tb = run(abp, w, schedule=2, steps_per_launch=131, **kw)
    assert ta["packed"] > 152 and ta["narrow"] == 0 and tb["packed"] == 0
    for k in sa:
        assert torch.equal(sa[k], sb[k]), k
    for k in ra:
        assert torch.equal(ra[k], rb[k]), k


def test_paired_packed_tile_astride_matches_its_shards(abp):
    w = small_sets(260, 90)
    cut = sum(w.n_traj[:101])  # inside a tile, between its two sets
    whole = run(abp, w, schedule=1, traj_base=(1 << 32) - cut)[1]
    one = lambda a, b: W.Workload(name="part", sets=w.sets[a:b], n_traj=w.n_traj[a:b], n_steps=w.n_steps[a:b], dt=1e-3,
                                  seed=11, v0_mode=1)
    low = run(abp, one(0, 101), schedule=2, traj_base=(1 << 32) - cut)[1]
    high = run(abp, one(101, len(w.sets)), schedule=2, traj_base=1 << 32)[1]
    for k in whole:
        assert torch.equal(whole[k], torch.cat([low[k], high[k]])), k

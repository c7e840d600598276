"""Adjoint launches that cover several segments: level 1 with a segment per grid row, the reverse
sweep over the launch's segments, with the bits of one segment per launch; and the small batches'
form, in which level 1 leaves every step's state for the sweep."""
import numpy as np
import pytest

from paper_1104_2499_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

STATES = 2 * 16 * 366  # both buffers of one step: a 16-byte row per trajectory
SEGMENT = 2 * 16 * 6 * 2 * 2 * 128  # both hand-off buffers of one segment: 6 blocks of 128, K = 8 or 5


@pytest.fixture(scope="module")
def abp():
    from paper_1104_2499_gb300 import abp as A
    from paper_1104_2499_gb300 import build as B

    B.build()
    A.lib()
    return A


def grads(abp, K, window):
    w = W.Workload(name="launches", sets=[W.params(D=0.05), W.params(D=0.2, q=2.0), W.params(D=0.1, F0=0.3)],
                   n_traj=[300, 65, 1], n_steps=[203, 64, 7], dt=1e-3, seed=22, v0_mode=1, checkpoint_every=K)
    with abp.Ensemble(w, particles_per_thread=2) as ens:
        ens.run()
        n0 = abp.abp_kernel_launches(ens.ctx)
        g = ens.backward(host=True, window=window).numpy()
        return abp.abp_kernel_launches(ens.ctx) - n0, g, ens.traj_grad(host=True).numpy()


# 26 and 41 segments; the hand-off budget holds one, three or five segments, or every one
@pytest.mark.parametrize("K,slots", [(8, 1), (5, 2)])
@pytest.mark.parametrize("window", [0, 40])
def test_segments_per_launch(abp, monkeypatch, K, slots, window):
    out = {}
    monkeypatch.setenv("ABP_ADJ_STATE_BYTES", "0")
    for n in (1, 3, 5, None):
        monkeypatch.setenv("ABP_ADJ_HANDOFF_BYTES", "" if n is None else str(n * slots * SEGMENT))
        out[n] = grads(abp, K, window)
    monkeypatch.setenv("ABP_ADJ_HANDOFF_BYTES", "0")
    out[0] = grads(abp, K, window)
    monkeypatch.delenv("ABP_ADJ_HANDOFF_BYTES")
    states = {}
    for n in (1, 3, 5, None):  # a buffer is rounded up to 256 bytes
        monkeypatch.setenv("ABP_ADJ_STATE_BYTES", "" if n is None else str(n * (K * STATES + 512)))
        states[n] = grads(abp, K, window)
    n_seg = -(-203 // K)
    for n, (launches, g, t) in [*out.items(), *states.items()]:
        runs = 1 if n is None else -(-n_seg // max(n, 1))  # drawing again: one by one
        assert launches == 2 * runs + 2  # level 1 and reverse per run, the tile and the set sums
        np.testing.assert_array_equal(g, out[1][1])
        np.testing.assert_array_equal(t, out[1][2])

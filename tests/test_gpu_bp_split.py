"""How many CTAs of a cluster share the views: as many as the GPU holds at once,
where the ring decides that too (a near source needs windows of which one or
two CTAs fill an SM's shared memory), and the result against the oracle on
sampled slices (bars as in test_gpu_parity.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REL_RMSE = 1e-5
MAX_REL = 2e-4


@pytest.fixture(scope="module")
def fd():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1708_07515_gb300 as fd
    fd.load()
    return fd


@pytest.mark.parametrize("N,P,s,D,ratio,split", [
    (128, 128, 2, 2, 4.0, 4),    # three CTAs per SM
    (128, 128, 2, 2, 1.2, 1),    # one: 256 CTAs are more than fit as it is
    (96, 134, 1, 2, 1.4, 4),     # two
    (96, 134, 1, 2, 1.2, 1),
    (64, 90, 1, 2, 1.2, 4),      # one, 32 CTAs
    (100, 140, 0, 1, 4.0, 4),    # two waves of four rather than one of two
])
def test_split_counts_resident_ctas(fd, oracle_mod, N, P, s, D, ratio, split):
    R, Nu = ratio * N, N + (-N) % 4
    Q = np.random.default_rng(N + P).standard_normal((P, N, Nu)).astype(np.float32)
    zs = np.array([0, 15, N // 2, N - 1])
    with fd.Plan(R, N, Nu, N, P, s, D) as plan:
        form = fd.fdkod_get_forms(plan.handle)
        assert form["bp_split"] == split, form
        got = plan.backproject(torch.from_numpy(Q).cuda())[torch.from_numpy(zs).cuda()].cpu().numpy()
        assert plan.device_status() == 0
    want = oracle_mod.fdkod_slices(Q, R, N, s, D, zs)
    err = got.astype(np.float64) - want
    assert np.linalg.norm(err) <= REL_RMSE * np.linalg.norm(want)
    assert np.abs(err).max() <= MAX_REL * np.abs(want).max()

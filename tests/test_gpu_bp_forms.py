"""Oracle parity of the backprojection's forms that volumes beyond the small
ones take: 16 and 32 pairs of slices per thread without shared views, with
enough views for the ring to wrap many times, in all row-group sizes (16, 8, 4
and any drift: R = 4 N and 1.6 N), and the host-buffer reconstruction over
them.  The form is asserted, so that a change of the dispatch cannot move the
tests to another one.  Bars as in test_gpu_parity.py: rel-RMSE <= 1e-5, max
error <= 2e-4 of the largest value (float32 arithmetic on identical Q)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REL_RMSE = 1e-5
MAX_REL = 2e-4
_TYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module")
def fd():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1708_07515_gb300 as fd
    fd.load()
    return fd


def _cmp(got, want, what):
    err = got.astype(np.float64) - want
    rel = np.linalg.norm(err) / np.linalg.norm(want)
    mx = np.abs(err).max() / np.abs(want).max()
    assert rel <= REL_RMSE and mx <= MAX_REL, f"{what}: rel-RMSE {rel:.3e}, max-rel {mx:.3e}"


def _q(seed, P, Nv, Nu, dtype):
    Q = np.random.default_rng(seed).standard_normal((P, Nv, Nu)).astype(np.float32)
    for ax in (1, 2):
        Q = (Q + np.roll(Q, 1, ax) + np.roll(Q, -1, ax)).astype(np.float32)
    return torch.from_numpy(Q).to(dtype).cuda()


@pytest.mark.parametrize("ratio", [4.0, 1.6])
@pytest.mark.parametrize("N,P,s,D,qtype,slices", [
    (192, 67, 2, 1, "f32", 16),     # views 67: a short last chunk
    (192, 130, 2, 2, "f32", 16),
    (184, 64, 2, 1, "bf16", 16),
    (250, 65, 2, 1, "f32", 32),     # at 1.6 N the windows of 32 slices are too large: 16
    (245, 128, 2, 2, "f32", 32),
    (248, 61, 2, 1, "f16", 16),     # 16-bit windows: 32 for far sources and many tiles only
    (432, 26, 0, 1, "f16", 32),
])
def test_many_views_without_a_cluster(fd, oracle_mod, N, P, s, D, qtype, slices, ratio):
    R, Nu = ratio * N, N + (-N) % 8
    Qd = _q(N + P, P, N - 1, Nu, _TYPES[qtype])
    zs = np.array([0, 15, 16, 31, 32, N // 2, N - 33, N - 1])
    with fd.Plan(R, N, Nu, N - 1, P, s, D, qtype=qtype) as plan:
        form = fd.fdkod_get_forms(plan.handle)
        if ratio < 2.0:
            slices = 16
        assert form["bp_slices"] == slices and form["bp_split"] == 1, form
        assert P // D > 2 * form["bp_views"] * form["bp_slots"]
        got = plan.backproject(Qd)[torch.from_numpy(zs).cuda()].cpu().numpy()
        assert plan.device_status() == 0
    _cmp(got, oracle_mod.fdkod_slices(Qd.float().cpu().numpy(), R, N, s, D, zs), f"N={N} P={P} {qtype} R={ratio}N")


@pytest.mark.parametrize("N,P,s,D,slices", [(192, 48, 2, 1, 16), (250, 48, 2, 2, 32), (256, 24, 2, 1, 32)])
def test_host_reconstruction_equals_the_device_calls(fd, N, P, s, D, slices):
    """Groups of slice pairs on two streams give the whole launch's volume bit
    for bit (even detector height)."""
    proj = _q(N, P, N, N + (-N) % 4, torch.float32).cpu().pin_memory()
    with fd.Plan(4.0 * N, N, proj.shape[2], N, P, s, D) as plan:
        form = fd.fdkod_get_forms(plan.handle)
        assert form["bp_slices"] == slices and form["bp_split"] == 1, form
        want = plan.backproject(plan.filter(proj.cuda())).cpu()
        for _ in range(2):
            assert torch.equal(torch.from_numpy(fd.reconstruct(plan, proj)), want)

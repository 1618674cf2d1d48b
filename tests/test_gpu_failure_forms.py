"""Failure paths of every form of the staged backprojection.

The small plans of test_gpu_failures.py take the cluster form, whose CTAs
meet at barriers after a wait that ran out.  Here the same host-set hook (one
staging copy left out, 20 ms limit on the bounded waits; or every window
counted as too small) drives the forms that large volumes and slabs take:
their consumer warps return and the producer waits for its copies in flight.
The chosen form is asserted, so that a change of the dispatch cannot move the
test to another one.  After each, the status is read and cleared and the same
plan matches the oracle again (bars as in test_gpu_failures.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REL_RMSE = 1e-5
MAX_REL = 2e-4
WAIT_NS = 20_000_000  # 20 ms


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


@pytest.mark.parametrize("N,P,s,D,slab,slices", [
    (245, 24, 2, 1, None, 32),       # the whole volume, 32 pairs of slices per thread
    (192, 24, 2, 1, None, 16),       # 16 pairs
    (245, 24, 2, 2, (30, 192), 32),  # slabs: consecutive slices
    (192, 24, 2, 1, (64, 40), 16),
])
def test_forms_without_a_cluster_report_and_recover(fd, oracle_mod, N, P, s, D, slab, slices):
    R, Nu = 4.0 * N, N + (-N) % 4
    Q = np.random.default_rng(N + P).standard_normal((P, N, Nu)).astype(np.float32)
    for ax in (1, 2):
        Q = (Q + np.roll(Q, 1, ax) + np.roll(Q, -1, ax)).astype(np.float32)
    Qd = torch.from_numpy(Q).cuda()
    z0, nz = slab or (0, N)
    zs = np.unique([0, 15, 16, 31, 32, nz // 2, nz - 1])
    with fd.Plan(R, N, Nu, N, P, s, D) as plan:
        form = fd.fdkod_get_forms(plan.handle, nz if slab else 0)
        assert form["bp_slices"] == slices and form["bp_split"] == 1, form
        if slab:
            v0, nr = plan.slab_rows(z0, nz)
            rows = Qd[:, v0:v0 + nr].contiguous()
            work = torch.empty(max(1, plan.slab_workspace_elems(nr)), device="cuda")

        def run():
            return plan.backproject_slab(rows, v0, work, z0, nz) if slab else plan.backproject(Qd)

        fd.fdkod_set_test_fault(plan.handle, fd.FDKOD_TEST_SKIP_COPY, WAIT_NS)
        run()
        torch.cuda.synchronize()
        assert plan.device_status() == -5   # FDKOD_ERR_TIMEOUT
        assert plan.device_status() == 0    # read and cleared
        fd.fdkod_set_test_fault(plan.handle, fd.FDKOD_TEST_SMALL_WINDOW, WAIT_NS)
        assert float(run().abs().max()) == 0.0
        assert plan.device_status() == -6   # FDKOD_ERR_BOUNDS
        fd.fdkod_set_test_fault(plan.handle, fd.FDKOD_TEST_NONE, 0)
        got = run()[torch.from_numpy(zs).cuda()].cpu().numpy()
        assert plan.device_status() == 0
    _cmp(got, oracle_mod.fdkod_slices(Q, R, N, s, D, z0 + zs), f"after the failures, N={N} slab={slab}")


def test_the_cluster_form_is_the_one_the_small_plans_take(fd):
    """What test_gpu_failures.py and the smallest group tests cover."""
    for N, P, s, D, split in ((64, 64, 1, 1, 8), (64, 64, 1, 2, 4), (64, 64, 2, 4, 2)):
        with fd.Plan(4.0 * N, N, N, N, P, s, D) as plan:
            form = fd.fdkod_get_forms(plan.handle)
            assert form["bp_slices"] == 16 and form["bp_split"] == split, (N, P, s, D, form)


def test_forms_reject_bad_arguments(fd):
    with fd.Plan(256.0, 64, 64, 64, 8, 1, 2) as plan:
        for nz in (-1, 65):
            with pytest.raises(fd.FdkodError):
                fd.fdkod_get_forms(plan.handle, nz)
    with fd.Plan(256.0, 64, 63, 64, 8, 1, 1) as plan:   # rows TMA cannot describe
        assert not any(fd.fdkod_get_forms(plan.handle).values())

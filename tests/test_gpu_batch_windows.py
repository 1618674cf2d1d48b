"""A batch whose windows are too large for the persistent kernel's stages (a near
source) is refused as unsupported, leaves no error behind, and
BatchReconstructor falls back to the per-volume launches."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fd():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1708_07515_gb300 as fd
    fd.load()
    return fd


def test_large_windows_are_unsupported(fd):
    from paper_1708_07515_gb300.batch import BatchReconstructor, Instance
    N, P = 96, 48   # windows of 64 columns x about 138 rows, eight of them: 283 KB
    with fd.Plan(1.2 * N, N, N, N, P, 1, 2) as plan:
        vol = torch.empty(plan.vol_shape, device="cuda")
        with pytest.raises(fd.FdkodError) as e:
            fd.BatchBackprojection([plan], [None], [vol])
        assert e.value.status == -2   # FDKOD_ERR_UNSUPPORTED
        # the next call does not inherit an error
        Q = torch.randn(plan.q_shape, device="cuda")
        want = plan.backproject(Q)
        assert plan.device_status() == 0
    br = BatchReconstructor([Instance(1.2 * N, N, N, N, P, 1, 2)], persistent=True)
    try:
        assert br.batch is None
        br.Q[0].copy_(Q)
        assert torch.equal(br.plans[0].backproject(br.Q[0]), want)
    finally:
        br.close()


@pytest.mark.parametrize("N,ratio", [(64, 1.156), (144, 1.328)])
def test_the_largest_windows_that_fit_are_taken(fd, N, ratio):
    """48 x 150 and 64 x 113 windows: 230528 and 231552 bytes of the 232448 a
    block can have.  Per-volume launches to float32 rounding, as elsewhere."""
    P = 48
    Q = torch.randn((P, N, N), device="cuda", generator=torch.Generator(device="cuda").manual_seed(N))
    with fd.Plan(ratio * N, N, N, N, P, 1, 2) as plan:
        vol = torch.empty(plan.vol_shape, device="cuda")
        want = plan.backproject(Q)
        batch = fd.BatchBackprojection([plan], [None], [vol])
        batch.run()
        assert plan.device_status() == 0
        d = vol.double() - want.double()
        assert float(d.norm() / want.double().norm()) <= 1e-5
        batch.close()

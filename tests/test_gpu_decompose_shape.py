"""The staged decomposition's launch shape: the CTAs per SM that the choice of
ranges reckons with fit the SM (registers and shared memory, as the runtime
counts them), for squares of every number of column segments, both tap lengths
and all storage types; and the shape never changes the result (the generic
kernel's bits)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

_TYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module")
def fd():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1708_07515_gb300 as fd
    fd.load()
    return fd


@pytest.mark.parametrize("qtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("taps", ["triangle", "sinc"])
@pytest.mark.parametrize("N,s,P", [
    (16, 1, 24), (16, 0, 24), (40, 1, 48), (48, 0, 64), (64, 0, 96), (72, 0, 96),   # 1 to 7 segments
    (80, 0, 240), (84, 0, 96), (300, 2, 420),                                       # 8: two CTAs of four
    (96, 0, 128), (150, 0, 200), (165, 0, 200), (170, 0, 96), (176, 0, 96), (352, 1, 480),   # wider
    (64, 2, 6000),                                                                  # tables as large as the ring
])
def test_resident_ctas_fit_the_sm(fd, qtype, taps, N, s, P):
    Nu, Nv = (N + 7) // 8 * 8, min(N, 35)
    with fd.Plan(4.0 * N, N, Nu, Nv, P, s, 2, qtype=qtype, taps=taps) as plan:
        form = fd.fdkod_get_forms(plan.handle)
        assert 1 <= form["dec_warps"] and 1 <= form["dec_resident"] <= form["dec_occupancy"], (
            plan.info["T_stride"], form)
        if P > 1000:
            return
        Q = torch.randn(plan.q_shape, device="cuda").to(_TYPES[qtype])
        off = torch.empty(Q.numel() + 1, dtype=Q.dtype, device="cuda")[1:].view(Q.shape).copy_(Q)
        assert torch.equal(plan.decompose(Q), plan.decompose(off))
        assert plan.device_status() == 0


@pytest.mark.parametrize("N,s,segments,warps", [(84, 0, 8, 4), (96, 0, 9, 3), (142, 0, 13, 7), (170, 0, 16, 4)])
def test_segments_split_evenly(fd, N, s, segments, warps):
    """As few CTAs side by side as hold a square's column segments, or one more
    where fewer segments stay empty."""
    with fd.Plan(4.0 * N, N, (N + 7) // 8 * 8, 64, 24, s, 2) as plan:
        assert (plan.info["T_stride"] + 15) // 16 == segments, plan.info["T_stride"]
        assert fd.fdkod_get_forms(plan.handle)["dec_warps"] == warps


@pytest.mark.parametrize("qtype", ["f32", "bf16"])
@pytest.mark.parametrize("taps", ["triangle", "sinc"])
@pytest.mark.parametrize("N,Nu,P,s,D", [
    (72, 72, 96, 0, 8),     # staged
    (40, 40, 24, 0, 2),
    (49, 49, 72, 0, 6),     # generic: rows TMA cannot describe
    (33, 33, 32, 0, 16),    # two decimated views
])
def test_few_ctas_take_every_range(fd, qtype, taps, N, Nu, P, s, D):
    """Grids far smaller than the GPU split into ranges of one decimated view
    (a CTA walks its views one after the other), with the same bits as one
    launch that reads from another address takes."""
    with fd.Plan(4.0 * N, N, Nu, N, P, s, D, qtype=qtype, taps=taps) as plan:
        form = fd.fdkod_get_forms(plan.handle)
        assert form["dec_ranges"] == P // D and (form["dec_warps"] > 0) == (Nu % 8 == 0), form
        Q = torch.randn(plan.q_shape, device="cuda").to(_TYPES[qtype])
        off = torch.empty(Q.numel() + 1, dtype=Q.dtype, device="cuda")[1:].view(Q.shape).copy_(Q)
        assert torch.equal(plan.decompose(Q), plan.decompose(off))
        assert plan.device_status() == 0

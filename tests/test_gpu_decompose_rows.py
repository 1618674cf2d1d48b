"""The staged decomposition (lane = detector row, 16 columns per warp) against
the generic kernel, bit for bit.

All forms add the same products in the same order, so on the same Q they must
agree exactly.  The generic kernel runs when Q or the output is not 16-byte
aligned or Q's rows are not whole 16-byte units, and is itself checked against
the FP64 oracle here.  Shapes: squares whose shifted
rows end on and beside a multiple of 16 columns, one to eight column segments,
squares wider than 128 columns (several CTAs side by side), detectors of 1,
31, 32, 33 and more rows, few and many views (ranges of decimated views), both
tap lengths, every storage type."""
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


def _past_aligned(shape, dtype):
    """A contiguous tensor one element past an aligned address."""
    n = int(np.prod(shape))
    return torch.empty(n + 1, dtype=dtype, device="cuda")[1:].view(shape)


def _forms(plan, Q):
    """Decomposed data of the same Q: staged, from a misaligned Q, to a misaligned output."""
    off = _past_aligned(Q.shape, Q.dtype).copy_(Q)
    a, b = plan.decompose(Q), plan.decompose(off)
    c = plan.decompose(Q, _past_aligned(plan.decomposed_shape, torch.float32))
    assert plan.device_status() == 0
    return a, b, c


@pytest.mark.parametrize("qtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("taps", ["triangle", "sinc"])
@pytest.mark.parametrize("N,Nu,Nv,P,s,D,r", [
    (16, 16, 1, 12, 0, 2, 4.0),      # one detector row
    (40, 40, 31, 36, 2, 3, 4.0),     # one column segment, several row groups per CTA
    (64, 64, 33, 60, 1, 2, 4.0),     # one row past a band
    (96, 104, 32, 48, 1, 4, 2.5),
    (128, 128, 40, 16, 0, 16, 4.0),  # wider than 128 columns; one decimated view
    (250, 256, 35, 40, 0, 4, 3.0),   # three CTAs side by side
    (200, 200, 64, 400, 1, 2, 4.0),  # ranges of decimated views
    (61, 64, 70, 900, 3, 2, 1.6),    # many views, ragged squares, a near source
    (125, 125, 45, 60, 1, 3, 2.5),   # odd detector
    (61, 63, 45, 60, 1, 3, 2.5),     # narrower
    (150, 149, 40, 48, 0, 2, 4.0),   # wider than 128 columns
])
def test_staged_equals_generic(fd, qtype, taps, N, Nu, Nv, P, s, D, r):
    Q = torch.from_numpy(np.random.default_rng(N + P).standard_normal((P, Nv, Nu)).astype(np.float32))
    Q = Q.to(_TYPES[qtype]).cuda()
    with fd.Plan(r * N, N, Nu, Nv, P, s, D, qtype=qtype, taps=taps) as plan:
        a, b, c = _forms(plan, Q)
        assert torch.equal(a, c), (plan.info["T_stride"], float((a - c).abs().max()))
        assert torch.equal(b, c), (plan.info["T_stride"], float((b - c).abs().max()))


def test_generic_against_the_oracle(fd, oracle_mod):
    N, P, s, D = 40, 36, 1, 3
    Q = np.random.default_rng(5).standard_normal((P, 31, 40)).astype(np.float32)
    with fd.Plan(4.0 * N, N, 40, 31, P, s, D) as plan:
        c = _forms(plan, torch.from_numpy(Q).cuda())[2]
        got, T = c.cpu().numpy(), plan.bounds()["T"]
    for q in range(4):
        want = oracle_mod.shift_decimate(Q, 4.0 * N, N, s, D, q)
        assert np.abs(got[q, :, :, :T[q]] - want).max() <= 1e-6 * np.abs(Q).max()

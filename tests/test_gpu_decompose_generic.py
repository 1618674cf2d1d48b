"""The generic decomposition (rows that TMA cannot describe, or misaligned
buffers) against the FP64 oracle: odd detector widths, every storage type, both
tap lengths, row counts that leave one to three rows of a thread's four, one
and several ranges of decimated views, near and far sources.

Tolerance: a float32 sum of n = 2 H D products h x, |h| summing to at most 1.3
over the taps (1 for the triangle), of samples interpolated in float32
(three roundings): |error| <= 1.3 (n + 3) 2^-24 max|Q|, below 1e-5 max|Q| for
the D <= 8 here."""
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
@pytest.mark.parametrize("N,Nu,Nv,P,s,D,r,ranges", [
    (40, 41, 1, 24, 1, 3, 4.0, 8),       # one detector row, ranges of one view
    (61, 63, 45, 60, 1, 3, 2.5, None),   # one row past a thread's four
    (125, 125, 38, 60, 2, 2, 2.5, None), # two
    (67, 65, 35, 64, 0, 8, 1.6, 8),      # three; a near source, columns past the detector
    (150, 149, 40, 48, 0, 2, 4.0, None), # wide squares
    (333, 333, 333, 8, 3, 2, 4.0, 1),    # enough CTAs for a single range
])
def test_generic_kernel_against_the_oracle(fd, oracle_mod, qtype, taps, N, Nu, Nv, P, s, D, r, ranges):
    Q = torch.from_numpy(np.random.default_rng(N + D).standard_normal((P, Nv, Nu)).astype(np.float32))
    Q = Q.to(_TYPES[qtype]).cuda()
    Qr = Q.float().cpu().numpy()
    with fd.Plan(r * N, N, Nu, Nv, P, s, D, qtype=qtype, taps=taps) as plan:
        form = fd.fdkod_get_forms(plan.handle)
        assert form["dec_warps"] == 0 and (ranges is None or form["dec_ranges"] == ranges), form
        assert ranges is not None or form["dec_ranges"] > 1, form
        got = plan.decompose(Q).cpu().numpy()
        assert plan.device_status() == 0
        T, h = plan.bounds()["T"], plan.taps
    n = len(T)
    for q in sorted({0, n // 3, n - 1}):
        want = oracle_mod.shift_decimate(Qr, r * N, N, s, D, q, taps=h)
        assert want.shape == (P // D, Nv, T[q])
        assert np.abs(got[q, :, :, :T[q]] - want).max() <= 1e-5 * np.abs(Qr).max()
        assert not got[q, :, :, T[q]:].any()

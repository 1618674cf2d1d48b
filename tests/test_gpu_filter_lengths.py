"""The filter at every transform length: detector widths at both ends of each
power of two, with an odd number of rows and a band of rows, against the FP64
oracle.  Bar as in test_gpu_parity.py: per row, 2 log2(L) 2^-24 times the norm
of the row pair that shares its complex transform (FFT round-off)."""
import numpy as np
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


@pytest.mark.parametrize("Nu", [3, 8, 32, 33, 64, 65, 127, 128, 129, 256, 257, 511, 513, 1024, 1025, 2047, 2049])
def test_transform_lengths(fd, oracle_mod, Nu):
    P, Nv, R = 3, 7, 5000.0
    proj = np.random.default_rng(Nu).uniform(0.0, 1.0, (P, Nv, Nu)).astype(np.float32)
    want = oracle_mod.filter(proj, R)
    a = np.arange(Nu) - (Nu - 1) / 2
    b = np.arange(Nv) - (Nv - 1) / 2
    q = proj.astype(np.float64) * (R / np.sqrt(R * R + a[None, :] ** 2 + b[:, None] ** 2))[None]

    def check(got, want, q):
        rn = np.linalg.norm(q, axis=-1).reshape(-1)
        pair = np.repeat(np.sqrt(np.add.reduceat(rn ** 2, np.arange(0, rn.size, 2))), 2)[:rn.size]
        err = np.abs(got.astype(np.float64) - want).max(axis=-1).reshape(-1)
        assert np.all(err <= 2 * np.log2(L) * 2.0 ** -24 * pair)

    with fd.Plan(R, 8, Nu, Nv, P, 0, 1) as plan:
        L = plan.info["fft_length"]
        assert L >= 2 * Nu
        check(plan.filter(torch.from_numpy(proj).cuda()).cpu().numpy(), want, q)
        rows = torch.from_numpy(np.ascontiguousarray(proj[:, 2:5])).cuda()
        check(plan.filter_rows(rows, 2).cpu().numpy(), want[:, 2:5], q[:, 2:5])
        assert plan.device_status() == 0

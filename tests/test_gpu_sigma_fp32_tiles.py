"""fp32 Sigma's tiles: every split, whole and partial pieces, an output at any alignment."""
import pytest
import torch

from paper_2309_01885_gb300 import qe

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qe.load()


@pytest.mark.parametrize("p,n", [(4, 16), (60, 64), (62, 256), (68, 512), (132, 1024), (127, 2048), (1000, 300), (2050, 70)])
@pytest.mark.parametrize("offset", [0, 1, 2])
def test_output_pieces(p, n, offset):
    """Sigma at an offset of floats: the same bits as in an aligned buffer, symmetric, added to
    what is there; binary64 within n rounding errors of the terms' magnitudes; the floats
    around it stay."""
    g = torch.Generator(device="cuda").manual_seed(p + n)
    X = torch.randn(p, n, generator=g, device="cuda")
    S = qe.qe_build_sigma(X)
    F = X.double()
    assert torch.all((S.double() - F @ F.t()).abs() <= 2.0 ** -24 * (n + 1) * (F.abs() @ F.abs().t()))
    assert torch.equal(S, S.t())
    buf = torch.full((p * p + 8,), 7.0, device="cuda")
    out = buf[offset:offset + p * p].view(p, p)
    qe.qe_build_sigma(X, Sigma=out)
    assert torch.equal(out, S)
    qe.qe_build_sigma(X, Sigma=out, accumulate=True)
    assert torch.equal(out, S + S)
    assert torch.all(buf[:offset] == 7.0) and torch.all(buf[offset + p * p:] == 7.0)

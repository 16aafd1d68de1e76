"""Token counts beyond 31 bits."""
import pytest
import torch

from paper_2309_01885_gb300 import qe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", [qe.QE_TOKEN_MAJOR, qe.QE_FEATURE_MAJOR])
def test_sigma_beyond_2_31_tokens(layout):
    """The tokens past 2^31 count (34 GB of X: all zero but the first ones and those around the
    boundary), and none is looked for at a coordinate of more than 31 bits."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, p = 2 ** 31 + 100, 8
    if torch.cuda.mem_get_info()[0] < 3 * n * p:
        pytest.skip("not enough device memory")
    X = torch.zeros(n * p + 64 * p, dtype=torch.bfloat16, device="cuda")
    if layout == qe.QE_TOKEN_MAJOR:
        X = X[:n * p].view(n, p)
        tokens = X
    else:
        ld = n + -n % 8
        X = X[:ld * p].view(p, ld)[:, :n]
        tokens = X.t()
    g = torch.Generator(device="cuda").manual_seed(5)
    ends = [slice(0, 50), slice(2 ** 31 - 50, 2 ** 31), slice(2 ** 31, n)]
    for s in ends:
        tokens[s] = torch.randn(tokens[s].shape, generator=g, device="cuda").bfloat16()
    F = torch.cat([tokens[s] for s in ends]).double()
    S = qe.qe_build_sigma(X, layout)
    assert qe.qe_sync_status() == qe.QE_OK
    ref = F.t() @ F
    assert torch.all((S.double() - ref).abs() <= 1e-5 * torch.sqrt(torch.outer(ref.diagonal(), ref.diagonal())))

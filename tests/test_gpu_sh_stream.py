"""The SH forward with streamed coefficients (over 100 MB of them) against the same primitives in calls
small enough to be read as usual: the loads' cache policy changes no bit. Sizes either side of the line
and one that no block size divides."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degree,n", [(3, 520_833), (3, 520_834), (2, 925_927), (0, 8_333_335)])
def test_streamed_equals_parts(lib, degree, n):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    nb = (degree + 1) ** 2
    coeffs = torch.randn((nb, 3, n), generator=gen, device="cuda") * 0.3
    means = torch.rand((n, 3), generator=gen, device="cuda")
    whole = lib.sh_eval_fwd(coeffs, means, (0.0, 0.0, 3.0), degree)
    parts = [lib.sh_eval_fwd(coeffs[:, :, i:i + 200_000].contiguous(), means[i:i + 200_000].contiguous(), (0.0, 0.0, 3.0),
                             degree) for i in range(0, n, 200_000)]
    torch.testing.assert_close(whole, torch.cat(parts), rtol=0, atol=0)

"""Gaussian accumulator over more normals than one round of the chip takes (two per thread, two CTAs of 512 threads per
SM): at the edges of a round and over several, with mask, stride and cells, against the same normals in calls of one
partial round each (whose cells test_fastga_gpu.py holds to the oracle)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_2007_12065_gb300 as pl3d  # noqa: E402

LEVEL = 4
PART = 90_000


@pytest.fixture(scope="module")
def ctx():
    c = pl3d.pl3d_create(0)
    yield c
    pl3d.pl3d_destroy(c)


def _call(ctx, x, m, stride):
    n = m.numel()
    counts = torch.full((20 * 4 ** LEVEL,), -1, dtype=torch.int32, device="cuda")
    cells = torch.empty(n, dtype=torch.int32, device="cuda")
    pl3d.pl3d_fastga(ctx, x, m, n, LEVEL, stride, counts, cells)
    return counts, cells


@pytest.mark.parametrize("rounds,extra,stride", [(1, -1, 1), (1, 0, 1), (1, 1, 1), (2, 17, 1), (7, -3, 1), (7, 5, 3)])
@pytest.mark.parametrize("spread", [0.05, 10.0])
def test_rounds(ctx, rounds, extra, stride, spread):
    per_round = 2 * 2 * 512 * torch.cuda.get_device_properties(0).multi_processor_count
    n = rounds * per_round + extra
    g = torch.Generator(device="cuda")
    g.manual_seed(rounds * 100 + stride)
    x = torch.tensor([0.0, 0.0, 1.0], device="cuda") + spread * torch.randn(n, 3, device="cuda", generator=g)
    x = x / x.norm(dim=1, keepdim=True)
    x[torch.rand(n, device="cuda", generator=g) < 0.05] = float("nan")
    m = (torch.rand(n, device="cuda", generator=g) < 0.9).to(torch.uint8)
    counts, cells = _call(ctx, x, m, stride)
    part = PART // stride * stride
    want = torch.cat([_call(ctx, x[i:i + part], m[i:i + part], stride)[1] for i in range(0, n, part)])
    pl3d.pl3d_sync(ctx)
    cells = cells.cpu().numpy()
    np.testing.assert_array_equal(cells, want.cpu().numpy())
    np.testing.assert_array_equal(counts.cpu().numpy(), np.bincount(cells[cells >= 0], minlength=20 * 4 ** LEVEL))
    sampled = np.arange(n) % stride == 0
    finite = np.isfinite(x[:, 0].cpu().numpy())
    np.testing.assert_array_equal(cells >= 0, sampled & finite & (m.cpu().numpy() != 0))

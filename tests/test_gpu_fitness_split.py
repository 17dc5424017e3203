"""dpso_fitness where the number of warps per tour changes: lengths around its
rounds of 256 edges, and counts from one tour to more than are resident.  Sums
of whole numbers: exact."""
import pytest
import torch

from paper_1706_04399_gb300 import dpso

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 255, 256, 257, 512, 513, 1025, 2049])
@pytest.mark.parametrize("count", [1, 7, 609, 1217, 2433, 4865])
def test_fitness_split(n, count):
    g = torch.Generator(device="cuda").manual_seed(n * 10007 + count)
    C = torch.randint(0, 4_000_000, (n, n), dtype=torch.int32, device="cuda", generator=g)
    t = torch.argsort(torch.rand(count, n, device="cuda", generator=g), 1)
    edges = C[t, torch.roll(t, -1, 1)].to(torch.int64)
    # the last tour has one label out of range: its two edges count nothing
    at = (n * 7) // 9
    edges[-1, at] = 0
    edges[-1, at - 1] = 0
    t[-1, at] = n
    out = torch.full((count + 1,), -5, dtype=torch.int64, device="cuda")
    dpso.dpso_fitness(C, n, t.to(torch.int32).to(torch.uint16), count, out)
    torch.cuda.synchronize()
    assert torch.equal(out[:count], edges.sum(1))
    assert int(out[count]) == -5

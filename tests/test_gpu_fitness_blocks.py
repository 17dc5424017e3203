"""dpso_fitness at the counts and lengths at which whole tours share blocks of
eight or of two: 512 viewpoints, and 64 tours per SM (9728 on 152 SMs)."""
import pytest
import torch

from paper_1706_04399_gb300 import dpso

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [100, 257, 512, 513, 600])
@pytest.mark.parametrize("count", [4863, 9727, 9728, 9729, 20001])
def test_fitness_blocks(n, count):
    g = torch.Generator(device="cuda").manual_seed(n * 31 + count)
    C = torch.randint(0, 4_000_000, (n, n), dtype=torch.int32, device="cuda", generator=g)
    t = torch.argsort(torch.rand(count, n, device="cuda", generator=g), 1)
    want = C[t, torch.roll(t, -1, 1)].to(torch.int64).sum(1)
    out = torch.full((count + 1,), -5, dtype=torch.int64, device="cuda")
    dpso.dpso_fitness(C, n, t.to(torch.int32).to(torch.uint16), count, out)
    torch.cuda.synchronize()
    assert torch.equal(out[:count], want)
    assert int(out[count]) == -5

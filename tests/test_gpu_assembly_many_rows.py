"""Work items of the assembly kernel: a Gamma block with more than 2^31 rows (i, a), and rows on both
sides of the 128 elements that a warp holds at a time.  One fragment with coefficient 1, so the
output is the input to the bit."""
import pytest
import torch

from paper_2410_21888_gb300 import rimp2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("o,v,x", [(46341, 46342, 1), (3, 11, 127), (16, 1, 128), (5, 7, 129)])
def test_every_row(o, v, x):
    asm = rimp2.MBEAssembly([o], [v], [x], [(0,)], [1], [0], [-1], [-1])
    assert asm.gamma_elems == o * v * x
    g = torch.Generator(device="cuda").manual_seed(1)
    pool = torch.empty(o * v * x, dtype=torch.float64, device="cuda").uniform_(-1.0, 1.0, generator=g)
    out = torch.full_like(pool, float("nan"))
    asm.run(pool, None, None, out, None, None)
    torch.cuda.synchronize()
    assert torch.equal(out, pool)

"""A Gamma block with more than 2^31 rows (i, a): every row is gathered.  One fragment with
coefficient 1, so the output is the input to the bit."""
import pytest
import torch

from paper_2410_21888_gb300 import rimp2

pytestmark = pytest.mark.gpu


def test_rows_past_two_to_the_31():
    o, v = 46341, 46342
    assert o * v > 2 ** 31
    asm = rimp2.MBEAssembly([o], [v], [1], [(0,)], [1], [0], [-1], [-1])
    assert asm.gamma_elems == o * v
    g = torch.Generator(device="cuda").manual_seed(1)
    pool = torch.empty(o * v, dtype=torch.float64, device="cuda").uniform_(-1.0, 1.0, generator=g)
    out = torch.full_like(pool, float("nan"))
    asm.run(pool, None, None, out, None, None)
    torch.cuda.synchronize()
    assert torch.equal(out, pool)

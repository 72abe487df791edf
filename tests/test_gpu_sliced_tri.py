"""The line c <= r mod tri of the sliced product over all of its 64-bit range:
rows and tri around tile edges, tri past the rows, past 32 bits and at their
wrap, on one panel and with entries above the line left as they were."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,Nc", [(5, 7), (300, 300), (513, 130)])
@pytest.mark.parametrize("tri", [1, 3, 255, 256, 300, 512, 2 ** 31, 2 ** 32, 2 ** 32 + 5, 2 ** 33 + 256, 2 ** 63 - 1])
def test_line_of_every_size(M, Nc, tri):
    rng = np.random.default_rng(1)
    A = rng.integers(-1000, 1000, size=(M, 70))
    B = rng.integers(-1000, 1000, size=(Nc, 70))
    out = torch.full((M, Nc), 0.5, dtype=torch.float64, device="cuda")
    with D.Context(G.make_blocks(G.CONFIGS["tiny_2x2x2"])) as ctx:
        ctx.sliced_gemm(torch.from_numpy(A.astype(np.float64)).cuda(), torch.from_numpy(B.astype(np.float64)).cuda(),
                        out=out, tri=tri)
    c = np.arange(Nc)[None, :]
    want = np.where(c <= np.array([[int(x) % tri] for x in range(M)]), (A @ B.T).astype(np.float64), 0.5)
    assert np.array_equal(out.cpu().numpy(), want)

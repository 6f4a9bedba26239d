"""Calls with more right-hand sides than a grid has layers."""
import numpy as np
import pytest

from paper_2103_16841_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def op():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2103_16841_gb300 as stb
    ctx = stb.Context(0)
    return stb.Operator(ctx, stb.Mesh.from_spacetime(ctx, inputs.sphere_mesh(0, 1, 0.5, 0.2, seed=2)), "mixed")


@pytest.mark.parametrize("dtype", ["fp64", "fp32"])
@pytest.mark.parametrize("nrhs", [4 * 65535 - 1, 4 * 65535 + 1, 4 * 65535 + 6])
def test_products_of_more_vectors_than_a_grid_has_layers(op, dtype, nrhs):
    """The same numbers as in pieces (a vector's sum does not depend on the others)."""
    g = torch.Generator(device="cuda").manual_seed(nrhs)
    x = torch.randn((nrhs, op.n), dtype=torch.float64, device="cuda", generator=g)
    y = op.matvec(x, dtype=dtype)
    cut = 4 * 30000
    pieces = [op.matvec(x[i:i + cut].contiguous(), dtype=dtype) for i in range(0, nrhs, cut)]
    assert torch.equal(y, torch.cat(pieces))

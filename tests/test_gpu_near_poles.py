"""FP64 entries whose conic arcs end next to a pole of their integrand (an
asymptote of a hyperbolic conic), against the oracle."""
import os

import numpy as np
import pytest

import oracle
from paper_2103_16841_gb300 import inputs
from test_gpu_mixed_geometry import _cube

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_entries_with_arcs_next_to_a_pole():
    """Rows of a box whose arcs come within 1e-7 half-lengths of a pole and
    closer: 1e-9 of the largest entry (2^-53 in the position of a node there)."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2103_16841_gb300 as stb
    v, f = _cube(3)
    m = inputs.prism_mesh(v, f, 5, 2.5, 0.2, seed=1)
    ctx = stb.Context(0)
    op = stb.Operator(ctx, stb.Mesh.from_spacetime(ctx, m), "fp64")
    om = oracle.Mesh.from_spacetime(m)
    rows = np.array([150, 151, 270, 271, 285, 286], dtype=np.int32)
    ij = np.array([(r, c) for r, cols in zip(rows, om.pattern_rows(rows)) for c in cols])
    ref = om.entries(ij, nthreads=os.cpu_count())
    assert np.abs(op.entries(ij) - ref).max() <= 1e-9 * np.abs(ref).max()

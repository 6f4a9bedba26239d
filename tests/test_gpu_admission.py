"""The server's reservation covers what a request's operator and solve use."""
import pytest

from paper_2103_16841_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slabs", [1, 3])
@pytest.mark.parametrize("inner", ["tf32", "bf16"])
def test_reservation_covers_the_tensor_core_product(inner, slabs):
    """Columns of 3 and 9 panels share a 128-row tile, so chunk slots are padded
    to the widest band of up to 42 columns. Of two servers that differ in the
    inner arithmetic alone, the one with the tensor-core product reserves at least
    as much more as its resident operator (values, structure, workspace, tables
    and slots) holds more."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2103_16841_gb300 as stb
    ctx = stb.Context(0)
    m = inputs.sphere_mesh(1, slabs, 1.0, 0.2, seed=6)
    params = inputs.pulse_params(5, seed=7)
    got = {}
    for k in ("fp32", inner):
        srv = stb.Server(ctx, max_slots=1, precision="mixed", inner=k, tol=1e-6, cache_operators=True)
        t = srv.submit(m, params=params)
        r = srv.wait([t])[t]
        st = srv.stats()
        assert r["status"] == 0 and st["cached_operators"] == 1
        got[k] = (r["reserved_bytes"], st["cached_bytes"])
        srv.close()
    assert got[inner][0] - got["fp32"][0] >= got[inner][1] - got["fp32"][1]

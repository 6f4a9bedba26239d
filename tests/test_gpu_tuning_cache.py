"""Cache files of launch shapes from builds whose tuned kernel was another one."""
import json
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _tuned(cache):
    code = ("import json, sys; sys.path.insert(0, %r); import paper_2103_16841_gb300 as stb; "
            "from paper_2103_16841_gb300 import inputs; c = stb.Context(0); c.set_tuning(1, %r); "
            "m = inputs.sphere_mesh(1, 6, 2.0, 0.2, seed=9); "
            "o = stb.Operator(c, stb.Mesh.from_spacetime(c, m), 'mixed'); print(json.dumps(o.tuning()))" % (ROOT, str(cache)))
    out = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, out.stderr
    return json.loads(out.stdout.strip().splitlines()[-1])["tuned"]


def test_choices_for_another_kernel_are_not_taken(tmp_path):
    """The same class without the tuned stage's name, as files of builds before the
    stages have it, is timed again; this build's own line is taken."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    cache = tmp_path / "tune.txt"
    assert _tuned(cache) == "timed"
    assert _tuned(cache) == "cache"
    old = tmp_path / "old.txt"
    old.write_text(cache.read_text().replace("|apex|", "|"))
    assert _tuned(old) == "timed"

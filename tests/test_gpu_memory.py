"""Device memory a mesh holds, against what it held when charge sums kept no
workspaces, charge trees were built for direct sums too and the multipoles were
split into a buffer of their own (bytes after each call, recorded then)."""
import json
import os

import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "mesh_bytes.json")
MESHES = {
    "s6 p=6": (lambda: synth.globular(6), {"p": 6}),
    "s6 p=12": (lambda: synth.globular(6), {"p": 12}),
    "s5 FP64": (lambda: synth.globular(5), {"precision": 1}),
}


def held(pkg, name):
    """{call: device_bytes after it}"""
    make, opt = MESHES[name]
    m = make()
    out = {}
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, **opt) as g:
        out["create"] = g.info()["device_bytes"]
    return out


@pytest.mark.parametrize("name", sorted(MESHES))
def test_mesh_holds_no_more_than_before(name):
    """At most 2 % more (rows on whole lines where the tensor cores read them)."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1007_4591_gb300 as pkg
    pkg.load_library()
    with open(GOLDEN) as f:
        before = json.load(f)[name]
    for call, n in held(pkg, name).items():
        assert n <= before[call] * 1.02, (call, n / before[call])

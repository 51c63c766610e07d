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
    "s5 2,000 charges": (lambda: synth.globular(5), {}),
    "s5 4,000 charges": (lambda: synth.globular(5, n_charges=4000), {}),
    "s6 2,000 charges": (lambda: synth.globular(6), {}),
    "s6 4,000 charges": (lambda: synth.globular(6, n_charges=4000), {}),
    "s6 p=6": (lambda: synth.globular(6), {"p": 6}),
    "s6 p=12": (lambda: synth.globular(6), {"p": 12}),
    "s5 Galerkin": (lambda: synth.globular(5), {"galerkin": 1}),
    "s5 FP64": (lambda: synth.globular(5), {"precision": 1}),
}


def held(pkg, name):
    """{call: device_bytes after it}"""
    make, opt = MESHES[name]
    m = make()
    out = {}
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, **opt) as g:
        out["create"] = g.info()["device_bytes"]
        sigma, _ = g.solve()
        out["solve"] = g.info()["device_bytes"]
        g.energy(sigma, want_phi=True)
        out["energy"] = g.info()["device_bytes"]
        g.set_charges(m.charges)
        out["set_charges"] = g.info()["device_bytes"]
        g.energy_backward()
        out["backward"] = g.info()["device_bytes"]
    return out


@pytest.mark.parametrize("name", sorted(MESHES))
def test_mesh_holds_no_more_than_before(name):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1007_4591_gb300 as pkg
    pkg.load_library()
    with open(GOLDEN) as f:
        before = json.load(f)[name]
    for call, n in held(pkg, name).items():
        assert n <= before[call], (call, n / before[call])

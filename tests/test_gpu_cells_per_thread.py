"""One or four cells a thread in the default 2-D stencils, on either side of the sizes where the choice changes with the
layers: the fields of the TMA strips, bit for bit."""
import numpy as np
import pytest

from tests.adapters import FIELDS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,cpml,cpt", [(700, 714, 0, 1), (704, 714, 0, 4), (704, 714, 16, 4), (700, 714, 16, 1),
                                            (860, 870, 2, 1), (868, 870, 2, 4), (1044, 1050, 8, 1), (1048, 1052, 8, 4),
                                            (1048, 1052, 10, 4), (1220, 1224, 5, 1), (1228, 1224, 5, 4)])
def test_default_cells_per_thread(nx, ny, cpml, cpt):
    from paper_2211_05647_gb300 import Solver
    out = []
    for tz in (0, 32):
        s = Solver(dict(ndim=2, nx=nx, ny=ny, nz=1, dx=1e-3, courant=0.5, cpml_cells=cpml, mur=0, precision="f32"))
        s.set_source(kind="gauss", amp=1.0, tau=1e-11, t0=0.0, i=nx // 2, j=ny // 2)
        if tz:
            s.set_option("stencil_tz", tz)
        else:
            assert s.launch_shapes()["cells_per_thread"] == cpt
        rng = np.random.default_rng(3)
        for q in FIELDS[2]:
            s.write(q, rng.standard_normal(nx * ny, dtype=np.float32) / (1.0 if q[0] == "e" else 377.0))
        s.step(11)
        out.append([s.read(q) for q in FIELDS[2]])
    assert all(bool((a == b).all()) for a, b in zip(*out))

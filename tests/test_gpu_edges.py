"""Kernels at the sizes where their work splits can go wrong (edges of pieces,
tiles and chunks, remainders, the smallest grids), against the FP64 oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_05097_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf():
    from paper_2311_05097_gb300 import build
    build.build()
    from paper_2311_05097_gb300 import pf as _pf
    _pf.load()
    return _pf


def _pair(pf, c, steps, precision="p64", particles=(), walls=False, config=None):
    g = pf.Sim(c["shape"], precision=precision, walls_y=walls, **c["params"])
    o = O.OracleSim(c["shape"], O.make_params(**c["params"]))
    if walls:
        o.set_walls(True)
    for k, q in enumerate(particles):
        g.set_particle(k, **q)
        o.set_particle(k, O.Particle(**q))
    g.init(c["phi0"], c["phi"], c.get("u"))
    o.init(c["phi0"], c["phi"], c.get("u"))
    if config is not None:
        g.set_config(*config)
    g.step(steps)
    o.step(steps)
    return g, o


@pytest.mark.parametrize("shape,walls", [
    ((4, 4), False), ((5, 31), True), ((33, 32), False), ((37, 65), True), ((700, 33), False),
    ((4, 4, 4), False), ((5, 6, 33), True), ((9, 8, 64), False),
])
def test_diagnostics_row_pieces(pf, shape, walls):
    """The diagnostics' row pieces of 32 cells: rows shorter than, equal to and
    one past a piece, more rows than warps.  Sums of FP64 terms in another
    order: 1e-12 relative, as the fields' parity."""
    c = W.small_case(shape, seed=3, solid=min(shape) > 8, theta_deg=70.0, u_amp=0.01)
    g, o = _pair(pf, c, 3, walls=walls)
    for _ in range(2):  # (the ticket of the last block is reset by each call)
        dg, do = g.diagnostics(), o.diagnostics()
        for k in ("mass", "E_F", "E_K"):
            assert abs(dg[k] - do[k]) <= 1e-12 * max(abs(do[k]), 1e-3), (k, dg[k], do[k])
        assert dg["nan_flag"] == 0

"""GPU step kernels chosen by size, type or option, at the sizes where each can
go wrong, against the FP64 oracle or bitwise against the plain one-step kernels."""
import numpy as np
import pytest

import inputs
from test_gpu_parity import D2, D3, FP64, T  # noqa: F401  (T: the library fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,shape,pm", [(D2, (5, 4, 1), 0), (D2, (37, 6, 1), 3), (D3, (5, 4, 3), 0),
                                              (D3, (34, 3, 4), 7)])
@pytest.mark.parametrize("inplace", [False, True])
def test_fp64_collision_with_a_force_on_every_axis(T, O, lattice, shape, pm, inplace):  # noqa: F811
    """The FP64 two-relaxation-time collision with a body force along every axis
    (and buoyancy), from random populations: three steps against the oracle.
    Tolerance: a step's stored values are O(0.3) and differ by a few roundings
    of 2^-53 each; three steps of them stay below 1e-14."""
    nx, ny, nz = shape
    kw = dict(periodic_mask=pm, body_force=[1e-3, -2e-3, 5e-4 if lattice == D3 else 0.0])
    o = O.Sim(nx, ny, nz, lattice=lattice, Ra=1e5, Pr=0.71, Ma=0.1, **kw)
    qf, qg = (9, 5) if lattice == D2 else (19, 7)
    f = inputs.uniform_array(31 + nx, (qf,) + o.shape, 0.02, 0.2)
    gg = inputs.uniform_array(32 + nx, (qg,) + o.shape, -0.1, 0.1)
    g = T.Sim(nx, ny, nz, lattice=lattice, Ra=1e5, Pr=0.71, Ma=0.1, precision=FP64,
              streaming=T.TLBM_STREAM_INPLACE if inplace else T.TLBM_STREAM_PULL, **kw)
    g.set_populations(f, gg)
    o.set_populations(f, gg)
    g.step(3)
    o.step(3)
    (fg, tg), (fo, to) = g.get_populations(), o.get_populations()
    assert np.abs(fg - fo).max() < 1e-14 and np.abs(tg - to).max() < 1e-14
    g.close()

"""The same bits whichever kernel steps a cell: calls of one step and of many,
either streaming scheme, a batch, a resumed checkpoint."""
import numpy as np
import pytest

from test_gpu_parity import D2, D3, T  # noqa: F401  (T: the library fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,shape,pm", [(D2, (65, 41, 1), 0), (D2, (130, 67, 1), 1), (D2, (53, 18, 1), 2),
                                              (D2, (700, 500, 1), 0), (D3, (35, 9, 12), 0)])
@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("prec", [0, 1, 2, 3])
def test_wall_values_do_not_depend_on_the_kernel(T, tmp_path, lattice, shape, pm, walls, prec):  # noqa: F811
    """Isothermal walls at temperatures whose product with the thermal weight is
    not exact (0.7 and -0.3), a body force, and for 16-bit storage a scale other
    than the default: single steps, blocks of steps, in-place streaming, a
    batch and a resumed checkpoint give the same state, bit for bit."""
    kw = dict(lattice=lattice, precision=prec, walls=walls, periodic_mask=pm, Th=0.7, Tc=-0.3,
              body_force=[1e-4, -2e-4, 3e-4])
    if prec > 1:
        kw["store_scale"] = 64.0
    phys = dict(Ra=1e6, Pr=0.71, Ma=0.1)

    def sim(calls, streaming=T.TLBM_STREAM_PULL):
        s = T.Sim(*shape, **phys, **kw, streaming=streaming)
        s.init(5, 1e-2)
        for n in calls:
            s.step(n)
        out = s.get_populations()
        s.close()
        return out

    def resumed():
        a, b = (T.Sim(*shape, **phys, **kw) for _ in range(2))
        a.init(5, 1e-2)
        a.step(17)
        path = str(tmp_path / "state.ckpt")
        a.save(path)
        b.load(path)
        b.step(20)
        out = b.get_populations()
        a.close()
        b.close()
        return out

    def batch(calls):
        b = T.Batch([shape + (1e6, 0.71, 0.1, 5)], **kw)
        b.init(1e-2)
        for n in calls:
            b.step(n)
        out = b.get_populations(0)
        b.close()
        return out

    ref = sim([1] * 37)
    assert np.isfinite(ref[0]).all() and np.isfinite(ref[1]).all()
    others = {"block": sim([37]), "blocks": sim([20, 1, 16]), "in place": sim([37], T.TLBM_STREAM_INPLACE),
              "resumed": resumed(), "batch": batch([37]), "batch of single steps": batch([1] * 37)}
    differ = [k for k, v in others.items() if not (np.array_equal(ref[0], v[0]) and np.array_equal(ref[1], v[1]))]
    assert not differ, differ


@pytest.mark.parametrize("lattice,shape", [(D2, (65, 41, 1)), (D3, (35, 9, 12)), (D3, (384, 5, 6))])
@pytest.mark.parametrize("prec", [1, 2, 3])
def test_a_body_force_gives_the_same_bits_in_every_variant(T, lattice, shape, prec):  # noqa: F811
    """FP32 and 16-bit cells with buoyancy and a body force along the same axis:
    one node or several per thread, rows in a pipeline, the staged kernel,
    in-place streaming and a batch step bitwise as the default kernel (of 384
    nodes a row that is the staged one in 16 bits, one thread per node in place)."""
    kw = dict(lattice=lattice, precision=prec, body_force=[1e-4, -2e-4, 3e-4])

    def sim(choose, streaming=T.TLBM_STREAM_PULL):
        s = T.Sim(*shape, Ra=1e6, Pr=0.71, Ma=0.1, **kw, streaming=streaming)
        try:
            choose(s)
        except T.TlbmError as e:
            assert e.code == T.TLBM_ERR_UNSUPPORTED  # a variant that is not built
            return None
        s.init(5, 1e-2)
        for _ in range(11):
            s.step(1)
        out = s.get_populations()
        s.close()
        return out

    ref = sim(lambda s: None)
    others = {f"{v} nodes, {r} rows": sim(lambda s, v=v, r=r: s.set_variant(v, 2, 0, 0, r)) for v in (1, 2, 4, 8)
              for r in (1, 2, 4)}
    others["staged"] = sim(lambda s: s.set_staged())
    others["in place"] = sim(lambda s: None, T.TLBM_STREAM_INPLACE)
    b = T.Batch([shape + (1e6, 0.71, 0.1, 5)], **kw)
    b.init(1e-2)
    for _ in range(11):
        b.step(1)
    others["batch"] = b.get_populations(0)
    b.close()
    assert sum(v is not None for v in others.values()) >= 6
    differ = [k for k, v in others.items()
              if v is not None and not (np.array_equal(ref[0], v[0]) and np.array_equal(ref[1], v[1]))]
    assert not differ, differ

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


def _reference_fields(f, g, lattice, derived):
    """rho, u, T in FP64 from populations f, g (the definitions of §2.2)."""
    if lattice == D2:
        E = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
    else:
        E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
             (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
             (0, 1, -1), (0, -1, 1)]
    rho, T = f.sum(0), g.sum(0)
    dim = len(E[0])
    j = [sum(e[a] * f[i] for i, e in enumerate(E) if e[a]) for a in range(dim)]
    j[-1] = j[-1] + 0.5 * rho * derived["gbeta"] * T
    return rho, [v / rho for v in j], T


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("lattice,shape", [(D2, (3, 3, 1)), (D2, (33, 5, 1)), (D2, (64, 40, 1)), (D3, (5, 4, 3)),
                                           (D3, (65, 3, 4))])
@pytest.mark.parametrize("inplace", [False, True])
def test_fields_and_reductions_of_every_state_order(T, prec, lattice, shape, inplace):  # noqa: F811
    """Fields (FP64 and FP32 arrays), Nusselt number, energy and mass against
    their definitions, for every storage and state order (pull, natural,
    swapped).  FP64 fields: a few roundings of 2^-53 of O(1) values.  FP32 fields:
    the FP64 ones rounded, at most one unit apart where a rounding boundary
    falls between the two evaluations.  Sums: FP64 storage to 1e-13 of the
    terms' magnitudes, the others to the 2^-24 roundings of an FP32 term (about
    20 of them)."""
    import torch

    nx, ny, nz = shape
    qf, qg = (9, 5) if lattice == D2 else (19, 7)
    full = (ny, nx) if lattice == D2 else (nz, ny, nx)
    s = T.Sim(nx, ny, nz, lattice=lattice, Ra=1e5, Pr=0.71, Ma=0.1, precision=prec,
              streaming=T.TLBM_STREAM_INPLACE if inplace else T.TLBM_STREAM_PULL)
    w = np.array([16, 4, 4, 4, 4, 1, 1, 1, 1] if lattice == D2 else [12] + [2] * 6 + [1] * 12) / 36.0
    f = w.reshape((qf,) + (1,) * len(full)) * (1 + 0.1 * inputs.uniform_array(3 + nx, (qf,) + full, -1, 1))
    g = inputs.uniform_array(4 + nx, (qg,) + full, -0.1, 0.1)
    s.set_populations(f, g)
    d = s.derived()
    for n in (0, 1, 1):
        s.step(n)
        fs, gs = s.get_populations()
        rho, u, tt = _reference_fields(fs, gs, lattice, d)
        m = {k: v.cpu().numpy() for k, v in s.macros().items()}
        for name, ref in (("rho", rho), ("T", tt), ("ux", u[0]), ("uy", u[1])) + ((("uz", u[2]),) if lattice else ()):
            assert np.abs(m[name] - ref).max() < 2e-14, (name, n)
        m32 = {k: v.cpu().numpy() for k, v in s.macros(torch.float32).items()}
        for name in m32:
            r = m[name].astype(np.float32)
            assert (np.abs(m32[name] - r) <= np.spacing(np.abs(r))).all(), (name, n)
        uh = u[-1]
        terms = {"nu": uh * tt, "e": 0.5 * rho * sum(v * v for v in u), "m": rho}
        tol = {k: (1e-13 if prec == 0 else 20 * 2.0 ** -24) * np.abs(v).sum() for k, v in terms.items()}
        L, alpha = full[0], d["alpha"]
        nu = s.nusselt(allow_diverged=True)
        e, mass = s.energy(allow_diverged=True)
        assert abs((nu - 1) * alpha / L * rho.size - terms["nu"].sum()) <= tol["nu"]
        assert abs(e - terms["e"].sum()) <= tol["e"] and abs(mass - rho.sum()) <= tol["m"]
    s.close()


@pytest.mark.parametrize("prec", [1, 3])
def test_fields_outside_the_double_fp32_range(T, prec):  # noqa: F811
    """FP32 fields of nodes whose density, momentum or temperature is too large,
    zero, negative or not finite for the double-FP32 evaluation are those of FP64
    arithmetic, cast."""
    import torch

    s = T.Sim(40, 6, Ra=1e5, Pr=0.71, Ma=0.1, precision=prec)
    s.init(1, 0.0)
    f, g = s.get_populations()
    for k, v in enumerate((1e17, -1e20, np.inf, -np.inf, np.nan, -1.0, -40.0 / 9.0)):
        f[1, 2, 5 * k] = v
        g[2, 4, 5 * k] = v
    s.set_populations(f, g)
    m = s.macros()
    m32 = s.macros(torch.float32)
    for k in m:
        a, b = m32[k].cpu().numpy(), m[k].float().cpu().numpy()
        fin = np.isfinite(b)
        assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b)), k
        assert (np.abs(a[fin] - b[fin]) <= np.spacing(np.abs(b[fin]))).all(), k
    s.close()


@pytest.mark.parametrize("lattice,prec,n", [(D2, 1, 70), (D2, 2, 64), (D3, 0, 65), (D2, 0, 1)])
def test_reductions_of_a_batch_equal_those_of_its_cells(T, lattice, prec, n):  # noqa: F811
    """tlbm_batch_nusselt and tlbm_batch_status reduce up to 64 cells per launch:
    bitwise the numbers of the cells reduced alone, also past the first 64, and
    a diverged cell is named."""
    size = lambda i: (17 + 3 * (i % 7), 12 + i % 5, 9 if lattice == D3 else 1)  # noqa: E731
    b = T.Batch([size(i) + (1e5, 0.71, 0.1, i) for i in range(n)], lattice=lattice, precision=prec)
    b.init(1e-2)
    b.step(11)
    nu = b.nusselt()
    assert nu == [T.tlbm_nusselt(b.instance(i)) for i in range(n)] and b.status() == [False] * n
    f, g = b.get_populations(n - 1)
    f[1] = np.nan
    T.tlbm_set_populations(b.instance(n - 1), f, g)
    assert b.status() == [False] * (n - 1) + [True]
    with pytest.raises(T.TlbmError) as ei:
        b.nusselt()
    assert ei.value.code == T.TLBM_ERR_DIVERGED and f"instance {n - 1} " in str(ei.value)
    b.close()


@pytest.mark.parametrize("lattice,shape,walls,pm", [
    (D2, (3, 3, 1), 0, 0), (D2, (31, 5, 1), 1, 0), (D2, (33, 4, 1), 0, 1), (D2, (129, 9, 1), 0, 2),
    (D3, (3, 3, 3), 0, 0), (D3, (33, 4, 5), 0, 0), (D3, (65, 3, 4), 1, 5), (D3, (7, 5, 6), 0, 6)])
@pytest.mark.parametrize("inplace", [False, True])
def test_fp64_threads_in_memory_order_equal_rows(T, lattice, shape, walls, pm, inplace):  # noqa: F811
    """The FP64 default (one thread per node in memory order, warps over row and
    plane ends) steps bitwise as the kernels with warps inside a row."""
    out = []
    for rows in (False, True):
        s = T.Sim(*shape, lattice=lattice, Ra=1e5, Pr=0.71, Ma=0.1, precision=FP64, walls=walls, periodic_mask=pm,
                  streaming=T.TLBM_STREAM_INPLACE if inplace else T.TLBM_STREAM_PULL)
        if rows:
            s.set_variant(2 if lattice == D2 else 1, 2, 32, 1, 1)
        s.init(3, 1e-2)
        s.step(7)
        out.append(s.get_populations())
        s.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("shape,walls,pm", [((16, 16), 0, 0), ((17, 33), 0, 0), ((65, 31), 1, 0), ((3, 9), 0, 0),
                                            ((130, 67), 0, 1), ((53, 18), 0, 2), ((29, 29), 0, 3), ((129, 129), 0, 0),
                                            ((270, 40), 1, 2)])
def test_several_steps_per_launch_equal_single_steps(T, prec, shape, walls, pm):  # noqa: F811
    """Small 2D cells advance several steps per launch in calls of 16 steps or
    more: bitwise the states, counters and diagnostics of one-step launches, for
    step counts that are no multiple of a launch's or a graph block's, on walls
    and periodic faces, and from either buffer."""
    kw = dict(Ra=1e5, Pr=0.71, Ma=0.1, precision=prec, walls=walls, periodic_mask=pm)
    a, b = T.Sim(*shape, **kw), T.Sim(*shape, **kw)
    T.tlbm_set_graph(b.h, 0)  # one launch per step
    for s in (a, b):
        s.init(3, 1e-2)
    for n in (17, 1, 16, 139):
        la = a.launches
        a.step(n)
        b.step(n)
        assert n < 16 or a.launches - la <= n // 2 + 2
        assert (a.launches - la - n) % 2 == 0  # the buffer that single steps end in
        (fa, ga), (fb, gb) = a.get_populations(), b.get_populations()
        assert np.array_equal(fa, fb) and np.array_equal(ga, gb), n
        assert a.status() == b.status() and a.nusselt() == b.nusselt()
    a.close()
    b.close()


@pytest.mark.parametrize("shape,walls", [((560, 450), 0), ((561, 447), 1), ((562, 449), 0), ((614, 410), 0),
                                         ((615, 409), 1), ((101, 2500), 0), ((8193, 31), 0), ((30000, 9), 1),
                                         ((100000, 3), 0), ((513, 513), 0)])
@pytest.mark.parametrize("prec", [1, 2, 3])
def test_three_steps_per_pass_equal_single_steps(T, shape, walls, prec):  # noqa: F811
    """Larger FP32, FP16 and BF16 cells march three steps per pass over memory in strips of 56
    columns: bitwise one-step launches at every remainder of the width by the
    strip and of the step count by three, on both wall configurations, short
    and long segments, and from either buffer."""
    kw = dict(Ra=1e6, Pr=0.71, Ma=0.1, precision=prec, walls=walls)
    a, b = T.Sim(*shape, **kw), T.Sim(*shape, **kw)
    T.tlbm_set_graph(b.h, 0)
    for s in (a, b):
        s.init(3, 1e-2)
    for n in (16, 20, 1, 33):
        la = a.launches
        a.step(n)
        b.step(n)
        assert n < 16 or a.launches - la == n // 3 + n % 3 or (prec > 1 and shape[0] * shape[1] < 270000)
        (fa, ga), (fb, gb) = a.get_populations(), b.get_populations()
        assert np.array_equal(fa, fb) and np.array_equal(ga, gb), n
        assert a.status() == b.status() and a.nusselt() == b.nusselt()
    a.close()
    b.close()


@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("n", [1, 5, 70])
@pytest.mark.parametrize("prec", [1, 2, 3])
def test_marching_batch_equals_single_steps(T, walls, n, prec):  # noqa: F811
    """An FP32, FP16 or BF16 batch marches three steps per launch in calls of 16 steps or more,
    64 cells to a launch: bitwise the batch with one step per launch, for cells
    from one warp to several blocks, every remainder of the step count by three,
    before and after tuning, and with work on a borrowed cell in between."""
    size = lambda i: ((3, 57, 112, 113, 200, 65, 56)[i % 7], (9, 3, 70, 31, 129)[i % 5], 1)  # noqa: E731
    inst = [size(i) + (1e5 * (1 + i), (0.71, 7.0)[i % 2], 0.1, i) for i in range(n)]
    a, b = T.Batch(inst, precision=prec, walls=walls), T.Batch(inst, precision=prec, walls=walls)
    v = b.variant
    b.set_variant(v[0], v[1], v[2], v[3], 0)  # one step per launch
    for s in (a, b):
        s.init(1e-2)
    for steps in (16, 35, 1, 18):
        la = a.launches
        a.step(steps)
        b.step(steps)
        if steps == 16:  # not yet tuned
            assert a.launches - la == 5 * (1 + (n > 64)) + 1
        for k in range(0, n, 9 if n > 9 else 1):
            (fa, ga), (fb, gb) = a.get_populations(k), b.get_populations(k)
            assert np.array_equal(fa, fb) and np.array_equal(ga, gb), (steps, k)
        assert a.nusselt(True) == b.nusselt(True) and a.status() == b.status()
        if steps == 16:
            f, g = a.get_populations(0)
            for s in (a, b):
                T.tlbm_set_populations(s.instance(0), f * 1.001, g)
                s.step(0)
            a.autotune(2)
    a.close()
    b.close()


@pytest.mark.parametrize("choice,n", [("variant", 40), ("staged", 40), ("graph", 40), ("none", 15)])
def test_launch_choices_of_the_caller_stay(T, choice, n):  # noqa: F811
    """A handle whose step variant, staged kernel or graph the caller chose keeps
    one launch per step; so do short calls."""
    s = T.Sim(65, 40, Ra=1e5, Pr=0.71, Ma=0.1, precision=1)
    if choice == "variant":
        s.set_variant(2, 2, 0, 0, 1)
    elif choice == "staged":
        s.set_staged()
    elif choice == "graph":
        T.tlbm_set_graph(s.h, 16)
    s.init(1, 1e-3)
    c0 = s.launches
    s.step(n)
    assert s.launches - c0 == n
    s.close()


@pytest.mark.parametrize("prec", [2, 3])
@pytest.mark.parametrize("shape,walls,pm,inplace", [
    ((3, 3, 3), 0, 0, False), ((33, 5, 7), 1, 0, False), ((65, 4, 3), 0, 5, False), ((31, 6, 4), 0, 1, False),
    ((383, 5, 6), 0, 0, False), ((384, 5, 6), 0, 0, False), ((448, 6, 3), 1, 0, False), ((449, 6, 3), 0, 4, False),
    ((160, 158, 158), 0, 0, False),
    ((3, 3, 3), 0, 0, True), ((33, 5, 7), 1, 0, True), ((65, 4, 3), 0, 5, True), ((31, 6, 4), 0, 1, True),
    ((161, 160, 162), 0, 0, True), ((192, 160, 140), 0, 0, True)])
def test_16bit_3d_kernels_by_size_equal_node_pairs(T, shape, walls, pm, inplace, prec):  # noqa: F811
    """The kernel a 3D FP16 or BF16 cell gets by its size (either side of each
    border) steps bitwise as warps of node pairs inside a row."""
    import torch

    out = []
    for pairs in (False, True):
        s = T.Sim(*shape, lattice=D3, Ra=1e5, Pr=0.71, Ma=0.1, precision=prec, walls=walls, periodic_mask=pm,
                  streaming=T.TLBM_STREAM_INPLACE if inplace else T.TLBM_STREAM_PULL)
        if pairs:
            s.set_variant(2, 2, 32, 1, 1)
        s.init(3, 1e-2)
        s.step(5)
        n = shape[0] * shape[1] * shape[2]
        if n < 10000:
            out.append([torch.from_numpy(np.ascontiguousarray(q)) for q in s.get_populations()])
        else:
            m = s.macros()
            out.append([m[k].cpu() for k in sorted(m)])
        s.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))


BOUNDS_SCRIPT = """
import hashlib, json, sys
sys.path.insert(0, {root!r})
from paper_2211_03160_gb300 import tlbm as T
out = {{}}
for lattice, shape, walls, pm, prec, inplace, steps in {cases!r}:
    s = T.Sim(*shape, lattice=lattice, Ra=1e5, Pr=0.71, Ma=0.1, precision=prec, walls=walls, periodic_mask=pm,
              streaming=1 if inplace else 0)
    s.init(5, 1e-2)
    s.step(steps)
    m = s.macros()
    f, g = s.get_populations()
    h = hashlib.sha256(f.tobytes() + g.tobytes() + m["T"].cpu().numpy().tobytes()).hexdigest()
    try:
        bad = T.tlbm_bounds_violations(s.h)
    except T.TlbmError:
        bad = None
    out[repr((lattice, shape, walls, pm, prec, inplace))] = [h, s.nusselt(), bad]
    s.close()
print("RESULT " + json.dumps(out))
"""


def test_default_kernels_stay_inside_their_buffers(T):  # noqa: F811
    """The kernels a default handle runs in calls of 16 steps and more, on the
    bounds-checked build: no access leaves the population buffers, and states,
    fields and reductions are those of the release build."""
    import json
    import os
    import subprocess
    import sys

    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    cases = [(D2, (nx, ny, 1), walls, pm, prec, False, 37) for nx, ny, walls, pm in
             ((3, 9, 0, 0), (37, 16, 1, 0), (130, 21, 0, 1), (33, 70, 0, 3), (700, 500, 0, 0)) for prec in (0, 1, 2)]
    cases += [(D3, (35, 6, 5), 0, 4, 0, inplace, 17) for inplace in (False, True)]
    script = BOUNDS_SCRIPT.format(root=root, cases=cases)
    res = []
    for debug in ("0", "1"):
        r = subprocess.run([sys.executable, "-c", script], env=dict(os.environ, TLBM_DEBUG_BOUNDS=debug),
                           capture_output=True, text=True, timeout=900)
        assert r.returncode == 0, r.stderr[-2000:]
        res.append(json.loads(r.stdout.split("RESULT ")[1]))
    for k in res[0]:
        assert res[1][k][2] == 0, k
        assert res[0][k][:2] == res[1][k][:2], k


def _field_time(T, shape, prec, dtype, reduce=False):  # noqa: F811
    """Seconds of one call for the fields (or the Nusselt number) of a 3D state, the least of 8."""
    import time

    import torch

    s = T.Sim(*shape, lattice=D3, Ra=1e6, Pr=0.71, Ma=0.1, precision=prec)
    s.init(1, 1e-2)
    out = [torch.empty(s.N, dtype=dtype, device="cuda") for _ in range(5)]
    code = T.TLBM_OUT_F32 if dtype == torch.float32 else T.TLBM_OUT_F64
    best = 1e9
    for _ in range(8):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(10):
            if reduce:
                s.nusselt(allow_diverged=True)
            else:
                T.tlbm_macros(s.h, *out, code)
        torch.cuda.synchronize()
        best = min(best, (time.perf_counter() - t0) / 10)
    s.close()
    return best


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
def test_fields_of_narrow_rows_cost_as_those_of_wide_ones(T, prec):  # noqa: F811
    """What the FP64 pipe bounds (FP64 fields, and fields and reductions of FP64
    states) takes for a cell with three nodes a row at most three times as long
    as for as many nodes in rows of 100: no warp is spent on a row (which costs
    about ten times)."""
    import torch

    narrow, wide = (3, 600, 600), (100, 108, 100)
    kinds = [(torch.float64, False)] + ([(torch.float32, False), (torch.float64, True)] if prec == 0 else [])
    for dtype, reduce in kinds:
        t = [_field_time(T, sh, prec, dtype, reduce) for sh in (narrow, wide)]
        assert t[0] < 3 * t[1], (dtype, reduce, t)


@pytest.mark.parametrize("prec", [2, 3])
def test_fp64_fields_of_16bit_states_cost_as_those_of_fp32_ones(T, prec):  # noqa: F811
    """FP64 fields are bound by the FP64 pipe: unscaling every 16-bit value there
    would take 1.3 times the FP32 state's fields."""
    import torch

    shape = (161, 161, 161)
    t16, t32 = (_field_time(T, shape, q, torch.float64) for q in (prec, 1))
    assert t16 < 1.15 * t32, (t16, t32)


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("inplace", [False, True])
def test_periodic_faces_cost_as_walls(T, prec, inplace):  # noqa: F811
    """The steps of a small 3D cell with every axis periodic take at most 1.3
    times those of the cell with walls (the populations leaving through each
    face are as many)."""
    import torch

    best = []
    for pm in (0, 7):
        s = T.Sim(9, 9, 9, lattice=D3, Ra=1e5, Pr=0.71, Ma=0.1, precision=prec, periodic_mask=pm,
                  streaming=T.TLBM_STREAM_INPLACE if inplace else T.TLBM_STREAM_PULL)
        s.init(1, 1e-3)
        ms = []
        for _ in range(10):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            s.step(64)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        best.append(min(ms))
        s.close()
    assert best[1] < 1.3 * best[0], best


@pytest.mark.parametrize("lattice,shape,prec,inplace", [
    (D2, (129, 129, 1), FP64, False), (D2, (513, 513, 1), 1, False), (D2, (700, 500, 1), 2, False),
    (D3, (33, 33, 33), FP64, False), (D3, (33, 33, 33), FP64, True), (D3, (33, 33, 33), 2, True),
    (D3, (33, 33, 33), 3, False)])
def test_default_arguments_give_the_choice_back(T, lattice, shape, prec, inplace):  # noqa: F811
    """tlbm_set_variant with every argument 0, at once and after another variant:
    the launches and the bits of a handle as created, and its speed (within a
    quarter; the kernels a chosen variant leaves take 1.4 times as long or more)
    where no staged kernel is behind it."""
    import torch

    got = []
    for calls in ((), ((),), ((2 if lattice == D2 or prec > 1 else 1, 2, 32, 1, 1), ())):
        s = T.Sim(*shape, lattice=lattice, Ra=1e6, Pr=0.71, Ma=0.1, precision=prec,
                  streaming=T.TLBM_STREAM_INPLACE if inplace else T.TLBM_STREAM_PULL)
        for c in calls:
            s.set_variant(*c)
        s.init(3, 1e-2)
        l0 = s.launches
        s.step(64)
        n = s.launches - l0
        state = s.get_populations()
        best = 1e9
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            s.step(64)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        got.append((n, state, best))
        s.close()
    for n, state, ms in got[1:]:
        assert n == got[0][0] and ms < 1.25 * got[0][2], (n, ms, got[0][0], got[0][2])
        assert all(np.array_equal(p, q) for p, q in zip(state, got[0][1]))


@pytest.mark.parametrize("shape,walls", [((560, 490), 0), ((561, 487), 1), ((562, 489), 0), ((614, 450), 0),
                                         ((615, 449), 1), ((101, 2700), 0), ((8193, 37), 0), ((700, 500), 1)])
@pytest.mark.parametrize("prec", [2, 3])
def test_16bit_cells_march_as_single_steps(T, shape, walls, prec):  # noqa: F811
    """FP16 and BF16 cells of 270,000 nodes and more, all of which march: bitwise
    one-step launches, with the launches of three steps a pass, at remainders of
    the width by the strip and of the step count by three, in tall and flat
    cells, and from either buffer."""
    kw = dict(Ra=1e6, Pr=0.71, Ma=0.1, precision=prec, walls=walls)
    a, b = T.Sim(*shape, **kw), T.Sim(*shape, **kw)
    T.tlbm_set_graph(b.h, 0)
    for s in (a, b):
        s.init(3, 1e-2)
    for n in (16, 20, 1, 33):
        la = a.launches
        a.step(n)
        b.step(n)
        assert a.launches - la == (n // 3 + n % 3 if n >= 16 else n)
        (fa, ga), (fb, gb) = a.get_populations(), b.get_populations()
        assert np.array_equal(fa, fb) and np.array_equal(ga, gb), n
        assert a.status() == b.status() and a.nusselt() == b.nusselt()
    a.close()
    b.close()


BATCH_BOUNDS_SCRIPT = """
import hashlib, json, sys
sys.path.insert(0, {root!r})
from paper_2211_03160_gb300 import tlbm as T
out = {{}}
def count(h):
    try:
        return T.tlbm_bounds_violations(h)
    except T.TlbmError:
        return None
for lattice, shape, walls, pm, prec, inplace, steps in {cells!r}:
    s = T.Sim(*shape, lattice=lattice, Ra=1e5, Pr=0.71, Ma=0.1, precision=prec, walls=walls, periodic_mask=pm,
              streaming=1 if inplace else 0)
    s.init(5, 1e-2)
    s.step(steps)
    m = [s.macros(d) for d in (None, __import__("torch").float32)]
    f, g = s.get_populations()
    h = hashlib.sha256(f.tobytes() + g.tobytes() + b"".join(q[k].cpu().numpy().tobytes() for q in m for k in sorted(q)))
    out[repr((lattice, shape, walls, pm, prec, inplace))] = [h.hexdigest(), s.nusselt(), count(s.h)]
    s.close()
for prec, sizes, steps in {batches!r}:
    b = T.Batch([tuple(q) + (1, 1e5 * (1 + i), 0.71, 0.1, i) for i, q in enumerate(sizes)], precision=prec)
    b.init(1e-2)
    l0 = b.launches
    b.step(steps)
    n = b.launches - l0
    nu = b.nusselt()
    for k in range(len(sizes)):
        f, g = b.get_populations(k)
        out[repr((prec, len(sizes), k))] = [hashlib.sha256(f.tobytes() + g.tobytes()).hexdigest(), [n, nu[k]], count(b.instance(k))]
    b.close()
print("RESULT " + json.dumps(out))
"""


def test_marching_batches_and_16bit_defaults_stay_inside_their_buffers(T):  # noqa: F811
    """The bounds-checked build on batches that march (70 cells, two launches a
    pass), on BF16 and 16-bit 3D cells by size, on narrow cells (whose fields
    are walked in memory order) and with every face periodic: no access leaves
    the population buffers, and all results are those of the release build."""
    import json
    import os
    import subprocess
    import sys

    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    cells = [(D2, s, w, pm, 3, False, 37) for s, w, pm in
             (((3, 9, 1), 0, 0), ((33, 70, 1), 0, 3), ((130, 21, 1), 0, 1), ((562, 489, 1), 1, 0))]
    cells += [(D3, (nx, 6, 5), w, pm, prec, inplace, 17) for nx, w, pm in
              ((3, 0, 0), (35, 0, 7), (384, 0, 0), (448, 1, 0), (449, 0, 4)) for prec in (2, 3) for inplace in (False, True)]
    cells += [(D3, (5, 4, 6), 0, pm, prec, inplace, 17) for pm in (3, 5, 7) for prec in (0, 1) for inplace in (False, True)]
    sizes = [((3, 57, 112, 113, 200, 65, 56)[i % 7], (9, 3, 70, 31, 129)[i % 5]) for i in range(70)]
    script = BATCH_BOUNDS_SCRIPT.format(root=root, cells=cells, batches=[(prec, sizes, 20) for prec in (1, 2, 3)])
    res = []
    for debug in ("0", "1"):
        r = subprocess.run([sys.executable, "-c", script], env=dict(os.environ, TLBM_DEBUG_BOUNDS=debug),
                           capture_output=True, text=True, timeout=900)
        assert r.returncode == 0, r.stderr[-2000:]
        res.append(json.loads(r.stdout.split("RESULT ")[1]))
    for k in res[0]:
        assert res[1][k][2] == 0, k
        assert res[0][k][:2] == res[1][k][:2], k
    assert sum(v[1][0] == 6 * 2 + 2 for v in res[0].values() if isinstance(v[1], list)) == 3 * 70  # they marched


@pytest.mark.parametrize("lattice,shape", [(D2, (513, 400, 1)), (D2, (33, 300, 1)), (D3, (65, 50, 40))])
@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("noise,steps", [(1e-2, 300), (1e-6, 60), (1e-9, 200)])
def test_fp32_fields_of_weak_and_developed_flow(T, lattice, shape, prec, noise, steps):  # noqa: F811
    """FP32 fields are the FP64 ones rounded also where the populations nearly
    cancel (a velocity far below them, as at the onset of convection): within
    half a unit and 2^-8 of one, what the two evaluations may differ by."""
    import torch

    s = T.Sim(*shape, lattice=lattice, Ra=1e7, Pr=0.71, Ma=0.1, precision=prec)
    s.init(7, noise)
    s.step(steps)
    m, m32 = s.macros(), s.macros(torch.float32)
    for k in m32:
        ref = m[k].cpu().numpy()
        ulp = np.spacing(np.abs(ref.astype(np.float32))).astype(np.float64)
        assert (np.abs(m32[k].cpu().numpy().astype(np.float64) - ref) <= (0.5 + 2.0 ** -8) * ulp).all(), k
    s.close()

"""The channels-last layer kernels (forward, both gradients, bias gradient) and
the one-launch optimiser step against the FP64 CPU oracle and the NCHW calls.
Tolerances are those of the NCHW kernels' tests: FP32 accumulation of BF16
products to 1e-5 of the largest value, BF16 results to 2^-8 of their value."""
import numpy as np
import pytest

import inputs
from oracle import conv_oracle as CO
from test_gpu_surrogate import T, _bf16, _np  # noqa: F401  (T: the library fixture)

pytestmark = pytest.mark.gpu

# one group and two, ragged channels, one pixel row, strips (W > 126), the widest
# strip (two tiles in shared memory), tiles that end inside an image
SHAPES = [(2, 5, 32, 13, 11), (3, 32, 32, 9, 17), (1, 32, 3, 65, 65), (2, 7, 5, 4, 3), (1, 17, 9, 5, 260),
          (2, 3, 2, 3, 127), (1, 16, 16, 1, 1), (2, 32, 32, 30, 126), (1, 20, 32, 40, 89), (5, 32, 17, 65, 65)]


def _cl(T, x, s):  # noqa: F811
    import torch

    B, ch, H, W = x.shape
    out = torch.full((B, H, W, 16 * ((ch + 15) // 16)), 7.0, dtype=torch.bfloat16, device="cuda")
    T.tlbm_conv_channels_last(x, B, ch, H, W, out, s)
    return out


@pytest.mark.parametrize("B,cin,cout,H,W", SHAPES)
def test_channels_last_layers_match_oracle(T, B, cin, cout, H, W):  # noqa: F811
    import torch

    s = torch.cuda.current_stream()
    x = _bf16(inputs.uniform_array(1 + cin, (B, cin, H, W), -1, 1)).cuda()
    w32 = torch.tensor(inputs.uniform_array(2 + cin, (cout, cin, 3, 3), -0.3, 0.3), dtype=torch.float32).cuda()
    bias = torch.tensor(inputs.uniform_array(3, (cout,), -0.1, 0.1), dtype=torch.float32).cuda()
    a = torch.empty(T.tlbm_conv3x3_weight_elems(cin), dtype=torch.bfloat16, device="cuda")
    T.tlbm_conv3x3_pack_weights(w32, cout, cin, a, s)
    xc = _cl(T, x, s)
    ref_cl = torch.zeros_like(xc)
    ref_cl[..., :cin] = x.permute(0, 2, 3, 1)
    assert torch.equal(xc, ref_cl)
    y = torch.empty((B, cout, H, W), dtype=torch.float32, device="cuda")
    act = torch.full((B, H, W, 16 * ((cout + 15) // 16)), 7.0, dtype=torch.bfloat16, device="cuda")
    T.tlbm_conv3x3_forward_cl(xc, a, bias, y, act, B, cin, cout, H, W, 1, s)
    xr, wr = _np(x), _np(w32.to(torch.bfloat16))
    ref = CO.conv3x3(xr, wr, _np(bias))
    scale = np.abs(ref).max()
    assert np.abs(_np(y) - ref).max() <= 1e-5 * scale
    assert np.abs(_np(act)[..., :cout].transpose(0, 3, 1, 2) - np.maximum(_np(y), 0)).max() <= 2.0 ** -8 * scale
    assert (_np(act)[..., cout:] == 0).all()
    act2 = torch.empty_like(act)
    T.tlbm_conv3x3_forward_cl(xc, a, bias, None, act2, B, cin, cout, H, W, 1, s)
    assert torch.equal(act, act2)

    dy16 = _bf16(inputs.uniform_array(4, (B, cout, H, W), -1, 1)).cuda()
    dyc = _cl(T, dy16, s)
    rdx, rdw, _ = CO.conv3x3_backward(xr, wr, _np(dy16))
    ws = torch.empty(T.tlbm_conv3x3_cl_workspace_bytes(B, cin, cout, H, W), dtype=torch.uint8, device="cuda")
    g = torch.full_like(xc, 7.0)
    db = torch.empty(cin, dtype=torch.float32, device="cuda")
    T.tlbm_conv3x3_backward_data_cl(dyc, w32, xc, g, db, B, cin, cout, H, W, ws, s)
    rg = np.where(xr > 0, rdx, 0.0)
    gs = np.abs(rdx).max()
    assert np.abs(_np(g)[..., :cin].transpose(0, 3, 1, 2) - rg).max() <= (2.0 ** -8 + 1e-5) * gs
    assert (_np(g)[..., cin:] == 0).all()
    assert np.abs(_np(db) - rg.sum((0, 2, 3))).max() <= 1e-5 * max(gs, np.abs(rg).sum((0, 2, 3)).max())
    dw, dw2 = (torch.empty((cout, cin, 3, 3), dtype=torch.float32, device="cuda") for _ in range(2))
    for d in (dw, dw2):
        T.tlbm_conv3x3_backward_weight_cl(xc, dyc, d, B, cin, cout, H, W, ws, s)
    assert np.abs(_np(dw) - rdw).max() <= 1e-5 * max(np.abs(rdw).max(), 1.0)
    assert torch.equal(dw, dw2)
    dy32 = torch.tensor(inputs.uniform_array(6, (B, cout, H, W), -1, 1), dtype=torch.float32).cuda()
    dbo = torch.empty(cout, dtype=torch.float32, device="cuda")
    T.tlbm_conv3x3_bias_grad(dy32, dbo, B, cout, H, W, torch.empty(8192, dtype=torch.uint8, device="cuda"), s)
    assert np.abs(_np(dbo) - _np(dy32).sum((0, 2, 3))).max() <= 1e-5 * np.abs(_np(dy32)).sum((0, 2, 3)).max()
    assert T.tlbm_conv3x3_status() == 0


def test_channels_last_layers_at_the_training_batch(T):  # noqa: F811
    """48 x 65 x 65 at 32 channels (every CTA takes several tiles) against the
    NCHW kernels: the same tensor-core products in the same order give the same
    forward bits; the gradients differ by the order of their sums."""
    import torch

    B, C, H, W = 48, 32, 65, 65
    s = torch.cuda.current_stream()
    x = _bf16(inputs.uniform_array(11, (B, C, H, W), -1, 1)).cuda()
    w32 = torch.tensor(inputs.uniform_array(12, (C, C, 3, 3), -0.1, 0.1), dtype=torch.float32).cuda()
    bias = torch.tensor(inputs.uniform_array(13, (C,), -0.1, 0.1), dtype=torch.float32).cuda()
    dy32 = torch.tensor(inputs.uniform_array(14, (B, C, H, W), -1, 1), dtype=torch.float32).cuda()
    dy16 = dy32.to(torch.bfloat16)
    a = torch.empty(T.tlbm_conv3x3_weight_elems(C), dtype=torch.bfloat16, device="cuda")
    T.tlbm_conv3x3_pack_weights(w32, C, C, a, s)
    xc, dyc = _cl(T, x, s), _cl(T, dy16, s)
    y, yc = torch.empty_like(dy32), torch.empty_like(dy32)
    T.tlbm_conv3x3_forward(x, a, bias, y, None, B, C, C, H, W, 0, s)
    T.tlbm_conv3x3_forward_cl(xc, a, bias, yc, None, B, C, C, H, W, 0, s)
    assert torch.equal(y, yc)
    dx = torch.empty_like(y)
    at = torch.empty(32 * 288, dtype=torch.bfloat16, device="cuda")
    T.tlbm_conv3x3_backward_data(dy16, w32.to(torch.bfloat16), dx, B, C, C, H, W, at, s)
    ws = torch.empty(T.tlbm_conv3x3_cl_workspace_bytes(B, C, C, H, W), dtype=torch.uint8, device="cuda")
    g = torch.empty_like(xc)
    db = torch.empty(C, dtype=torch.float32, device="cuda")
    T.tlbm_conv3x3_backward_data_cl(dyc, w32, xc, g, db, B, C, C, H, W, ws, s)
    rg = torch.where(x > 0, dx, 0.0)
    assert torch.equal(g, rg.permute(0, 2, 3, 1).to(torch.bfloat16))
    assert (db.double() - rg.double().sum((0, 2, 3))).abs().max() <= 1e-6 * rg.double().abs().sum((0, 2, 3)).max()
    ws0 = torch.empty(T.tlbm_conv3x3_workspace_bytes(B, C, C, H, W), dtype=torch.uint8, device="cuda")
    dw, dwc = torch.empty_like(w32), torch.empty_like(w32)
    T.tlbm_conv3x3_backward_weight(x, dy16, None, dw, None, B, C, C, H, W, ws0, s)
    T.tlbm_conv3x3_backward_weight_cl(xc, dyc, dwc, B, C, C, H, W, ws, s)
    # random-sign products: sums of 2e5 of them, FP32 partials of about 1e3 each
    assert (dw - dwc).abs().max() <= 1e-5 * dw.abs().max()
    assert T.tlbm_conv3x3_status() == 0


def test_optimiser_step_of_all_layers_equals_the_single_ones(T):  # noqa: F811
    """tlbm_conv_adam_layers: tlbm_adam_step of every tensor (to the rounding of
    one contracted operation) and the packed operands of the new weights."""
    import torch

    s = torch.cuda.current_stream()
    layers, singles = [], []
    for k, (co, ci) in enumerate(((32, 5), (32, 32), (3, 32), (1, 1))):
        t = [torch.tensor(inputs.uniform_array(20 + 8 * k + i, sh, lo, 0.3), dtype=torch.float32).cuda()
             for i, (sh, lo) in enumerate([((co, ci, 3, 3), -0.3)] * 3 + [((co, ci, 3, 3), 1e-4)] +
                                          [((co,), -0.3)] * 3 + [((co,), 1e-4)])]
        a = torch.empty(T.tlbm_conv3x3_weight_elems(ci), dtype=torch.bfloat16, device="cuda")
        T.tlbm_conv3x3_pack_weights(t[0], co, ci, a, s)
        singles.append([q.clone() for q in t])
        layers.append((*t, a, co, ci))
    T.tlbm_conv_adam_layers(layers, 2e-3, 0.9, 0.999, 1e-8, 7, s)
    for q, t in zip(layers, singles):
        for o in (0, 4):
            T.tlbm_adam_step(t[o], t[o + 1], t[o + 2], t[o + 3], t[o].numel(), 2e-3, 0.9, 0.999, 1e-8, 7, s)
        for u, v in zip(q[:8], t):
            assert (u - v).abs().max() <= 2.0 ** -22 * v.abs().max()
        a = torch.empty_like(q[8])
        T.tlbm_conv3x3_pack_weights(q[0], q[9], q[10], a, s)
        assert torch.equal(a, q[8])


def test_channels_last_calls_refuse_what_they_cannot_run(T):  # noqa: F811
    import torch

    s = torch.cuda.current_stream()
    x = torch.zeros(1024, dtype=torch.bfloat16, device="cuda")
    ok = torch.zeros(4608, dtype=torch.bfloat16, device="cuda")
    y = torch.zeros(64, dtype=torch.float32, device="cuda")
    for call in (lambda: T.tlbm_conv3x3_forward_cl(x[1:], ok, None, y, None, 1, 16, 3, 2, 2, 0, s),  # alignment
                 lambda: T.tlbm_conv3x3_forward_cl(x, ok, None, None, None, 1, 16, 3, 2, 2, 0, s),   # no output
                 lambda: T.tlbm_conv3x3_forward_cl(x, ok, None, y, None, 1, 33, 3, 2, 2, 0, s),      # channels
                 lambda: T.tlbm_conv_adam_layers([], 1e-3, 0.9, 0.999, 1e-8, 1, s),
                 lambda: T.tlbm_conv3x3_backward_weight_cl(x, x, y, 1, 1, 1, 2, 2, torch.zeros(16, device="cuda"), s)):
        with pytest.raises(T.TlbmError):
            call()


def test_layers_of_other_widths_run_beside_each_other(T, tmp_path):  # noqa: F811
    """Host threads call the channels-last layers with widths that need unlike
    amounts of shared memory: every call is accepted, and the results are those
    of a thread alone."""
    import ctypes as C
    import os
    import subprocess

    import torch

    here = os.path.dirname(os.path.abspath(__file__))
    so = str(tmp_path / "conv_threads.so")
    subprocess.run(["gcc", "-O2", "-std=c11", "-shared", "-fPIC", "-pthread", os.path.join(here, "c", "conv_threads.c"),
                    "-o", so], check=True)
    helper = C.CDLL(so)
    ch, H, widths = 32, 5, (65, 126, 20)
    a = torch.zeros(T.tlbm_conv3x3_weight_elems(ch), dtype=torch.bfloat16, device="cuda")
    w = torch.tensor(inputs.uniform_array(11, (ch, ch, 3, 3), -0.3, 0.3), dtype=torch.float32).cuda()
    T.tlbm_conv3x3_pack_weights(w, ch, ch, a, torch.cuda.current_stream())
    lib = T.lib()
    fns = [C.cast(getattr(lib, f), C.c_void_p) for f in
           ("tlbm_conv3x3_forward_cl", "tlbm_conv3x3_backward_data_cl", "tlbm_conv3x3_backward_weight_cl")]
    per, results = [], {}
    for W in widths:
        x = _bf16(inputs.uniform_array(W, (1, H, W, ch), -1, 1)).cuda()
        per.append([x, torch.empty_like(x), torch.empty_like(x), torch.empty_like(w), torch.empty(ch, device="cuda"),
                    torch.empty(T.tlbm_conv3x3_cl_workspace_bytes(1, ch, ch, H, W), dtype=torch.uint8, device="cuda"),
                    torch.cuda.Stream()])
    torch.cuda.synchronize()
    for calls in (1, 20000):
        for group in ([[k] for k in range(len(widths))] if calls == 1 else [range(len(widths))]):
            n = len(group)
            ptrs = (C.c_void_p * (7 * n))(*[(t.cuda_stream if i == 6 else t.data_ptr())
                                            for k in group for i, t in enumerate(per[k])])
            ws = (C.c_size_t * n)(*[per[k][5].numel() for k in group])
            wid = (C.c_int * n)(*[widths[k] for k in group])
            refused = helper.conv_threads(*fns, C.c_void_p(a.data_ptr()), C.c_void_p(w.data_ptr()), ch, H, n, wid, ptrs,
                                          ws, calls)
            torch.cuda.synchronize()
            assert refused == 0, (calls, refused)
        results[calls] = [[t.clone() for t in q[1:5]] for q in per]
    for W, p, q in zip(widths, results[1], results[20000]):
        assert all(torch.equal(u, v) for u, v in zip(p, q)), W

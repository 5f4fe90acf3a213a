"""The packed network kernels where their tiles end: x extents below, at and beyond the 16-voxel steps and the 64-voxel
chunks of the weight gradient, planes smaller than a 128-voxel tile, channel counts that do not fill 32, inputs of two
parts, single planes; against the FP64 reference with the same BF16 operand rounding (products are then exact and only
the FP32 accumulation differs: 1e-5 relative, as for the unpacked kernels) or exactly."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import nn_reference as ref
from paper_1712_01132_gb300 import dvm

pytestmark = pytest.mark.gpu


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _dev(a):
    return torch.tensor(np.asarray(a, dtype=np.float32), device="cuda")


def _rel(a, b):
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-30))


def _r32(c):
    return (c + 31) // 32 * 32


def _unpacked(xp, c, dims):
    """Channels-first interior of a packed tensor, after checking that its halo is the periodic image."""
    v = xp.float().cpu().numpy().transpose(3, 0, 1, 2)
    inner = v[:, 1:-1, 1:-1, 1:-1]
    assert np.array_equal(v, np.pad(inner, ((0, 0), (1, 1), (1, 1), (1, 1)), mode="wrap"))
    assert not inner[c:].any()
    return inner[:c]


@pytest.mark.parametrize("c0,c1,cout,dims", [(3, 0, 5, (3, 2, 17)), (8, 16, 8, (6, 10, 22)), (40, 0, 70, (2, 4, 16)),
                                             (3, 6, 3, (4, 6, 70)), (8, 16, 33, (4, 8, 128)), (16, 32, 96, (2, 2, 80)),
                                             (32, 0, 160, (4, 8, 8)), (100, 0, 32, (2, 3, 32)), (64, 0, 64, (1, 8, 16)),
                                             (32, 64, 32, (6, 8, 64)), (5, 0, 4, (2, 2, 2)),
                                             (4, 0, 4, (76, 64, 128))])        # (four row tiles a CTA)
def test_convolution_and_gradients(c0, c1, cout, dims):
    lib = dvm.load()
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    d, h, w = dims
    c0p = c0 if c0 % 8 == 0 else _r32(c0)                # where an input's second part begins
    cin, cinp, coutp = c0 + c1, _r32(c0p + c1), _r32(cout)
    rng = np.random.default_rng(cin * 100 + cout)
    x = rng.standard_normal((cin,) + dims).astype(np.float32)
    wt = (rng.standard_normal((cout, cin, 27)) / np.sqrt(cin * 27)).astype(np.float32)
    b = rng.standard_normal(cout).astype(np.float32)
    g = rng.standard_normal((cout,) + dims).astype(np.float32)
    packed = lambda c: torch.full((d + 2, h + 2, w + 2, c), float("nan"), dtype=torch.bfloat16, device="cuda")
    xp = packed(_r32(c0))
    xo = torch.empty(1 + x[:c0].size, device="cuda")[1:]             # any FP32 alignment
    xo.copy_(_dev(x[:c0]).ravel())
    assert lib.dvm_nn_pack(_p(xo), _p(xp), c0, _r32(c0), d, h, w, 0, st) == 0
    assert np.array_equal(_unpacked(xp, c0, dims), ref.round_bf16(x[:c0]))
    if c1:
        x2 = packed(_r32(c1))
        assert lib.dvm_nn_pack(_p(_dev(x[c0:])), _p(x2), c1, _r32(c1), d, h, w, 0, st) == 0
        pad = torch.zeros((d + 2, h + 2, w + 2, cinp - c0p - c1), dtype=torch.bfloat16, device="cuda")
        xp = torch.cat([xp[..., :c0p], x2[..., :c1], pad], 3).contiguous()
    wd, bd = _dev(wt), _dev(b)
    wb = torch.empty(lib.dvm_nn_packed_weight_elems(cin, cout, c0), dtype=torch.bfloat16, device="cuda")
    one = lambda v: (ctypes.c_int * 1)(v)
    args = (1, (ctypes.c_void_p * 1)(wd.data_ptr()), (ctypes.c_void_p * 1)(wb.data_ptr()), one(cin), one(cout), one(c0))
    assert lib.dvm_nn_pack_weights(*args, 0, st) == 0
    y, yp = torch.empty((cout,) + dims, device="cuda"), packed(coutp + 32)
    assert lib.dvm_nn_conv3d_packed(_p(xp), _p(wb), _p(bd), _p(y), _p(yp), coutp + 32, 32, cinp, cout, d, h, w, 1, st) == 0
    assert lib.dvm_nn_status(st) == 0
    xr, wr = ref.round_bf16(x), ref.round_bf16(wt)
    ry = np.maximum(ref.conv3d(xr, wr, b.astype(np.float64)), 0.0)
    assert _rel(y.cpu().numpy(), ry) < 1e-5
    assert np.array_equal(_unpacked(yp[..., 32:].contiguous(), cout, dims), ref.round_bf16(y.cpu().numpy()))
    assert bool(torch.isnan(yp[..., :32]).all())                    # the other part of a concatenation is left alone
    # gradients behind the ReLU of y
    gp, gw = packed(coutp), torch.full((d, h, (w + 15) // 16 * 16, coutp), float("nan"), dtype=torch.bfloat16, device="cuda")
    gf = _dev(g)                                                    # masked in place
    db = torch.full((cout,), 0.25, device="cuda")
    assert lib.dvm_nn_grad_pack(_p(gf), None, 0, _p(yp), coutp + 32, 32, _p(gp), _p(gw), _p(gf), _p(db), cout, d, h, w, st) == 0
    gm = g * (y.cpu().numpy() > 0)
    gr = ref.round_bf16(gm)
    assert np.array_equal(gf.cpu().numpy(), gm)
    assert np.array_equal(_unpacked(gp, cout, dims), gr)
    gwh = gw.float().cpu().numpy().transpose(3, 0, 1, 2)
    assert np.array_equal(gwh[:cout, :, :, :w], gr) and not gwh[:, :, :, w:].any() and not gwh[cout:].any()
    rdw, _ = ref.conv3d_wgrad(xr, gr)
    _, rdb = ref.conv3d_wgrad(x.astype(np.float64), gm.astype(np.float64))
    assert _rel(db.cpu().numpy(), rdb + 0.25) < 1e-5
    dw = torch.full((cout, cin, 27), 0.5, device="cuda")
    n = lib.dvm_nn_wgrad_packed_scratch_floats(cin, c0, cout, d, h, w)
    sc = torch.empty(n, device="cuda")
    assert lib.dvm_nn_conv3d_wgrad_packed(_p(xp), _p(gw), _p(dw), _p(sc), n, cin, c0, cout, d, h, w, st) == 0
    assert lib.dvm_nn_conv3d_wgrad_packed(_p(xp), _p(gw), _p(dw), _p(sc), 16, cin, c0, cout, d, h, w, st) != 0   # too small
    assert lib.dvm_nn_pack_weights(*args, 1, st) == 0
    dx = torch.empty((cin,) + dims, device="cuda")
    assert lib.dvm_nn_conv3d_packed(_p(gp), _p(wb), None, _p(dx), None, 0, 0, coutp, cin, d, h, w, 0, st) == 0
    assert lib.dvm_nn_status(st) == 0
    assert _rel(dw.cpu().numpy(), rdw + 0.5) < 1e-5
    assert _rel(dx.cpu().numpy(), ref.conv3d_dgrad(gr, wr)) < 1e-5
    # the unpacked functions sum in the same order (channels at their own places, the weight gradient's pieces of 32
    # voxels along x in the same splits)
    u = torch.empty(lib.dvm_nn_conv3d_scratch_bytes(cin, cout, d, h, w), dtype=torch.uint8, device="cuda")
    if c1 == 0 or c0 % 8 == 0:
        y1 = torch.empty_like(y)
        assert lib.dvm_nn_conv3d(_p(_dev(x)), _p(wd), _p(bd), _p(y1), cin, cout, d, h, w, 0, _p(u), u.numel(), st) == 0
        assert torch.equal(torch.relu(y1), y)
    if w <= 64 or w > 96:
        nu = lib.dvm_nn_wgrad_scratch_floats(cin, cout, d, h, w)
        su = torch.empty(nu, device="cuda")
        dw1, db1 = torch.full_like(dw, 0.5), torch.full_like(db, 0.25)
        assert lib.dvm_nn_conv3d_wgrad(_p(_dev(x)), _p(gf), _p(dw1), _p(db1), _p(su), nu, cin, cout, d, h, w, 1, st) == 0
        assert torch.equal(dw1, dw) and torch.equal(db1, db)


@pytest.mark.parametrize("c,dims", [(3, (2, 4, 6)), (40, (4, 2, 34)), (32, (2, 2, 64))])
def test_resampling(c, dims):
    lib = dvm.load()
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    d, h, w = dims
    low = tuple(n // 2 for n in dims)
    cp = _r32(c)
    rng = np.random.default_rng(c)
    x, g = rng.standard_normal((c,) + dims).astype(np.float32), rng.standard_normal((c,) + low).astype(np.float32)
    lp = torch.full((low[0] + 2, low[1] + 2, low[2] + 2, cp), float("nan"), dtype=torch.bfloat16, device="cuda")
    assert lib.dvm_nn_pack(_p(_dev(x)), _p(lp), c, cp, *low, 1, st) == 0
    mean = torch.empty((c,) + low, device="cuda")
    assert lib.dvm_nn_pool2(_p(_dev(x)), _p(mean), c, *dims, st) == 0
    assert np.array_equal(_unpacked(lp, c, low), ref.round_bf16(mean.cpu().numpy()))
    xp = torch.zeros((d + 2, h + 2, w + 2, cp + 32), dtype=torch.bfloat16, device="cuda")
    assert lib.dvm_nn_up2_packed(_p(lp), cp, _p(xp), cp + 32, 32, cp, *dims, st) == 0
    assert np.array_equal(_unpacked(xp[..., 32:].contiguous(), c, dims), ref.up2(_unpacked(lp, c, low)))
    # the gradients' two other sources: a skip with the pooling's gradient, the sum over upsampled children
    for mode, src, lo, out, expect in ((1, x, g, dims, x + ref.pool2_bwd(g.astype(np.float64))), (2, x, None, low, ref.up2_bwd(x.astype(np.float64)))):
        gw = torch.empty((out[0], out[1], (out[2] + 15) // 16 * 16, cp), dtype=torch.bfloat16, device="cuda")
        gf, db = torch.empty((c,) + out, device="cuda"), torch.zeros(c, device="cuda")
        assert lib.dvm_nn_grad_pack(_p(_dev(src)), _p(_dev(lo)) if lo is not None else None, mode, None, 0, 0, None, _p(gw), _p(gf),
                                    _p(db), c, *out, st) == 0
        got = gw.float().cpu().numpy().transpose(3, 0, 1, 2)[:c, :, :, :out[2]]
        assert np.abs(got - expect).max() <= 2.0 ** -8 * np.abs(expect).max()          # one BF16 rounding
        assert _rel(db.cpu().numpy(), expect.sum((1, 2, 3))) < 1e-5

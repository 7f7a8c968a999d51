"""The convolution layer where its tiles are shared: through the public calls, which pick the
CTAs of a tile from the shape; and each of the three passes with every number of CTAs forced:
one, clusters of 2, 4 and 8 on one tile, and pairs of CTAs on 256 x 256 tiles, on shapes whose
rows and columns do not fill a tile, with an odd number of pixel tiles (the last pair's second
one lies past the images), and with fewer reduction blocks than CTAs.  Outputs that are 16- but
not 32-byte aligned too.  Same oracle and tolerance as tests/test_gpu_conv.py."""
import ctypes

import numpy as np
import pytest

from gen import conv as gc
from oracle import conv as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2608_24204_gb300 import wici  # noqa: E402
from tests.test_gpu_conv import _close, _dev, _f32  # noqa: E402


@pytest.mark.parametrize("shape,offset", [
    (gc.ConvShape(n=1, c=256, h=4, w=4, k=256), 0),        # two by two outputs
    (gc.ConvShape(n=1, c=256, h=18, w=34, k=256), 0),      # tiles of one row and one column
    (gc.ConvShape(n=2, c=256, h=28, w=52, k=512), 16),
    (gc.ConvShape(n=1, c=512, h=40, w=96, k=512), 0),
    (gc.ConvShape(n=4, c=256, h=64, w=64, k=1024), 16),
    (gc.ConvShape(n=3, c=256, h=80, w=96, k=1024), 0),     # 45 pixel tiles
])
def test_conv_layer_on_clusters(shape, offset):
    x, w, dy = gc.make_conv_inputs(shape)
    s = wici.wici_conv_shape(shape.n, shape.c, shape.h, shape.w, shape.k)
    ws = torch.zeros(wici.wici_conv_workspace_bytes(s), dtype=torch.uint8, device="cuda")
    xd, wd, dyd = _dev(x), _dev(w), _dev(dy)

    def out(dims):   # NaN-filled, `offset` bytes past an aligned address
        n = int(np.prod(dims))
        return torch.full((n + 16,), float("nan"), device="cuda")[offset // 4:offset // 4 + n].view(dims)

    y, dx = out((shape.n, shape.p, shape.q, shape.k)), out((shape.n, shape.h, shape.w, shape.c))
    dw = out((shape.k, 3, 3, shape.c))
    st = torch.cuda.current_stream().cuda_stream
    wici.wici_conv_forward(st, s, xd.data_ptr(), wd.data_ptr(), y.data_ptr(), ws.data_ptr())
    wici.wici_conv_backward_data(st, s, dyd.data_ptr(), wd.data_ptr(), dx.data_ptr(), ws.data_ptr())
    wici.wici_conv_backward_filter(st, s, xd.data_ptr(), dyd.data_ptr(), dw.data_ptr(), ws.data_ptr())
    wici.wici_conv_status(st, ws.data_ptr())
    xf, wf, dyf = _f32(x), _f32(w), _f32(dy)
    _close(y.cpu().numpy(), C.conv_forward(xf, wf), C.abs_sum_bound(C.conv_forward, xf, wf), "forward")
    _close(dx.cpu().numpy(), C.conv_backward_data(dyf, wf, shape.h, shape.w),
           C.abs_sum_bound(C.conv_backward_data, dyf, wf, shape.h, shape.w), "data gradient")
    _close(dw.cpu().numpy(), C.conv_backward_filter(xf, dyf), C.abs_sum_bound(C.conv_backward_filter, xf, dyf),
           "filter gradient")


FORCED = [
    (gc.ConvShape(n=1, c=256, h=18, w=34, k=256), 0),      # tiles of one row and one column; 4 pixel tiles
    (gc.ConvShape(n=3, c=256, h=14, w=44, k=512), 16),     # 3 x 1 x 2 pixel tiles, ragged both ways
    (gc.ConvShape(n=1, c=512, h=40, w=24, k=256), 0),      # 3 pixel tiles: a pair without its second
    (gc.ConvShape(n=1, c=256, h=4, w=4, k=256), 0),        # filter gradient: one reduction block for 8 CTAs
]


@pytest.fixture(scope="module", params=FORCED, ids=lambda p: f"{p[0].n}x{p[0].c}x{p[0].h}x{p[0].w}x{p[0].k}")
def layer(request):
    shape, offset = request.param
    x, w, dy = gc.make_conv_inputs(shape)
    xf, wf, dyf = _f32(x), _f32(w), _f32(dy)
    passes = [
        (_dev(x), _dev(w), (shape.n, shape.p, shape.q, shape.k), C.conv_forward(xf, wf),
         C.abs_sum_bound(C.conv_forward, xf, wf)),
        (_dev(dy), _dev(w), (shape.n, shape.h, shape.w, shape.c), C.conv_backward_data(dyf, wf, shape.h, shape.w),
         C.abs_sum_bound(C.conv_backward_data, dyf, wf, shape.h, shape.w)),
        (_dev(x), _dev(dy), (shape.k, 3, 3, shape.c), C.conv_backward_filter(xf, dyf),
         C.abs_sum_bound(C.conv_backward_filter, xf, dyf)),
    ]
    return shape, offset, passes


@pytest.mark.parametrize("ctas", [0, 1, 2, 4, 8])
@pytest.mark.parametrize("mode", [0, 1, 2], ids=["forward", "data gradient", "filter gradient"])
def test_conv_pass_with_the_ctas_of_a_tile_forced(layer, mode, ctas):
    shape, offset, passes = layer
    a, b, dims, want, bound = passes[mode]
    s = wici.wici_conv_shape(shape.n, shape.c, shape.h, shape.w, shape.k)
    ws = torch.zeros(wici.wici_conv_workspace_bytes(s), dtype=torch.uint8, device="cuda")
    n = int(np.prod(dims))
    out = torch.full((n + 16,), float("nan"), device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    vp = ctypes.c_void_p
    rc = wici.lib().wici_internal_conv(mode, ctas, vp(st), ctypes.byref(s), vp(a.data_ptr()), vp(b.data_ptr()),
                                       vp(out.data_ptr() + offset), vp(ws.data_ptr()))
    assert rc == wici.WICI_OK, wici.wici_last_error(None)
    wici.wici_conv_status(st, ws.data_ptr())
    got = out[offset // 4:offset // 4 + n].view(dims).cpu().numpy()
    _close(got, want, bound, f"{ctas} CTAs")
    assert torch.isnan(out[:offset // 4]).all() and torch.isnan(out[offset // 4 + n:]).all()   # nothing past the output

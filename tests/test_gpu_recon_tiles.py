"""The 3x3 layers at the sizes where their tiles end: images whose 128-position
row groups fill the SMs' rounds exactly, leave one over or fall short, channel
counts that take each tile width, against an fp32 convolution of the same bf16
values (one bf16 rounding plus the fp32 summation-order bound, as the existing
layer test)."""
import pytest

from paper_2601_19901_gb300 import lfdpr

pytestmark = pytest.mark.gpu

# (input channels, output channels, rows, columns)
SHAPES = [(32, 32, 1, 1), (16, 32, 150, 126), (32, 32, 151, 126), (32, 32, 302, 126), (32, 64, 150, 126),
          (32, 64, 153, 126), (48, 32, 610, 126), (16, 96, 40, 60), (32, 160, 33, 47), (16, 128, 303, 126),
          (32, 256, 31, 30), (16, 256, 200, 126), (16, 32, 20, 1300), (16, 64, 9, 1300), (16, 128, 5, 1000)]


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available()
    torch.backends.cudnn.allow_tf32 = False
    torch.backends.cuda.matmul.allow_tf32 = False
    from paper_2601_19901_gb300 import build
    build.build()
    return torch


@pytest.mark.parametrize("cin,cout,h,w", SHAPES)
def test_conv3x3_tiles(torch, cin, cout, h, w):
    g = torch.Generator(device="cpu").manual_seed(cin + cout * 7 + h * 31 + w)
    x = torch.randn((h, w, cin), generator=g).to(torch.bfloat16).cuda()
    wt = (torch.randn((cout, 3, 3, cin), generator=g) * (2.0 / (9 * cin)) ** 0.5).to(torch.bfloat16).cuda()
    b = (torch.randn((cout,), generator=g) * 0.1).float().cuda()
    out = torch.full((h, w, cout), 7.0, dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    lfdpr.lfdpr_conv3x3_bf16(x.data_ptr(), h, w, cin, wt.data_ptr(), b.data_ptr(), out.data_ptr(), cout,
                             status.data_ptr())
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    xf, wf = x.float().permute(2, 0, 1)[None], wt.float().permute(0, 3, 1, 2)
    conv = torch.nn.functional.conv2d
    ref = conv(xf, wf, b, padding=1)[0].permute(1, 2, 0).relu()
    mag = conv(xf.abs(), wf.abs(), b.abs(), padding=1)[0].permute(1, 2, 0)
    tol = ref.abs() * 2.0 ** -8 + mag * (9 * cin) * 2.0 ** -24
    err = (out.float() - ref).abs()
    assert torch.all(err <= tol), float((err - tol).max())


def test_widths_beyond_two_stages_are_refused(torch):
    """Real buffers: a call that were accepted would be an ordinary one."""
    for cout, h, w in ((64, 9, 2600), (128, 5, 1300)):
        x = torch.zeros((h, w, 16), dtype=torch.bfloat16, device="cuda")
        wt = torch.zeros((cout, 3, 3, 16), dtype=torch.bfloat16, device="cuda")
        b = torch.zeros(cout, device="cuda")
        out = torch.zeros((h, w, cout), dtype=torch.bfloat16, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        with pytest.raises(lfdpr.LfdprError) as e:
            lfdpr.lfdpr_conv3x3_bf16(x.data_ptr(), h, w, 16, wt.data_ptr(), b.data_ptr(), out.data_ptr(), cout,
                                     status.data_ptr())
        assert e.value.status == lfdpr.EINVAL

"""Export of a matrix to a destination on each alignment, with even and odd row lengths, to device and to pinned host
memory: the same bytes as the padded matrix holds."""

import ctypes

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402


@pytest.mark.parametrize("which", ["T_A", "LPLUS"])
@pytest.mark.parametrize("cut,offset,host", [(0, 0, False), (1, 0, False), (0, 4, False), (1, 8, False), (0, 1, False),
                                             (1, 0, True)])
def test_export(which, cut, offset, host):
    from paper_1803_08333_gb300 import build

    build.build()
    m = synth.geodesic_sphere(11)  # rows of more than one pass of a thread block: 3630 and 2420 entries
    op = rf.Operator(rf.Context(0), m.verts, m.tris[: len(m.tris) - cut], 1.0, scaling="k")
    want = op.export(which)
    n = want.shape[0]
    buf = torch.zeros(n * n * 8 + 16, dtype=torch.uint8, device="cpu" if host else "cuda", pin_memory=host)
    rf._check(rf.lib().rfcmp_op_export(op._h, rf.EXPORT[which], ctypes.c_void_p(buf.data_ptr() + offset), n * n * 8,
                                       rf._stream()))
    torch.cuda.synchronize()
    got = buf[offset : offset + n * n * 8].clone().cuda()
    assert torch.count_nonzero(buf[offset + n * n * 8 :]) == 0
    if which == "T_A":
        assert torch.equal(got.view(torch.complex64).view(n, n), want)
        x = torch.randn(n, dtype=torch.complex128, device="cuda")
        y = op.apply("T_A", x)[0]
        assert torch.linalg.norm(want.to(torch.complex128) @ x - y) <= 1e-11 * torch.linalg.norm(y)
    else:
        hi, lo = got.view(torch.float32).view(2, n, n).double()
        assert torch.equal(hi + lo, want)
        assert torch.equal(want, want.T)

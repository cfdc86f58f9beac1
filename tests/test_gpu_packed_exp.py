"""The exponential of the decision chain in packed form, which decides every alpha, equals the scalar form that the
oracle restates, bit for bit: at every float of [-80, 0] (the short form's range), and at a sample of all arguments."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def exps(x):
    from paper_2605_10760_gb300 import raster as R
    lib, y = R.L.load(), [torch.empty_like(x) for _ in range(3)]
    ptr = lambda t: C.c_void_p(t.data_ptr())
    assert lib.gs_debug_expf(ptr(x), ptr(y[0]), None, x.numel(), R._stream()) == 0
    assert lib.gs_debug_exp2(ptr(x), ptr(y[1]), ptr(y[2]), x.numel(), R._stream()) == 0
    return [t.view(torch.int32) for t in y]


def test_every_float_up_to_80():
    end, step, bad = int(np.float32(80).view(np.int32)) + 1, 1 << 27, [0, 0]
    for a in range(0, end, step):
        x = -(torch.arange(a, min(end, a + step), dtype=torch.int32, device="cuda").view(torch.float32))
        scalar, packed, neg = exps(x)
        bad[0] += int((packed != scalar).sum())
        bad[1] += int((neg != scalar).sum())
    assert bad == [0, 0]


def test_any_argument():
    bits = torch.randint(-(1 << 31), (1 << 31) - 1, (1 << 22,), dtype=torch.int64, generator=torch.Generator().manual_seed(1))
    x = bits.to(torch.int32).view(torch.float32).cuda()
    x = torch.cat([x, torch.linspace(-90, 90, 1 << 20, device="cuda"), torch.tensor([0.0, -0.0, 88.0, -87.0, 1e-40], device="cuda")])
    scalar, packed, _ = exps(x)
    assert torch.equal(packed, scalar)

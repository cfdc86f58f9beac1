"""The Adam step goes over groups of scalars four at a time where N and the addresses allow it, one at a time
elsewhere, and over whole Gaussians where the isotropy regulariser needs them: against FP64 at counts around the
warps' shares, both alignments."""
import numpy as np
import pytest
import torch

from oracle import losses as OL

pytestmark = pytest.mark.gpu
DIMS = {"means": 3, "log_scales": 3, "quats": 4, "opacities": 1, "colors": 3}
LR = (1.6e-4, 5e-3, 1e-3, 5e-2, 2.5e-3)


def _at(x, shift):
    """x at an address `shift` floats beyond a 16-byte boundary."""
    buf = torch.empty(x.size + 8, device="cuda")
    t = buf[shift:shift + x.size].view(*x.shape)
    t.copy_(torch.from_numpy(x))
    return t


@pytest.mark.parametrize("n", [1, 3, 4, 31, 33, 124, 128, 132, 1023, 1028])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("iso,zero", [(0.0, True), (10.0, False)])
def test_matches_oracle_at_every_layout(n, shift, iso, zero):
    from paper_2605_10760_gb300 import raster as R
    rng = np.random.default_rng(n)
    shape = {k: (n, d) if d > 1 else (n,) for k, d in DIMS.items()}
    par = {k: rng.normal(0, 0.5, shape[k]).astype(np.float32) for k in DIMS}
    par["opacities"] = rng.uniform(0.1, 0.9, n).astype(np.float32)
    g = R.Gaussians(*[_at(par[k], shift) for k in DIMS])
    st = R.AdamState(g, lr=LR)
    ref = {k: v.astype(np.float64) for k, v in par.items()}
    ref["opacities"] = st.logits.cpu().numpy().astype(np.float64)
    mom = {k: (np.zeros(shape[k]), np.zeros(shape[k])) for k in DIMS}
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    for step in (1, 2):
        grad = {k: rng.normal(0, 1, shape[k]).astype(np.float32) for k in DIMS}
        gg = R.Gaussians(*[_at(grad[k], shift) for k in DIMS])
        st.apply(gg, zero_grads=zero, iso_weight=iso, iso_loss=loss if iso else None)
        for k, lr in zip(DIMS, LR):
            gk = grad[k].astype(np.float64)
            if k == "opacities":
                o = 1 / (1 + np.exp(-ref[k]))
                gk = gk * o * (1 - o)
            if k == "log_scales" and iso:
                val, giso = OL.iso_loss(ref[k], iso)
                assert abs(loss.item() - val) <= 1e-5 * abs(val)
                gk = gk + giso
            ref[k], m, v = OL.adam_step(ref[k], gk, *mom[k], step, lr)
            mom[k] = (m, v)
            left = getattr(gg, k).cpu().numpy()
            assert not left.any() if zero else np.array_equal(left, grad[k])
    for k in ("means", "log_scales", "quats", "colors"):
        np.testing.assert_allclose(getattr(g, k).cpu().numpy(), ref[k], rtol=1e-5, atol=2e-6)
    np.testing.assert_allclose(st.logits.cpu().numpy(), ref["opacities"], rtol=1e-5, atol=1e-5)
    np.testing.assert_allclose(g.opacities.cpu().numpy(), 1 / (1 + np.exp(-ref["opacities"])), rtol=1e-5, atol=1e-6)
    assert int(st.step.item()) == 2

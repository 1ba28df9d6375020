"""The fused training pass (loss and gradient) at the edges of its tiling, against the oracle's
BF16 reading: two 64-sample tiles; two tiles more than the 152 CTAs of a launch; several tiles
per CTA with a ragged last round. Bounds as for one batch in test_gpu_siren.py (FP32 summation
order and the BF16 rounding flips it causes). The last case has first-layer arguments on both
sides of the fast sine's range (|z| <= 30000): there FP32 itself leaves z uncertain by three
roundings of 2^-24 |z|, 7e-3 rad at 4e4, in every h1, so the gradient is held to 5e-2 (an
argument sent through the wrong reduction would leave nothing of it)."""
import numpy as np
import pytest

from oracle import siren
from paper_2403_06706_gb300 import synth

pytestmark = pytest.mark.gpu
gcpush = pytest.importorskip("paper_2403_06706_gb300.gcpush")
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,omega0,tol", [(128, 30.0, 2e-3), (154 * 64, 30.0, 2e-3), (458 * 64, 30.0, 2e-3),
                                          (1024, 4.0e4, 5e-2)])
def test_gradient_at_tile_edges(n, omega0, tol):
    rng = np.random.default_rng(n)
    p = synth.siren_init(seed=n)
    x = rng.uniform(-0.6, 0.6, (n, 3)).astype(np.float32)
    t = (rng.normal(size=(n, 8)) * 0.3).astype(np.float32)
    with gcpush.Context() as c:
        c.siren_set(p, omega0=omega0)
        g = torch.full((gcpush.SIREN_NPARAMS,), float("nan"), device="cuda")
        loss = c.siren_loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), g)
        again = c.siren_loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), None)
    Lo, go = siren.loss_and_grad(p.astype(np.float64), x.astype(np.float64), t.astype(np.float64), omega0, bf16=True)
    g = siren.unpack(g.cpu().numpy().astype(np.float64))
    go = siren.unpack(go)
    assert abs(loss - Lo) < tol / 20 * Lo
    assert abs(loss - again) < 1e-12 * Lo  # FP64 atomics in another order
    for k in go:
        err = np.linalg.norm(g[k] - go[k]) / np.linalg.norm(go[k])
        print(k, err)
        assert err < 5 * tol, k

"""The fused training pass (loss and gradient) at the edges of its tiling, against the oracle's
BF16 reading: two 64-sample tiles; two tiles more than the 152 CTAs of a launch; several tiles
per CTA with a ragged last round; the last batch that takes the library's sines and the first
that takes the fast ones. Bounds as for one batch in test_gpu_siren.py (FP32 summation
order and the BF16 rounding flips it causes). The cases at omega0 = 4e4 have first-layer
arguments on both sides of the fast sine's range (|z| <= 30000): there FP32 itself leaves z
uncertain by three
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
                                          (1024, 4.0e4, 5e-2), (16384, 30.0, 2e-3), (16512, 30.0, 2e-3),
                                          (16512, 4.0e4, 5e-2)])
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


def test_targets_are_the_rounded_interpolant():
    """Training targets from an FP32 grid (pairs of floats; FP64 where those end) against the
    FP64 interpolant: within a float's rounding (2^-24) of each value, plus 1e-10 of the
    channel's scale for index coordinates that agree to 1e-11. Points inside, across the cell
    faces, at the poles and on the axis, at phi = 0, outside the shell on both sides, and so
    near the origin that pairs would underflow; scales at both ends of what pairs hold."""
    w = synth.WindSpec(33, 17, 21, eps=0.1, n_modes=4, phi1_v=100.0)
    nodes = synth.wind_grid(w, dtype=np.float32)
    rng = np.random.default_rng(3)
    x = rng.normal(size=(20000, 3))
    x *= (rng.uniform(0.02, 1.2, (len(x), 1)) / np.linalg.norm(x, axis=1, keepdims=True))
    r = (w.r_min_au + w.dr_au * rng.integers(0, w.n_r, 4000)) / w.r_max_au
    th = np.pi * rng.integers(0, w.n_th, 4000) / (w.n_th - 1)
    ph = 2 * np.pi * rng.integers(0, w.n_ph, 4000) / w.n_ph
    node = np.stack([r * np.sin(th) * np.cos(ph), r * np.sin(th) * np.sin(ph), r * np.cos(th)], 1)
    special = np.array([[0, 0, 0.5], [0, 0, -0.5], [0.5, 0, 0], [-0.5, 0, 0], [0.5, -0.0, 0.1], [1e-15, 0, 0.4],
                        [1e-30, 1e-30, 1e-30], [0.3, -1e-20, 0.2], [3, 2, 1], [1e-3, 1e-3, 1e-3]])
    x = np.concatenate([x, node, special]).astype(np.float32)
    for B_s, E_s in ((3.5e-9, 1.4e-3), (1e-25, 1.4e-3), (3.5e-9, 1e22)):
        with gcpush.Context() as c:
            c.field_load(nodes, w.r_min_au, w.r_max_au)
            c.siren_set(synth.siren_init(0), r_max_au=w.r_max_au, B_scale=B_s, E_scale=E_s)
            t = torch.full((len(x), 8), float("nan"), device="cuda")
            c.field_targets(torch.from_numpy(x).cuda(), t)
            odd = torch.full((8 * len(x) + 1,), float("nan"), device="cuda")  # output at 4-byte alignment
            c.field_targets(torch.from_numpy(x).cuda(), odd[1:].view(-1, 8))
        t = t.cpu().numpy()
        assert np.array_equal(t, odd[1:].cpu().numpy().reshape(-1, 8))
        to = siren.grid_targets(nodes.astype(np.float64), w.r_min_au * siren.AU, w.r_max_au * siren.AU,
                                x.astype(np.float64), w.r_max_au * siren.AU, B_s, E_s)
        scale = np.sqrt((to * to).mean(0))
        err = np.abs(t - to) / (2.0**-24 * np.abs(to) * 1.0001 + 1e-10 * scale + 1e-45)
        print(err.max(0))
        assert err.max() <= 1.0


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_targets_of_points_that_are_no_numbers(dtype):
    """A NaN coordinate gives NaN targets (the potential's may stay a number where only z is
    one) and reads inside the grid; infinities are beyond the shell. The points beside them
    have the targets that they have alone."""
    w = synth.WindSpec(17, 9, 12, eps=0.1, n_modes=2, phi1_v=100.0)
    x = np.random.default_rng(1).uniform(-0.5, 0.5, (300, 3)).astype(np.float32)
    nan, inf = np.nan, np.inf
    x[100:109] = [[nan, 0.3, 0.2], [0.3, nan, 0.2], [0.3, 0.2, nan], [nan, nan, 0.1], [nan, nan, nan],
                  [inf, nan, 0.1], [inf, 0.1, 0.1], [-inf, -inf, inf], [nan, 0.0, -inf]]
    good = np.r_[:100, 109:300]
    with gcpush.Context(precision=gcpush.PREC_FP64 if dtype == np.float64 else gcpush.PREC_FP32_MIXED) as c:
        c.field_load(synth.wind_grid(w, dtype=dtype), w.r_min_au, w.r_max_au)
        c.siren_set(synth.siren_init(0), r_max_au=w.r_max_au, B_scale=w.B1, E_scale=w.B1 * w.u_sw)
        t = torch.zeros((300, 8), device="cuda")
        c.field_targets(torch.from_numpy(x).cuda(), t)
        alone = torch.zeros((len(good), 8), device="cuda")
        c.field_targets(torch.from_numpy(x[good]).cuda(), alone)
    t, alone = t.cpu().numpy(), alone.cpu().numpy()
    assert np.isnan(t[100:106, :7]).all() and np.isnan(t[108, :7]).all()
    assert np.isnan(t[[100, 101, 103, 104, 105, 108], 7]).all()
    assert np.isfinite(alone).all() and np.array_equal(t[good], alone)


@pytest.mark.parametrize("off", [1, 2, 3])
def test_gradient_into_a_slice_of_a_flat_buffer(off):
    """A gradient buffer at 4-byte alignment gets the aligned one's gradient and nothing beside
    it is written. The two differ by the order of FP32 atomics alone: up to two tiles x four
    row groups are added per parameter, 7 roundings of at most 2^-24 of the terms' sum, held to
    1e-5 of the gradient's norm."""
    n = 128
    rng = np.random.default_rng(off)
    x = torch.from_numpy(rng.uniform(-0.6, 0.6, (n, 3)).astype(np.float32)).cuda()
    t = torch.from_numpy((rng.normal(size=(n, 8)) * 0.3).astype(np.float32)).cuda()
    flat = torch.full((gcpush.SIREN_NPARAMS + 8,), 7.0, device="cuda")
    view = flat[off:off + gcpush.SIREN_NPARAMS]
    g = torch.empty(gcpush.SIREN_NPARAMS, device="cuda")
    assert view.data_ptr() % 16 != 0 and g.data_ptr() % 16 == 0
    with gcpush.Context() as c:
        c.siren_set(synth.siren_init(seed=1), omega0=30.0)
        loss = c.siren_loss_grad(x, t, g)
        assert abs(c.siren_loss_grad(x, t, view) - loss) < 1e-12 * loss
    assert float((view - g).norm()) < 1e-5 * float(g.norm()) > 0.0
    assert bool((flat[:off] == 7.0).all()) and bool((flat[off + gcpush.SIREN_NPARAMS:] == 7.0).all())


def test_gradient_of_a_large_batch_is_the_mean_of_its_parts():
    """2^22 samples against the mean over eight parts, summed in FP64. Sums in tensor memory are
    rounded towards zero: terms of one sign (targets of a common mean) lose up to 1e-7 of the
    gradient per 64 samples added there, 2.6e-4 between the whole and its parts where each of
    25 splits of the batch is one such sum. Rounded to nearest instead, the 2622 additions of a
    split and the 25 of the splits leave sqrt(2647 / 3) 2^-25, 1e-6. Held to 4e-6."""
    n, parts = 1 << 22, 8
    g = torch.Generator(device="cuda").manual_seed(4)
    x = torch.rand((n, 3), generator=g, device="cuda") * 1.2 - 0.6
    t = torch.randn((n, 8), generator=g, device="cuda") * 0.3 + 0.5
    whole = torch.empty(gcpush.SIREN_NPARAMS, device="cuda")
    with gcpush.Context() as c:
        c.siren_set(synth.siren_init(seed=9), omega0=30.0)
        c.siren_loss_grad(x, t, whole)
        mean = torch.zeros(gcpush.SIREN_NPARAMS, dtype=torch.float64, device="cuda")
        part = torch.empty_like(whole)
        for xs, ts in zip(x.chunk(parts), t.chunk(parts)):
            c.siren_loss_grad(xs, ts, part)
            mean += part.double() / parts
    hidden = slice(1024, 198400)
    err = float((whole.double() - mean)[hidden].norm() / mean[hidden].norm())
    print(err)
    assert err < 4e-6

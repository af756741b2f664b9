"""The FP32 value / gradient kernels where their work division changes: patches of a warp
chunk's pixels (64), one more or less, of an item's (512) and more; pixels under more patches
than an item stages (8) and than the grouping mask has bits (64); the per-source epilogue
with warps sharing a source of few or many images and with a warp per source.  Against the
FP64 pass (held to the oracle elsewhere) at the tolerances of the parity tests: local ELBO
1e-5, gradient 1e-4 in the 2-norm; the value-only call gives the value + gradient call's bits."""
import numpy as np
import pytest

from paper_1801_10277_gb300 import synth

pytestmark = pytest.mark.gpu


def _problem(n_src, H, W, n_img, boxes, seed=5):
    """n_src sources; boxes[s]: (x0, y0, w, h) of its patch, the same in every image."""
    rng = np.random.default_rng(seed)
    images = [synth._single_field_images(rng, H, W)[i % 5] for i in range(n_img)]
    truth, is_gal = synth.draw_truth(rng, n_src)
    for s, (x0, y0, w, h) in enumerate(boxes):
        truth[s, 0:2] = [x0 + 0.5 * (w - 1), y0 + 0.5 * (h - 1)]
    theta = synth.perturb_start(rng, truth, is_gal)
    for im in images:
        im.pixels = rng.poisson(160.0, size=(H, W)).astype(np.float32)
    mix = [np.stack([rng.dirichlet(np.full(n, 3.0)), np.sort(rng.uniform(0.02, 4.0, size=n))], 1) for n in (6, 8)]
    ps, pr, pc = synth.draw_priors(rng)
    pa = np.array([(i, *b) for b in boxes for i in range(n_img)], np.int32)
    po = np.arange(0, n_img * n_src + 1, n_img, dtype=np.int32)
    no, nb = np.zeros(n_src + 1, np.int32), np.zeros(0, np.int32)   # (neighbours matter to fits only)
    return synth.Problem(images=images, exp_mix=mix[0], dev_mix=mix[1], prior_star=ps, prior_r=pr, prior_c=pc,
                         theta=theta, truth=truth, patch_offsets=po, patches=pa, nbr_offsets=no, nbrs=nb)


CASES = {
    "chunk edges": lambda: _problem(6, 90, 120, 2, [(3, 3, 63, 1), (3, 6, 64, 1), (3, 9, 65, 1), (40, 20, 1, 1),
                                                    (60, 30, 8, 8), (64, 34, 13, 11)]),
    "item edges": lambda: _problem(5, 140, 160, 2, [(2, 2, 32, 16), (20, 10, 27, 19), (50, 20, 73, 7),
                                                    (40, 30, 101, 101), (80, 60, 32, 32)]),
    "ten patches on a pixel": lambda: _problem(11, 60, 60, 1, [(20 + s, 20 - s, 18, 16 + s) for s in range(11)]),
    "seventy patches on a pixel": lambda: _problem(72, 60, 60, 1, [(10 + s % 9, 10 + s // 9, 20, 20) for s in range(72)]),
    "many images": lambda: _problem(2, 24, 24, 520, [(4, 4, 5, 5), (7, 6, 9, 8)]),
    "many sources": lambda: _problem(2600, 128, 256, 1, [(4 * (s % 60), 2 * (s // 60), 5, 3) for s in range(2600)]),
}


@pytest.mark.parametrize("case", CASES)
def test_items(case):
    from paper_1801_10277_gb300 import celeste as cel
    prob = CASES[case]()
    P = cel.Problem(prob)
    t64, l64, g64 = P.elbo_grad(prob.theta, precision=cel.FP64)
    t32, l32, g32 = P.elbo_grad(prob.theta, precision=cel.FP32)
    tv, lv = P.elbo(prob.theta, precision=cel.FP32)
    assert tv == t32 and np.array_equal(lv, l32)
    assert abs(t32 - t64) <= 1e-5 * abs(t64)
    assert np.all(np.abs(l32 - l64) <= 1e-5 * np.abs(l64))
    assert np.all(np.linalg.norm(g32 - g64, axis=1) <= 1e-4 * np.linalg.norm(g64, axis=1))
    P.close()

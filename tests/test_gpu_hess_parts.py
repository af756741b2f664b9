"""The FP64 value / gradient pass and both Hessian passes where their work division and their
tables change shape: patches of a pixel, of a warp's pixels and one more or less, of several
parts; one to four PSF components; profile counts other than the model's 6 + 8 (the unrolled
kernel's); sky maps; parts of 32, 64 and 128 pixels.  Against the FP64 oracle at the
tolerances of the parity tests: ELBO 1e-10 / 1e-5, gradient and Hessian 1e-8 / 1e-4 in the
2-norm (FP64 / FP32)."""
import numpy as np
import pytest

from paper_1801_10277_gb300 import synth

pytestmark = pytest.mark.gpu

TOL_E = {0: 1e-10, 1: 1e-5}
TOL_D = {0: 1e-8, 1: 1e-4}


def _check(P, prec, theta, idx, loc, grad, hess):
    g_loc, g_grad, g_hess = P.hess(theta, precision=prec)
    _, e_loc, e_grad = P.elbo_grad(theta, precision=prec)
    for got, tol, ref in ((g_loc, TOL_E, loc), (e_loc, TOL_E, loc)):
        assert np.all(np.abs(got[idx] - ref) <= tol[prec] * np.abs(ref))
    for got, ref in ((g_grad, grad), (e_grad, grad), (g_hess, hess)):
        for k, s in enumerate(idx):
            assert np.linalg.norm(got[s] - ref[k]) <= TOL_D[prec] * np.linalg.norm(ref[k]), (prec, s)


@pytest.mark.parametrize("sizes", [((1, 1), (31, 1), (32, 1)), ((33, 1), (1, 65), (8, 8)), ((23, 11), (16, 16), (17, 15))])
@pytest.mark.parametrize("n_psf,n_exp,n_dev,sky_map", [(1, 1, 1, False), (2, 6, 8, True), (4, 5, 9, False), (4, 8, 8, True)])
def test_patch_sizes_and_table_shapes(sizes, n_psf, n_exp, n_dev, sky_map):
    from oracle.oracle import Oracle
    from paper_1801_10277_gb300 import celeste as cel
    rng = np.random.default_rng(7)
    H = W = 72
    images = synth._single_field_images(rng, H, W)
    for im in images:
        psf = np.concatenate([synth.draw_psf(rng), synth.draw_psf(rng, k=1)])
        psf[:, 0] *= 0.5
        im.psf = psf[:n_psf]
        if sky_map:
            im.sky_map = rng.uniform(140, 160, size=(H, W)).astype(np.float32)
    truth, is_gal = synth.draw_truth(rng, 3)
    truth[:, 0:2] = [[30, 30], [36, 33], [40, 28]]
    theta = synth.perturb_start(rng, truth, is_gal)
    synth.render_blobs(rng, images, truth, is_gal)
    mix = [np.stack([rng.dirichlet(np.full(n, 3.0)), np.sort(rng.uniform(0.02, 4.0, size=n))], 1) for n in (n_exp, n_dev)]
    prior_star, prior_r, prior_c = synth.draw_priors(rng)
    rows, offs = [], [0]
    for s, (w, h) in enumerate(sizes):
        x0, y0 = int(theta[s, 0]) - min(w, 30) // 2, min(int(theta[s, 1]) - min(h, 30) // 2, H - h)
        rows += [(n, x0, y0, w, h) for n in range(5)]
        offs.append(len(rows))
    po, pa = np.array(offs, np.int32), np.array(rows, np.int32)
    no, nb = synth.make_neighbours(3, po, pa)
    prob = synth.Problem(images=images, exp_mix=mix[0], dev_mix=mix[1], prior_star=prior_star, prior_r=prior_r,
                         prior_c=prior_c, theta=theta, truth=truth, patch_offsets=po, patches=pa, nbr_offsets=no,
                         nbrs=nb)
    orc = Oracle(prob)
    _, loc = orc.elbo(theta)
    _, grad, hess = orc.derivs(theta, hess=True)
    P = cel.Problem(prob)
    for prec in (cel.FP64, cel.FP32):
        _check(P, prec, theta, range(3), loc, grad, hess)
    P.close()


@pytest.mark.parametrize("n_src,side", [(60, 61), (110, 101)])
def test_larger_parts(n_src, side):
    """Problems of 1.1 and 5.6 million source-pixels (parts of 64 and 128 pixels); two sampled
    sources against the oracle on the sub-problem of them and their neighbours."""
    from oracle.oracle import Oracle
    from paper_1801_10277_gb300 import celeste as cel
    prob = synth.one_field(seed=11, n_src=n_src, H=1489, W=2048)
    c = np.clip(np.rint(prob.theta[:, :2]).astype(int), side // 2, [2047 - side // 2, 1488 - side // 2])
    prob.patches = np.array([(n, x - side // 2, y - side // 2, side, side) for x, y in c for n in range(5)], np.int32)
    prob.patch_offsets = np.arange(0, 5 * n_src + 1, 5, dtype=np.int32)
    prob.nbr_offsets, prob.nbrs = synth.make_neighbours(n_src, prob.patch_offsets, prob.patches)
    P = cel.Problem(prob)
    for s in (0, n_src - 1):
        keep = sorted({s, *prob.nbrs[prob.nbr_offsets[s]:prob.nbr_offsets[s + 1]].tolist()})
        sub = synth.subset(prob, keep)
        orc = Oracle(sub)
        _, loc = orc.elbo(sub.theta)
        _, grad, hess = orc.derivs(sub.theta, hess=True)
        k = keep.index(s)
        for prec in (cel.FP64, cel.FP32):
            _check(P, prec, prob.theta, [s], loc[k:k + 1], grad[k:k + 1], hess[k:k + 1])
    P.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_fit_does_not_depend_on_batch_sizes(prec):
    """One Cyclades sweep of the 500-source field in one sample (batches of 0.8 million
    source-pixels) and in samples of 32 (0.07 million): the same random order, so the same
    iterates bit for bit."""
    from paper_1801_10277_gb300 import celeste as cel
    prob = synth.config(1)
    order = np.random.default_rng(3).permutation(prob.n_src).astype(np.int32)[None]
    P = cel.Problem(prob)
    fits = [P.fit(prob.theta, precision=prec, max_sweeps=1, max_iter=2, refine_fp64=0, schedule="cyclades", order=order,
                  sample_size=size) for size in (prob.n_src, 32)]
    np.testing.assert_array_equal(fits[0][0], fits[1][0])
    np.testing.assert_array_equal(fits[0][1], fits[1][1])
    P.close()

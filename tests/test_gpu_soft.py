"""Soft silhouette on the GPU (soft_eval, the autograd op, soft_refine) against
the FP64 oracle: losses, analytic gradients and FP64 central differences."""
import numpy as np
import pytest

import oracle
from oracle import soft
from paper_2603_11404_gb300 import workload as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_11404_gb300 import build
    build.build()
    from paper_2603_11404_gb300 import api as a
    return a


def _case(api, mesh, cam, n_inst, K, seed, lam):
    sc = wl.make_scene(mesh, cam, n_instruments=n_inst, K=K)
    rng = np.random.default_rng(seed)
    gt = np.concatenate([wl.sample_state(rng, sc.K) for _ in range(n_inst)])
    M = wl.corrupt_mask(oracle.render(sc, gt), rng)
    P = wl.population_around(rng, gt, lam)
    tr = api.Tracker(sc, lambda_max=max(lam, 1))
    Mp = tr.pack_mask(torch.from_numpy(M).cuda())
    return sc, tr, M, Mp, P


def _rel(g, ref, s):
    return np.linalg.norm((g - ref) * s) / np.linalg.norm(ref * s)


@pytest.mark.parametrize("which", ["c1", "bimanual", "lookat"])
def test_soft_loss_and_gradient_match_oracle(api, which):
    if which == "c1":
        sc, tr, M, Mp, P = _case(api, "c1", "c1", 1, None, 11, 4)
    elif which == "bimanual":
        sc, tr, M, Mp, P = _case(api, "800", "c1", 2, wl.Intrinsics(150.0, 150.0, 50.0, 38.5, 101, 77), 12, 3)
    else:
        sc = wl.make_scene("c1", "c1", rot_param=wl.ROT_LOOKAT)
        rng = np.random.default_rng(13)
        gt = wl.sample_state(rng, sc.K)
        gt[:3] = [0.2, -0.4, 0.3]  # look-at angles (alpha, beta, gamma)
        M = wl.corrupt_mask(oracle.render(sc, gt), rng)
        P = wl.population_around(rng, gt, 3)
        tr = api.Tracker(sc, lambda_max=3)
        Mp = tr.pack_mask(torch.from_numpy(M).cuda())
    loss, g = tr.soft_eval(torch.from_numpy(P).cuda(), Mp, grad=True)
    loss, g = loss.cpu().numpy(), g.cpu().numpy()
    s = wl.default_scales(sc.d)
    for c in range(P.shape[0]):
        L, gref = soft.soft_grad(sc, P[c].astype(np.float64), M)
        assert loss[c] == pytest.approx(L, rel=1e-4), c
        assert _rel(g[c], gref, s) < 1e-3, (c, g[c], gref)


def test_soft_gradient_matches_fp64_central_differences(api):
    sc, tr, M, Mp, P = _case(api, "c1", "c1", 1, None, 21, 2)
    _, g = tr.soft_eval(torch.from_numpy(P).cuda(), Mp, grad=True)
    g = g.cpu().numpy()
    s = wl.default_scales(9)
    for c in range(P.shape[0]):
        x = P[c].astype(np.float64)
        fd = np.array([(soft.soft_loss(sc, x + e, M) - soft.soft_loss(sc, x - e, M)) / (2 * e[k])
                       for k, e in enumerate(np.eye(9) * 1e-4 * s)])
        assert _rel(g[c], fd, s) < 1e-3, (c, g[c], fd)


def test_soft_full_size_candidate_matches_oracle(api):
    """640x512, 20k-triangle mesh: one candidate's loss and gradient."""
    sc, tr, M, Mp, P = _case(api, "c2", "c2", 1, None, 31, 64)
    loss, g = tr.soft_eval(torch.from_numpy(P).cuda(), Mp, grad=True)
    L, gref = soft.soft_grad(sc, P[5].astype(np.float64), M)
    assert loss[5].item() == pytest.approx(L, rel=1e-4)
    assert _rel(g[5].cpu().numpy(), gref, wl.default_scales(9)) < 1e-3
    # the rest of the population: the loss alone
    for c in (0, 63):
        assert loss[c].item() == pytest.approx(soft.soft_loss(sc, P[c].astype(np.float64), M), rel=1e-4)


def test_autograd_function_backward_is_the_hand_written_gradient(api):
    sc, tr, M, Mp, P = _case(api, "c1", "c1", 1, None, 41, 5)
    x = torch.from_numpy(P).cuda().requires_grad_(True)
    w = torch.arange(1, 6, dtype=torch.float32, device="cuda")
    L = api.soft_silhouette_loss(x, tr, Mp)
    (L * w).sum().backward()
    _, g = tr.soft_eval(torch.from_numpy(P).cuda(), Mp, grad=True)
    assert torch.allclose(x.grad, w[:, None] * g, rtol=1e-4, atol=1e-3)
    assert torch.allclose(L, tr.soft_eval(torch.from_numpy(P).cuda(), Mp), rtol=1e-6)


def test_refine_improves_or_keeps_the_estimate(api):
    sc, tr, M, Mp, P = _case(api, "c1", "c1", 1, None, 51, 16)
    tr2 = api.Tracker(sc, loss_kind=wl.LOSS_XOR, lambda_max=16)
    init = P[0].astype(np.float64)
    es = api.CMAES(tr2, 16, init, wl.default_scales(9), sigma0=1.0, seed=7)
    es.track_frame(Mp, 5)
    before = es.state()["best_loss"]
    pose, picked = es.refine(Mp, top_k=8, steps=10, lr=0.05)
    st = es.state()
    assert st["best_loss"] <= before
    assert picked in range(-1, 8)
    assert (picked >= 0) == (st["best_loss"] < before)
    # the estimate is the adopted candidate and its fitness is the reported best
    l = tr2.eval_population(pose[None].contiguous(), Mp)
    assert l.item() == st["best_loss"]
    assert np.array_equal(pose.cpu().numpy(), st["best_x"])


def test_refine_adopts_candidates_after_a_short_search(api):
    """After a single generation from a displaced start the gradient steps
    find better binary fitness for some seeds: the refined candidates are
    scored with the same fitness kernel as the search (a refinement that could
    never be adopted would pass the test above)."""
    sc, tr, M, Mp, P = _case(api, "c1", "c1", 1, None, 53, 16)
    tr2 = api.Tracker(sc, loss_kind=wl.LOSS_XOR, lambda_max=16)
    adopted = 0
    for seed in range(6):
        es = api.CMAES(tr2, 16, P[seed].astype(np.float64), wl.default_scales(9), sigma0=1.0, seed=11 + seed)
        es.track_frame(Mp, 1)
        before = es.state()["best_loss"]
        pose, picked = es.refine(Mp, top_k=8, steps=10, lr=0.05)
        st = es.state()
        if picked >= 0:
            adopted += 1
            assert st["best_loss"] < before
            assert tr2.eval_population(pose[None].contiguous(), Mp).item() == st["best_loss"]
    assert adopted > 0


def test_soft_rejects_bad_arguments(api):
    from paper_2603_11404_gb300._abi import TrkError
    sc, tr, M, Mp, P = _case(api, "c1", "c1", 1, None, 61, 2)
    with pytest.raises(TrkError):
        tr.soft_eval(torch.from_numpy(P).cuda(), Mp, sigma=0.0)
    empty = torch.zeros((0, 9), dtype=torch.float32, device="cuda")
    assert tr.soft_eval(empty, Mp).numel() == 0


def test_soft_results_repeat_bit_for_bit(api):
    """The loss sums the tiles in a fixed order and the gradient sums are exact
    fixed-point integers: repeated calls (and a refinement run twice from the
    same state) give identical bits, at 640x512 with the 20k-triangle mesh."""
    sc, tr, M, Mp, P = _case(api, "c2", "c2", 1, None, 71, 16)
    Pd = torch.from_numpy(P).cuda()
    l0, g0 = tr.soft_eval(Pd, Mp, grad=True)
    for _ in range(3):
        l1, g1 = tr.soft_eval(Pd, Mp, grad=True)
        assert torch.equal(l0.view(torch.int32), l1.view(torch.int32))
        assert torch.equal(g0.view(torch.int32), g1.view(torch.int32))
    poses = []
    for _ in range(2):
        es = api.CMAES(tr, 16, P[0].astype(np.float64), wl.default_scales(9), sigma0=1.0, seed=3)
        es.track_frame(Mp, 3)
        pose, picked = es.refine(Mp, top_k=8, steps=5, lr=0.05)
        poses.append((pose.cpu().numpy().copy(), picked))
    assert np.array_equal(poses[0][0], poses[1][0]) and poses[0][1] == poses[1][1]


# Image sizes around the 8x4-pixel blocks of the pair kernels, triangle counts
# around the groups of 32, one and two instruments, sigma on both sides of 1.
# Tolerances: coordinates are rounded to about 3e-5 px in FP32, which moves an
# exponential's argument by 3e-5 / sigma; the bounds are those of the tests
# above (1e-4, 1e-3) at sigma >= 1 and twice them at sigma = 0.5.
@pytest.mark.parametrize("W,H,mesh,n_inst,sigma,lam", [
    (8, 4, "c1", 1, 1.0, 1), (9, 5, "c1", 1, 1.0, 2), (31, 33, "800", 2, 0.5, 3), (64, 64, "800", 1, 4.0, 2),
    (257, 67, "c1", 1, 1.0, 2), (100, 3, "900", 1, 0.5, 5),
])
def test_soft_block_edges_and_remainders(api, W, H, mesh, n_inst, sigma, lam):
    f = 1.25 * max(W, H)
    sc, tr, M, Mp, P = _case(api, mesh, "c1", n_inst, wl.Intrinsics(f, f, W / 2, H / 2, W, H), 91, lam)
    P[-1, 3:6] = [0.0, 0.0, -50.0]  # behind the camera: nothing drawn for this instrument
    loss, g = tr.soft_eval(torch.from_numpy(P).cuda(), Mp, sigma=sigma, grad=True)
    assert torch.equal(loss, tr.soft_eval(torch.from_numpy(P).cuda(), Mp, sigma=sigma))
    loss, g = loss.cpu().numpy(), g.cpu().numpy()
    s = wl.default_scales(sc.d)
    k = 1.0 if sigma >= 1.0 else 2.0
    for c in range(lam):
        L, gref = soft.soft_grad(sc, P[c].astype(np.float64), M, sigma)
        assert loss[c] == pytest.approx(L, rel=k * 1e-4, abs=1e-6), c
        if np.linalg.norm(gref * s) > 0:
            assert _rel(g[c], gref, s) < k * 1e-3, (c, g[c], gref)
        else:
            assert not g[c].any()


def test_soft_results_do_not_depend_on_the_population(api):
    """A population larger than one slice of the scratch (1280x1024, two
    instruments of 40k triangles: about 170 candidates) gives, candidate by
    candidate, the bits of a call on that candidate alone."""
    sc = wl.make_scene("40000", "c2", n_instruments=2, K=wl.Intrinsics(1600.0, 1600.0, 640.0, 512.0, 1280, 1024))
    rng = np.random.default_rng(95)
    gt = np.concatenate([wl.sample_state(rng, sc.K) for _ in range(2)])
    tr = api.Tracker(sc, lambda_max=1)
    M = api.unpack_mask(tr.render(torch.from_numpy(gt.astype(np.float32)).cuda()), 1280)
    Mp = tr.pack_mask(M)
    P = torch.from_numpy(wl.population_around(rng, gt, 190)).cuda()
    loss, g = tr.soft_eval(P, Mp, grad=True)
    for c in (0, 95, 169, 170, 171, 189):
        l1, g1 = tr.soft_eval(P[c:c + 1].contiguous(), Mp, grad=True)
        assert torch.equal(l1.view(torch.int32), loss[c:c + 1].view(torch.int32)), c
        assert torch.equal(g1.view(torch.int32), g[c:c + 1].view(torch.int32)), c


def test_autograd_forms_give_the_same_bits(api):
    """The op with the gradient taken along in the forward, the op that
    evaluates it in the backward, no_grad and a non-contiguous input."""
    sc, tr, M, Mp, P = _case(api, "c1", "c1", 1, None, 43, 5)
    wide = torch.from_numpy(np.repeat(P, 2, axis=1)).cuda()
    w = torch.arange(1, 6, dtype=torch.float32, device="cuda")
    l0, g0 = tr.soft_eval(torch.from_numpy(P).cuda(), Mp, grad=True)
    for x in (torch.from_numpy(P).cuda().requires_grad_(True), wide.requires_grad_(True)):
        y = x if x.shape[1] == 9 else x[:, ::2]
        for L in (api.soft_silhouette_loss(y, tr, Mp), api.SoftSilhouetteLoss.apply(y, tr, Mp)):
            assert torch.equal(L, l0)
            (g,) = torch.autograd.grad(L, y, w, retain_graph=True)
            assert torch.equal(g, w[:, None] * g0)
            assert torch.equal(torch.autograd.grad(L, y, w)[0], g)
    with torch.no_grad():
        assert torch.equal(api.soft_silhouette_loss(torch.from_numpy(P).cuda().requires_grad_(True), tr, Mp), l0)


def test_backward_after_an_inplace_change_is_refused(api):
    sc, tr, M, Mp, P = _case(api, "c1", "c1", 1, None, 44, 3)
    x = torch.from_numpy(P).cuda().requires_grad_(True)
    for L in (api.soft_silhouette_loss(x, tr, Mp), api.SoftSilhouetteLoss.apply(x, tr, Mp)):
        with torch.no_grad():
            x += 0.0
        with pytest.raises(RuntimeError, match="modified by an inplace operation"):
            L.sum().backward()


# Pixel centres exactly on an edge: the signed distance is smooth there and such a
# pixel carries the largest weight (a = 1/2).  Vertical, horizontal and diagonal
# edges through centres, in every column of a block; in the last two also corners,
# and in the last three bisectors, where the first of the nearest edges counts in
# the kernel and in the oracle.  The bound is that of the tests above.
@pytest.mark.parametrize("shift", range(8))
@pytest.mark.parametrize("quad", ["vertical", "horizontal", "triangle", "diagonal", "corners", "square"])
def test_soft_gradient_with_pixel_centres_on_edges(api, quad, shift):
    from _helpers import tiny_scene
    W, H, f = 64, 48, 100.0
    tris = [[0, 1, 2], [0, 2, 3]]
    if quad == "vertical":
        p = [(16, 8.5), (40, 8.5), (40, 32.25), (16, 32.25)]
    elif quad == "horizontal":
        p = [(16.5, 8), (40.25, 8), (40.25, 32), (16.5, 32)]
    elif quad == "diagonal":
        p = [(15.5, 8.5), (39.5, 8.5), (39.5, 32.5), (15.5, 32.5)]
    elif quad == "corners":
        p, tris = [(16, 8), (48, 8), (16, 32)], [[0, 1, 2]]
    elif quad == "square":
        p = [(16, 8), (40, 8), (40, 32), (16, 32)]
    else:
        p, tris = [(16.25, 8), (47.5, 8), (16.25, 31.5)], [[0, 1, 2]]
    verts = [[x + shift - W / 2, y - H / 2, 0.0] for x, y in p]  # at z = f a millimetre is a pixel
    sc = tiny_scene(W, H, f, verts, tris)
    M = np.zeros((H, W), np.uint8)
    M[12:36, 19 + shift:46 + shift] = 1
    tr = api.Tracker(sc, lambda_max=2)
    Mp = tr.pack_mask(torch.from_numpy(M).cuda())
    P = np.zeros((2, 9), np.float32)
    P[:, 5] = f
    P[1, 3] = 0.3125  # the same off the centres
    loss, g = tr.soft_eval(torch.from_numpy(P).cuda(), Mp, grad=True)
    s = wl.default_scales(9)
    for c in range(2):
        L, gref = soft.soft_grad(sc, P[c].astype(np.float64), M)
        assert loss[c].item() == pytest.approx(L, rel=1e-4), c
        assert _rel(g[c].cpu().numpy(), gref, s) < 1e-3, (c, g[c], gref)


@pytest.mark.parametrize("first", ["loss", "gradient"])
def test_soft_scratch_stays_within_its_bound(api, first):
    """A loss of 1024 candidates and a gradient of eight on one tracker, in either
    order: the scratch stays below its two gigabytes (a candidate of the largest
    image holds about 8 MB), and the results are those of a tracker of their own."""
    sc = wl.make_scene("c1", "c2", K=wl.Intrinsics(1600.0, 1600.0, 640.0, 640.0, 1280, 1280))
    rng = np.random.default_rng(97)
    gt = wl.sample_state(rng, sc.K)
    P = torch.from_numpy(wl.population_around(rng, gt, 1024)).cuda()
    fresh = api.Tracker(sc, lambda_max=1)
    Mp = fresh.pack_mask(api.unpack_mask(fresh.render(torch.from_numpy(gt.astype(np.float32)).cuda()), 1280))
    want = [x.clone() for x in fresh.soft_eval(P[:8].contiguous(), Mp, grad=True)]
    del fresh
    tr = api.Tracker(sc, lambda_max=1)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for kind in ("loss", "gradient") if first == "loss" else ("gradient", "loss"):
        if kind == "loss":
            loss = tr.soft_eval(P, Mp)
        else:
            got = tr.soft_eval(P[:8].contiguous(), Mp, grad=True)
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] < (2 << 30) + (64 << 20)
    for a, b in zip(got, want):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    assert torch.equal(loss[:8].view(torch.int32), want[0].view(torch.int32))


def test_soft_calls_of_both_kinds_under_capture(api):
    """After a loss on a population, a gradient on as many candidates can be
    captured, and a captured loss stays valid after it."""
    sc, tr, M, Mp, P = _case(api, "c1", "c1", 1, None, 98, 6)
    Pd = torch.from_numpy(P).cuda()
    want_l = tr.soft_eval(Pd, Mp)
    graphs, outs = [], []
    for grad in (False, True):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            outs.append(tr.soft_eval(Pd, Mp, grad=grad))
        graphs.append(g)
    l1, g1 = tr.soft_eval(Pd, Mp, grad=True)
    for g in graphs + graphs:
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(outs[0], want_l) and torch.equal(l1, want_l)
    assert torch.equal(outs[1][0], want_l) and torch.equal(outs[1][1], g1)


def test_soft_losses_of_the_fringe_keep_their_digits(api):
    """An instrument outside the image whose fringe reaches into it, no mask: losses
    from 3 down to 7e-10, within the bound of the tests above (and approx's own 1e-12:
    corners lie whole pixels away, and a pixel exactly at the cutoff adds 7e-13)."""
    from _helpers import tiny_scene
    W, H, f = 64, 48, 100.0
    verts = [[x - 10.0, y - 10.0, 0.0] for x, y in ((0, 0), (20, 1), (19, 22), (1, 20))]
    sc = tiny_scene(W, H, f, verts, [[0, 1, 2], [0, 2, 3]])
    tr = api.Tracker(sc, lambda_max=1)
    Mp = tr.pack_mask(torch.zeros((H, W), dtype=torch.uint8, device="cuda"))
    P = np.zeros((8, 9), np.float32)
    P[:, 5] = f
    P[:, 3] = [-42.3, -46.0, -48.0, -50.0, -51.0, -52.0, -53.0, -54.0]
    loss = tr.soft_eval(torch.from_numpy(P).cuda(), Mp).cpu().numpy()
    for c in range(8):
        L = soft.soft_loss(sc, P[c].astype(np.float64), np.zeros((H, W)))
        assert loss[c] == pytest.approx(L, rel=1e-4), c

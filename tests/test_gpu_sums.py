"""What the sums of the pair kernels hold: values that must not enter them, and bits that must.

Scenes are built so that the right sums are known without a reference of the same
precision: weights that are FP32 numbers (pairs at distance zero), counts that are exact.
"""
import numpy as np
import pytest

import oracle as O
import scenes

pytestmark = pytest.mark.gpu

LOSS_TOL, GRAD_TOL, H_TOL = 1e-5, 1e-4, 1e-4
ELL = 0.25
H_CELL = 3.0 * ELL * (1.0 + 1.0 / 1024.0)      # the grid's cell edge


@pytest.fixture(scope="module")
def pk():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2403_01254_gb300 as pk
    pk.load()
    return pk


def _reln(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(b), 1e-300))


def _pair(xa, xb, sem=None, rgb=None, **params):
    return dict(xyz=[np.asarray(xa, np.float64), np.asarray(xb, np.float64)], sem=sem, rgb=rgb,
                edges=np.array([[0, 1]], np.int32), poses0=np.stack([np.eye(4), np.eye(4)]),
                params=dict(dict(ell=ELL, cutoff_mult=3.0, sigma=1.0, sem_bf16=0), **params))


def _eval(pk, prob, **kw):
    g = pk.Problem.from_scene(prob)
    try:
        return g.eval(prob["poses0"], **kw)
    finally:
        g.close()


# Labels of 1e25: their products with each other (BF16) or their FP16 parts (FP32 labels) are
# infinite.  The two points that carry them are farther than r_c from every point of
# the other frame, but lie in the box of the other points, so they share tiles with them.
@pytest.mark.parametrize("bf16", [0, 1])
def test_infinite_label_products_outside_the_cutoff(pk, bf16):
    at = lambda *f: (0.5 + np.array(f)) * H_CELL
    near = [at(-0.48, -0.48, -0.48), at(0.48, 0.48, 0.48)]
    rng = np.random.default_rng(3)
    jit = lambda n: 0.003 * rng.standard_normal((n, 3))
    xa = np.concatenate([near[0] + jit(20), near[1] + jit(20), at(0.48, -0.48, 0.0)[None]])
    xb = np.concatenate([near[0] + jit(9), near[1] + jit(8), at(-0.48, 0.48, 0.0)[None]])
    sem = []
    for x in (xa, xb):
        s = scenes.round_to_bf16(scenes.dirichlet_labels(rng, rng.integers(0, 4, len(x)), 4))
        s[-1] = 2.0 ** 83
        sem.append(s)
    prob = _pair(xa, xb, sem, sem_bf16=bf16)
    ref = O.evaluate(prob, prob["poses0"])
    assert ref["edge_pairs"].tolist() == [20 * 9 + 20 * 8]
    out = _eval(pk, prob)
    assert out["edge_pairs"].tolist() == ref["edge_pairs"].tolist()
    assert abs(out["loss"] - ref["loss"]) <= LOSS_TOL * abs(ref["loss"])
    assert _reln(out["grad"], ref["grad"]) <= GRAD_TOL
    assert _reln(out["H"], ref["H"]) <= H_TOL


# Eight queries at the corners of their home cell, each with one candidate at its own
# place: a weight per lane that FP32 holds, whose sum (25 bits and more) it does not.  Only the
# rounding to 2^-51 (the fixed point's step for 8 x 8 points and labels of 4) is left.
@pytest.mark.parametrize("bf16,extra", [(0, dict(sem_min=1e-12)), (1, dict(sem_min=1e-12)), (0, dict(ell_color=0.2)),
                                        (1, dict(ell_color=0.2)), (0, dict(top_k=1)), (1, dict(top_k=3))])
def test_lanes_of_a_unit_are_summed_without_rounding(pk, bf16, extra):
    corners = np.array([[x, y, z] for z in (-1, 1) for y in (-1, 1) for x in (-1, 1)], np.float64)
    xyz = (0.5 + 0.4998 * corners) * H_CELL
    for big in range(8):
        s = np.zeros((8, 4))
        s[:, 1] = 3.0 * 2.0 ** -11
        s[big, 1] = 4.0
        rgb = [np.full((8, 3), 0.25)] * 2 if "ell_color" in extra else None
        out = _eval(pk, _pair(xyz, xyz, [s, s], rgb, sem_bf16=bf16, **extra))
        want = 16.0 + 7 * 9 * 2.0 ** -22
        assert out["edge_pairs"].tolist() == [8]
        assert abs(-out["loss"] - want) <= 1e-12 * want
        assert abs(out["H"][0, 0] - want) <= 1e-12 * want


# Every candidate and every query at the centre of one cell: each weight is the label product
# c, so a chain of n FP32 additions of it is off by up to n 2^-24, in one direction.  Chains
# end after 32 additions (lane unit) or 128 (dense unit), which are then added up: a few hundred in
# all for 51 200 candidates, where one chain would have 25 600 or 3 200.  The loss's tolerance
# is what every problem is promised.
def _one_cell(n, nb, c, **extra):
    xyz = [np.full((k, 3), 0.5 * H_CELL) for k in (n, nb)]
    return _pair(*xyz, [np.full((n, 1), c), np.ones((nb, 1))], **extra)


@pytest.mark.parametrize("c", [0.55, 0.6, 0.8371, 0.9, 1.0 / 3.0])
@pytest.mark.parametrize("nb", [3, 7, 13, 40])
def test_long_streams_of_equal_weights(pk, nb, c):
    n, c = 51200, float(np.float32(c))
    out = _eval(pk, _one_cell(n, nb, c, sem_min=1e-12))
    assert out["edge_pairs"].tolist() == [n * nb]
    assert abs(-out["loss"] / (n * nb * c) - 1.0) <= LOSS_TOL


@pytest.mark.parametrize("c", [0.6, 0.8371])
def test_long_streams_of_equal_weights_dense(pk, c):
    # 20 bits of c: exact in the labels' and the weights' two FP16 parts; queries enough that no
    # stream is shared by several warps
    n, nb, c = 51200, 160000, round(c * 2 ** 20) / 2.0 ** 20
    out = _eval(pk, _one_cell(n, nb, c))
    assert out["edge_pairs"].tolist() == [n * nb]
    assert abs(-out["loss"] / (n * nb * c) - 1.0) <= LOSS_TOL


# An edge's sums do not depend on what else is evaluated with it, also where long streams are
# shared by several warps.
@pytest.mark.parametrize("variant", ["plain", "fp32", "bf16", "color"])
def test_an_edge_alone_equals_the_same_edge_among_others(pk, variant):
    for n, extent in ((900, 1.2), (2500, 1.5)):
        prob = scenes.tiny_problem(seed=61, n_frames=5, n=n, extent=extent, ell=0.15, color=variant == "color")
        if variant == "plain":
            prob["sem"] = None
        if variant == "bf16":
            prob["sem"] = [scenes.round_to_bf16(s) for s in prob["sem"]]
            prob["params"] = dict(prob["params"], sem_bf16=1)
        full = _eval(pk, prob, want_blocks=True)
        for e in (0, 4, 9):
            alone = _eval(pk, dict(prob, edges=np.asarray(prob["edges"])[e:e + 1]), want_blocks=True)
            assert alone["edge_pairs"][0] == full["edge_pairs"][e]
            assert np.array_equal(alone["H_blocks"][0], full["H_blocks"][e])

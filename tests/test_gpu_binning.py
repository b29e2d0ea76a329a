"""Binning of the queries and cutting into units, at the sizes where they change course.

Edges of at most 4096 queries are binned by one block each (1 to 4 queries a
thread), larger ones by the tiled sort (tiles of 2048 and, from 5 M queries on,
4096) and the unit pass (blocks of 256): sizes around each step, cells longer than a block
whose first query is or is not the first of all, and streams long enough to be shared by
several warps.  Tolerances are those of the parity tests (loss 1e-5, gradient and
Gauss-Newton matrix 1e-4 relative); in the clumps every pair lies inside the cutoff, so
their counts are exact.  Units of few queries share a query among lanes (steps at 4, 8
and 16 queries): counts around them, with streams of a part of a batch to many.
"""
import numpy as np
import pytest

import oracle as O
import scenes

pytestmark = pytest.mark.gpu

LOSS_TOL, GRAD_TOL, H_TOL = 1e-5, 1e-4, 1e-4


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


def _check(pk, prob, exact_count=None):
    ref = O.evaluate(prob, prob["poses0"])
    g = pk.Problem.from_scene(prob)
    try:
        out = g.eval(prob["poses0"])
    finally:
        g.close()
    if exact_count is not None:
        assert out["edge_pairs"].tolist() == exact_count
    assert np.abs(out["edge_pairs"] - ref["edge_pairs"]).sum() <= 3
    assert abs(out["loss"] - ref["loss"]) <= LOSS_TOL * abs(ref["loss"])
    assert _reln(out["grad"], ref["grad"]) <= GRAD_TOL
    assert _reln(out["H"], ref["H"]) <= H_TOL


def _clump(na, nb, lead, variant):
    """na and nb points of the two frames inside one cell; `lead` lone points of frame b in cells before it."""
    rng = np.random.default_rng(1000 * nb + lead)
    prob = scenes.tiny_problem(seed=9, n_frames=2, n=8, extent=1.0, ell=0.15, color=variant == "color")
    lone = np.array([[-2.0 - 0.5 * k, 0.2, 0.2] for k in range(lead)]).reshape(lead, 3)
    box = [0.12 + 0.2 * rng.random((n, 3)) for n in (na, nb)]
    prob["xyz"] = [np.concatenate([lone + [0.0, 9.0, 0.0], box[0]]), np.concatenate([lone, box[1]])]
    prob["poses0"] = np.stack([np.eye(4), scenes.make_pose(
        scenes.rot_from_axis_angle(np.array([0.0, 0.0, 1.0]), 0.05), np.array([0.01, -0.01, 0.005]))])
    m = [len(x) for x in prob["xyz"]]
    prob["rgb"] = [rng.random((k, 3)) for k in m] if variant == "color" else None
    sem = [scenes.dirichlet_labels(rng, rng.integers(0, 4, k), 4) for k in m]
    prob["sem"] = None if variant == "plain" else sem
    if variant == "bf16":
        prob["sem"] = [scenes.round_to_bf16(s) for s in sem]
        prob["params"] = dict(prob["params"], sem_bf16=1)
    return prob


@pytest.mark.parametrize("variant", ["plain", "fp32", "bf16", "color"])
@pytest.mark.parametrize("na,nb,lead", [(1, 1, 0), (255, 255, 0), (257, 257, 0), (700, 700, 5), (1025, 1025, 0),
                                        (40, 1024, 3), (40, 2048, 0), (40, 2049, 1), (40, 3073, 0), (40, 4096, 0),
                                        (40, 4097, 0), (40, 4096, 1), (40, 9001, 300)])
def test_cells_longer_than_a_block(pk, variant, na, nb, lead):
    _check(pk, _clump(na, nb, lead, variant), exact_count=[na * nb])


@pytest.mark.parametrize("n", [1023, 1025, 2048, 3073, 4096, 4097, 6145, 10240, 10241])
def test_query_counts_around_a_tile(pk, n):
    _check(pk, scenes.tiny_problem(seed=40 + n % 7, n_frames=2, n=n, extent=2.5 if n < 4000 else 4.0, ell=0.1))


@pytest.mark.parametrize("variant,extra", [("plain", {}), ("color", {}), ("fp32", dict(sem_min=0.1)),
                                           ("bf16", dict(sem_min=0.1)), ("plain", dict(top_k=8)),
                                           ("color", dict(top_k=3)), ("fp32", dict(top_k=8)),
                                           ("bf16", dict(top_k=1, sem_min=0.1))])
@pytest.mark.parametrize("nb", [1, 4, 5, 8, 9, 16, 17, 32, 33])
def test_units_of_few_queries(pk, variant, extra, nb):
    for na in (1, 2, 33, 300):
        prob = _clump(na, nb, 1, variant)
        prob["params"] = dict(prob["params"], **extra)
        _check(pk, prob)

"""Batched swarms whose state is kept in panels of 8 dimensions: every swarm equals its
oracle run at the edges of the panels (the last one whole, one dimension, one short),
of the units of 16 particles and of the padding, next to swarms too narrow for panels."""
import pytest

from tests.gpu_common import BOUNDS, C12, W, load_cupso, oracle_swarm, same_bits

pytestmark = pytest.mark.gpu

WIDTHS = (25, 26, 31, 32, 33, 39, 40, 41, 100, 255, 256, 257)
SIZES = (1, 2, 15, 16, 17, 127, 128, 129, 500, 1025)


@pytest.fixture(scope="module")
def P():
    return load_cupso()


def check(P, probs, iters, statuses=None):
    rc, res = P.cupso_solve_batch(probs, iters)
    for k, p in enumerate(probs):
        ref = oracle_swarm(p["fitness_id"], p["N"], p["D"], p["seed"], swarm=p["swarm_id"], bounds=p["bounds"],
                           c1=p["c1"]).init().step_sync(iters)
        assert res[k]["status"] == (statuses or {}).get(k, P.CUPSO_OK), k
        assert res[k]["idx"] == ref.gbest_idx, (k, p)
        # a NaN's payload is the processor's own
        assert same_bits(res[k]["fit"], ref.gbest_fit) or (res[k]["fit"] != res[k]["fit"]
                                                           and ref.gbest_fit != ref.gbest_fit), (k, p)
        assert same_bits(res[k]["pos"], ref.gbest_pos), (k, p)
    return rc


def problem(fid, N, D, k, **kw):
    return dict(dict(D=D, N=N, bounds=BOUNDS[fid], w=W, c1=C12, c2=C12, fitness_id=fid, seed=50 + k,
                     swarm_id=k), **kw)


@pytest.mark.parametrize("narrow", [False, True])
@pytest.mark.parametrize("fid", [0, 1, 2, 3, 4])
def test_edges_match_oracle(P, fid, narrow, monkeypatch):
    """Every width against sizes around it; `narrow` adds swarms below the panels' width."""
    monkeypatch.delenv("CUPSO_BATCH_KERNEL", raising=False)
    probs = [problem(fid, SIZES[(3 * k + s) % len(SIZES)], D, 2 * k + s) for k, D in enumerate(WIDTHS) for s in (0, 1)]
    probs.append(problem(fid, 6500, 257, 60))       # enough particles for panels at these widths
    if narrow:
        probs += [problem((fid + k) % 5, 40 + 90 * k, D, 100 + k) for k, D in enumerate((1, 2, 3, 8, 23, 24))]
    assert check(P, probs, 30 if narrow else 9) == P.CUPSO_OK


def test_general_path_and_nan_match_oracle(P, monkeypatch):
    """Swarms off the fast path (a bound at 0, a tiny c1) and one that overflows."""
    monkeypatch.delenv("CUPSO_BATCH_KERNEL", raising=False)
    probs = []
    for k in range(15):
        kw = [dict(bounds=(0.0, 10.0, 2.0)), dict(c1=1e-38), {}][k % 3]
        probs.append(problem(k % 5, 60 + 61 * k, WIDTHS[k % len(WIDTHS)], k, **kw))
    probs.append(problem(4, 300, 30, 40, bounds=(-1e30, 1e30, 1.0)))
    probs.append(problem(1, 6500, 257, 60))
    probs.append(problem(2, 200, 33, 61, bounds=(-3e6, 3e6, 1e5)))   # beyond the small cosine arguments
    assert check(P, probs, 8, {15: P.CUPSO_ERR_NAN}) == P.CUPSO_ERR_NAN


@pytest.mark.parametrize("iters", [0, 1, 2, 21])
def test_iteration_counts_match_oracle(P, iters, monkeypatch):
    """Step 1 alone, single launches and replayed ones; a swarm of many units."""
    monkeypatch.delenv("CUPSO_BATCH_KERNEL", raising=False)
    probs = [problem(k % 5, 3000 if k == 3 else 100 + 50 * k, 25 + 9 * k, k) for k in range(8)]
    probs.append(problem(0, 6500, 88, 60))
    assert check(P, probs, iters) == P.CUPSO_OK


def test_large_batch_edges_match_oracle(P, monkeypatch):
    """A batch large enough for the deeper ring: the smallest widths it takes, edges of the
    panels and units, and narrower swarms, which then run outside the panels; the three
    that make it large are not compared."""
    monkeypatch.delenv("CUPSO_BATCH_KERNEL", raising=False)
    probs = [problem(k % 5, SIZES[(3 * k) % len(SIZES)], D, k)
             for k, D in enumerate((33, 34, 39, 40, 41, 48, 255, 256, 25, 32, 24, 8, 33, 40, 41))]
    large = [problem(k, 65536, 900, 70 + k) for k in (0, 1, 3)]
    rc, res = P.cupso_solve_batch(probs + large, 7)
    assert rc == P.CUPSO_OK
    for k, p in enumerate(probs):
        ref = oracle_swarm(p["fitness_id"], p["N"], p["D"], p["seed"], swarm=p["swarm_id"]).init().step_sync(7)
        assert res[k]["idx"] == ref.gbest_idx, (k, p)
        assert same_bits(res[k]["fit"], ref.gbest_fit) and same_bits(res[k]["pos"], ref.gbest_pos), (k, p)

"""Particles that move between the threads of a block at the end of an interval
(the 128-thread shape) against the 32-thread shape, which never moves any:
populations of many digesters (a moved particle takes its own digester's
constants along), cold starts from learned guesses (the count of guesses done
anew travels with the particle) and shards of a population."""
import numpy as np
import pytest

from paper_2311_08927_gb300 import chad as CH
from paper_2311_08927_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# FP64: 1e-16 per operation over some 1e2 steps and 1e4 operations.  Mixed: two
# runs that round apart may take steps a little apart, each within rtol = 1e-6.
FORMS = [(dict(precision=CH.PREC_FP64, h2_algebraic=True), 1e-10),
         (dict(precision=CH.PREC_MIXED, h2_algebraic=True), 1e-5)]
N = 20_011


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_08927_gb300 import build
    build.build()


def _run(pop, variant, network=None, **kw):
    sim = CH.Simulator(pop, learned=0 if network is None else 1, **kw)
    if network is not None:
        CH.chad_set_mlp(sim.ctx, *network)
    CH.chad_set_kernel_variant(sim.ctx, variant)
    sim.load()
    sim.step(60.0, 1)
    out = sim.read()
    sim.close()
    return out


def _same(a, b, tol, counters):
    floor = 1e-12 * np.abs(b["y"]).max(axis=1, keepdims=True) + 1e-300
    assert (np.abs(a["y"] - b["y"]) / np.maximum(np.abs(b["y"]), floor)).max() <= tol
    assert np.array_equal(a["status"], b["status"])
    for k in counters:
        assert a["stats"][k] == b["stats"][k], k


@pytest.mark.parametrize("kw,tol", FORMS)
def test_moved_particles_of_many_digesters(kw, tol):
    pop = I.config_population(5, n=N)
    fp64 = kw["precision"] == CH.PREC_FP64
    _same(_run(pop, 0, **kw), _run(pop, 5, **kw), tol,
          ("accepted_steps", "rejected_steps", "min_steps", "max_steps") if fp64 else ())


@pytest.mark.parametrize("kw,tol", FORMS)
def test_moved_particles_keep_their_learned_start(kw, tol):
    pop = I.config_population(3, n=N)
    rng = np.random.default_rng(3)
    params = 0.2 * rng.standard_normal(CH.MLP_NPARAM)
    norm = np.concatenate([np.full(32, -2.0), np.full(32, 0.3)])
    network = (params, norm, np.array([-7.4, -4.0, 0.5, 0.3]))
    a, b = _run(pop, 0, network, **kw), _run(pop, 5, network, **kw)
    # the guesses, and which of them are done anew, are the same in both runs
    _same(a, b, tol, ("mlp_redo",))
    assert 0 < a["stats"]["accepted_steps"]


@pytest.mark.parametrize("kw,tol", FORMS)
def test_shards_with_one_variant_match_the_whole_bit_for_bit(kw, tol):
    """A default launch shape follows the particle count; with the variant set
    a particle's run does not depend on the others, whichever thread ends it."""
    pop = I.config_population(3, n=N)
    whole = _run(pop, 0, **kw)
    for a, b in ((0, 700), (700, N)):
        part = I.Population([I.Digester(n=b - a)], np.ascontiguousarray(pop.y[:, a:b]), pop.T[a:b],
                            np.ascontiguousarray(pop.pos[:, a:b]), False, "shard")
        out = _run(part, 0, **kw)
        for k in ("y", "S_H", "h", "status"):
            assert np.array_equal(out[k], whole[k][..., a:b]), k

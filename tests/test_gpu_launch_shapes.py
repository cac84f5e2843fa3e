"""The launch shape that a context takes by its particle count (no autotuner,
no explicit variant) gives the results of an explicit shape, around the counts
where the rule changes and at the ends of the range."""
import numpy as np
import pytest

from paper_2311_08927_gb300 import chad as CH
from paper_2311_08927_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sms():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_08927_gb300 import build
    build.build()
    return torch.cuda.get_device_properties(0).multi_processor_count


def _run(pop, variant, **kw):
    sim = CH.Simulator(pop, fixed_substeps=2, **kw)
    if variant is not None:
        CH.chad_set_kernel_variant(sim.ctx, variant)
    sim.load()
    sim.step(60.0, 1)
    out = sim.read()
    sim.close()
    return out


# FP64: two fixed steps of the same operations, whose contraction may differ
# between the instances: some 1e3 roundings of 1.1e-16.  Mixed: FP32 stage
# vectors (6e-8) times the relative change of a state over the interval (< 1).
@pytest.mark.parametrize("kw,tol", [(dict(precision=CH.PREC_FP64, h2_algebraic=True), 1e-12),
                                    (dict(precision=CH.PREC_MIXED, h2_algebraic=True), 1e-6)])
@pytest.mark.parametrize("per_sm,extra", [(0, 1), (64, 0), (64, 1), (128, 0), (128, 1), (300, 7)])
def test_default_shape_equals_an_explicit_one(sms, kw, tol, per_sm, extra):
    pop = I.config_population(3, n=per_sm * sms + extra)
    a, b = _run(pop, None, **kw), _run(pop, 0, **kw)
    floor = 1e-12 * np.abs(b["y"]).max(axis=1, keepdims=True) + 1e-300
    assert (np.abs(a["y"] - b["y"]) / np.maximum(np.abs(b["y"]), floor)).max() <= tol
    assert np.array_equal(a["status"], b["status"])


@pytest.mark.parametrize("extra", [0, 1])
def test_mixed_default_shape_around_the_line_of_the_large_blocks(sms, extra):
    kw = dict(precision=CH.PREC_MIXED, h2_algebraic=True)
    pop = I.config_population(3, n=232 * sms + extra)
    a, b = _run(pop, None, **kw), _run(pop, 5, **kw)
    floor = 1e-12 * np.abs(b["y"]).max(axis=1, keepdims=True) + 1e-300
    assert (np.abs(a["y"] - b["y"]) / np.maximum(np.abs(b["y"]), floor)).max() <= 1e-6
    assert np.array_equal(a["status"], b["status"])


def _adaptive(pop, variant, **kw):
    sim = CH.Simulator(pop, **kw)
    CH.chad_set_kernel_variant(sim.ctx, variant)
    sim.load()
    sim.step(60.0, 1)
    out = sim.read()
    sim.close()
    return out


# At the end of an interval the particles of a block move together into its
# first threads.  32-thread blocks never move any: the same attempts, in another
# thread.  FP64: 1e-16 per operation over some 1e2 steps and 1e4 operations.
# Mixed: two runs that round apart may take steps a little apart, each within
# rtol = 1e-6, over some ten steps.
@pytest.mark.parametrize("variant", [0, 3, 4, 6])
@pytest.mark.parametrize("n", [1, 33, 700, 20_011])
@pytest.mark.parametrize("kw,tol", [(dict(precision=CH.PREC_FP64), 1e-10),
                                    (dict(precision=CH.PREC_FP64, h2_algebraic=True), 1e-10),
                                    (dict(precision=CH.PREC_MIXED), 1e-5),
                                    (dict(precision=CH.PREC_MIXED, h2_algebraic=True), 1e-5)])
def test_particles_that_move_between_threads_keep_their_run(sms, kw, tol, n, variant):
    pop = I.config_population(3, n=n)
    a, b = _adaptive(pop, variant, **kw), _adaptive(pop, 5, **kw)
    floor = 1e-12 * np.abs(b["y"]).max(axis=1, keepdims=True) + 1e-300
    assert (np.abs(a["y"] - b["y"]) / np.maximum(np.abs(b["y"]), floor)).max() <= tol
    assert np.array_equal(a["status"], b["status"])
    if kw["precision"] == CH.PREC_FP64:
        for k in ("accepted_steps", "rejected_steps", "min_steps", "max_steps", "failed_particles"):
            assert a["stats"][k] == b["stats"][k], k

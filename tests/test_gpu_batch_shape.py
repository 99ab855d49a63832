"""A batch takes passes of several steps per launch unless a shape of the
caller's own is in force: seen by the time of its steps, which passes shorten to a
third on lattices of this size."""
import pytest

from paper_2206_12412_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_12412_gb300 import lbm
    lbm.load_library()
    return lbm


def _ms(batch, n=256):
    import torch
    best = 1e30
    for _ in range(5):   # the first one captures graphs
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        batch.step(n)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def test_passes_in_the_librarys_shape(gpu):
    p = W.with_crack(W.base_problem(1000, 700), mode="prescribed", y=350.0, x_tip=100.0, v_rel=0.1)
    p["loads"] = [{"edge": "top", "kind": "const", "amp": 1e-3}]
    lats = [gpu.Lattice(p, "f32") for _ in range(48)]
    batch = gpu.Batch(lats)
    in_passes = _ms(batch)

    def passes():
        return _ms(batch) < 1.6 * in_passes

    batch.set_shape(64, 8)           # the caller's: single steps
    assert not passes()
    batch.set_shape(128, 16)         # the default
    assert passes()
    batch.set_lookahead(1)           # the value in force
    assert passes()
    batch.set_lookahead(2)
    assert not passes()
    batch.set_lookahead(1)
    assert passes()
    batch.set_shape(64, 16)
    assert not passes()
    batch.tune(trial_steps=2)
    assert passes()                  # the library's again
    tuned = batch.info()
    batch.set_lookahead(3 - tuned["lookahead"])
    assert not passes()
    batch.set_lookahead(tuned["lookahead"])
    assert passes()
    batch.close()
    batch = gpu.Batch(lats, band_rows=8)
    assert not passes()
    batch.close()

"""The K window of a crack in any direction, against the oracle: windows of
less than one pair, a few pairs in more than two lanes, and more sites than a
warp sifts at a time; unit and scaled spacings (the divisions skipped where
they are exact); one and two growing ends.  FP64 fields within 1e-12 of the
state's scale, K within 1e-9 of its largest value, tips, pair counts and cut
masks bit-exact: the tolerances of the other tests of this crack."""
import numpy as np
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


@pytest.mark.parametrize("mode", ["prescribed", "kcrit"])
@pytest.mark.parametrize("deg", [0.0, 23.0, 118.0])
@pytest.mark.parametrize("width", [0.6, 1.0, 2.0, 4.0, 40.0])
@pytest.mark.parametrize("dh", [1.0, 0.5])
def test_windows(oracle_mod, gpu, mode, deg, width, dh):
    nx, ny = 200, 160
    c, s = np.cos(np.radians(deg)), np.sin(np.radians(deg))
    p = W.base_problem(nx, ny, bc_mode="bounceback", edges=("free", "free", "dirichlet", "dirichlet"), cs=0.5)
    p["dh"], p["dt"] = dh, dh
    p["loads"] = [{"edge": "top", "kind": "linear", "amp": 4e-3, "t": 40.0 * dh},
                  {"edge": "bottom", "kind": "linear", "amp": -4e-3, "t": 40.0 * dh}]
    half = 24.0
    mid = (nx / 2 + 0.3, ny / 2 + 0.2)
    at = lambda r: ((mid[0] + r * c) * dh, (mid[1] + r * s) * dh)
    p = W.with_line_crack(p, mode=mode, start=at(-half), tip=at(half), v_rel=0.6,
                          K_C=0.2 * W.strip_reference_K(0.25, 4e-3, ny * dh), r0=2.0 * dh, fit_width=width * dh, two_tips=deg != 118.0)
    o, g = oracle_mod.Oracle(p), gpu.Lattice(p, "f64")
    for n in (3, 90, 40):
        o.step(n)
        g.step(n)
    (wo, wdo), (wg, wdg) = o.fields(), g.fields()
    for a, b in ((wo, wg), (wdo, wdg)):
        assert np.abs(a - b).max() <= 1e-12 * max(np.abs(wo).max(), np.abs(a).max())
    ch, cv = o.cuts()
    np.testing.assert_array_equal(g.cut_mask("h"), ch.astype(bool))
    np.testing.assert_array_equal(g.cut_mask("v"), cv.astype(bool))
    ends = [(o.history(), g.history(cap=133))] + ([(o.history_left(), g.history_left(cap=133))] if deg != 118.0 else [])
    for ho, hg in ends:
        for k in ("tip_q", "tip_yq", "npairs"):
            np.testing.assert_array_equal(hg[k], ho[k])
        np.testing.assert_allclose(hg["K"], ho["K"], rtol=0, atol=1e-9 * np.abs(ho["K"]).max())

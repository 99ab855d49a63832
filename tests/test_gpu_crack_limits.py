"""The crack step at the ends of its parameters' ranges: critical values that
1 / K_C or K / K_C does not fit a double for, speeds near that of shear waves,
and fields far below FP32's range."""
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


def _problem(nx, ny, scale_mu=1.0, scale_u=1.0, lattice="D2Q5", **crack):
    p = W.base_problem(nx, ny)
    p["mu"], p["rho"] = p["mu"] * scale_mu, p["rho"] * scale_mu
    p["hist_cap"] = 256
    crack = dict({"x_tip": nx / 4}, **crack)
    p = W.with_crack(p, mode="kcrit", y=float(ny // 2), **crack)
    p["loads"] = [{"edge": e, "kind": "linear", "amp": s * 1e-3 * scale_u, "t": 25.0} for e, s in (("bottom", -1), ("top", 1))]
    return dict(p, lattice=lattice)


def _run(lbm, p, storage, chunks, scale_u=1.0):
    lat = lbm.Lattice(p, storage)
    w0, wd0 = W.random_state(p["nx"], p["ny"], 11)
    lat.set_fields(w0 * scale_u, wd0 * scale_u)
    for n in chunks:
        lat.step(n)
    n = sum(chunks)
    two = p["crack"].get("two_tips") and "y" in p["crack"]
    h = [lat.history(n)] + ([lat.history_left(n)] if two else [])
    out = (*lat.fields(), lat.cut_mask("v"), *(d[k] for d in h for k in sorted(d))), lat.crack_state()
    lat.close()
    return out


def _same(a, b):
    for x, y in zip(a[0], b[0]):
        np.testing.assert_array_equal(x, y)
    assert a[1] == b[1]


@pytest.mark.parametrize("K_C", [5e-324, 1e-310, 1e-300])
@pytest.mark.parametrize("storage,lattice", [("f32", "D2Q5"), ("f64", "D2Q5"), ("f32_f16", "D2Q5"), ("f32", "D2Q9")])
def test_smallest_critical_values(gpu, K_C, storage, lattice):
    """K far above K_C: v_max, as at any K_C that far below K."""
    p, q = (_problem(300, 90, K_C=k, two_tips=True, x_start=60.0, lattice=lattice) for k in (K_C, 1e-200))
    ref = _run(gpu, q, storage, [1] * 50)
    assert ref[1]["v"] == p["crack"]["v_max"]
    _same(_run(gpu, p, storage, [50]), ref)
    _same(_run(gpu, p, storage, [1] * 50), ref)


@pytest.mark.parametrize("K_C", [5e-324, 1e-310, 1e-300])
@pytest.mark.parametrize("two", [False, True])
def test_smallest_critical_values_any_direction(gpu, K_C, two):
    got = []
    for k in (K_C, 1e-200):
        p = W.base_problem(200, 120, bc_mode="bounceback")
        p["hist_cap"] = 256
        p = W.with_line_crack(p, mode="kcrit", start=(60.3, 50.2), tip=(90.1, 61.7), K_C=k, two_tips=two)
        p["loads"] = [{"edge": "top", "kind": "linear", "amp": 1e-3, "t": 25.0}]
        got.append(_run(gpu, p, "f32", [50]))
    assert got[1][1]["v"] == 0.85
    _same(*got)


@pytest.mark.parametrize("r0", [0.6, 1.0, 2.0])
@pytest.mark.parametrize("v_max", [0.92, 0.95, 0.99])
def test_fast_ends(gpu, r0, v_max):
    p = _problem(900, 90, K_C=2e-7, v_max=v_max, r0=r0, x_start=430.2, x_tip=460.7, two_tips=True)
    _same(_run(gpu, p, "f32", [230]), _run(gpu, p, "f32", [1] * 230))


@pytest.mark.parametrize("K_C", [3e-5, 1.2e-4])
def test_fields_below_fp32(gpu, K_C):
    """A problem scaled by powers of two gives the scaled results, also where its
    jumps are no FP32 numbers: ends rest and grow in the same steps."""
    su, sm = 2.0 ** -150, 2.0 ** 100
    a = _run(gpu, _problem(150, 90, K_C=K_C), "f64", [120])
    b = _run(gpu, _problem(150, 90, scale_mu=sm, scale_u=su, K_C=K_C * sm * su), "f64", [120], su)
    assert a[1]["tip_q"] > int(150 / 4 * 2.0 ** 32)   # it grows
    assert a[1]["tip_q"] == b[1]["tip_q"]
    for x, y in zip(a[0][:2], b[0][:2]):
        np.testing.assert_array_equal(x * su, y)
    np.testing.assert_array_equal(a[0][2], b[0][2])

"""Passes of several time steps against single steps: the same arithmetic per
site, so fields, masks, crack states and histories agree bit for bit.  A run
of n steps in one call goes through passes (pairs of up to eight steps each,
the rest single steps); n calls of one step never do."""
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


def _strip(nx, ny, mode="prescribed", bc="macroscopic", edges=("free", "free", "dirichlet", "dirichlet"), jc=None,
           tip=None, start=0.0, u0=1e-3, **crack):
    p = W.base_problem(nx, ny, bc_mode=bc, edges=edges)
    p["hist_cap"] = 512
    if mode:
        p = W.with_crack(p, mode=mode, y=float(ny // 2 if jc is None else jc), x_start=start,
                         x_tip=nx / 4 if tip is None else tip, **crack)
    loads = []
    for k, e in enumerate(("left", "right", "bottom", "top")):
        if edges[k] == "dirichlet":
            kind = ("linear", "sin2", "halfsine", "const")[k]
            loads.append({"edge": e, "kind": kind, "amp": (-1) ** k * u0, "t": 25.0})
    p["loads"] = loads
    return p


# sizes at which a tile is whole, one vector or one row over, and thin
SIZES = [(24, 20), (97, 41), (128, 128), (129, 66), (240, 130), (241, 63), (352, 200), (1001, 97)]
KC = 0.02 * 0.25 * 1e-3 * 2


def cases():
    out = []
    for k, (nx, ny) in enumerate(SIZES):
        out.append((f"prescribed_{nx}x{ny}", _strip(nx, ny, v_rel=0.6), "f32", 37 + k))
        out.append((f"kcrit_{nx}x{ny}", _strip(nx, ny, mode="kcrit", K_C=KC), "f32", 50 - k))
        out.append((f"bb_periodic_{nx}x{ny}", _strip(nx, ny, bc="bounceback", v_rel=0.5,
                    edges=("periodic", "periodic", "dirichlet", "free"), start=nx * 0.7, tip=nx * 0.95), "f32", 48))
    for st in ("f64", "f32_bf16", "f32_f16", "f32_lf"):
        out.append((f"kcrit_{st}", _strip(300, 150, mode="kcrit", K_C=KC), st, 61))
        out.append((f"two_{st}", _strip(500, 80, mode="kcrit", K_C=KC, start=200.0, tip=215.0, two_tips=True), st, 90))
        out.append((f"edges_{st}", _strip(300, 150, mode="kcrit", bc="macroscopic_edges", K_C=KC), st, 50))
    for tip in range(40, 140, 7):   # the tip at any place relative to the tiles' boundaries
        out.append((f"tip_{tip}", _strip(331, 60, mode="kcrit", tip=tip + 0.3, K_C=KC), "f32", 64))
        out.append((f"tips_{tip}", _strip(480, 60, mode="kcrit", start=tip + 0.2, tip=tip + 31.9, K_C=KC, two_tips=True),
                    "f32", 64))
    for k, kc in enumerate((3e-5, 6e-5, 1.2e-4, 2.4e-4)):   # ends that rest, grow and rest again
        out.append((f"rest_{k}", _strip(300, 150, mode="kcrit", K_C=kc), "f32", 91))
        out.append((f"rest_two_{k}", _strip(300, 150, mode="kcrit", K_C=kc, start=140.2, tip=143.9, two_tips=True), "f32", 91))
        out.append((f"rest_wide_{k}", _strip(700, 300, mode="kcrit", K_C=kc, start=140.0, tip=181.0, two_tips=True,
                                             fit_width=3.5), "f64", 60))
    nine = []
    for nm, p, st, n in out:   # the same on nine velocities
        if st in ("f32", "f64"):
            nine.append((nm + "_q9", dict(p, lattice="D2Q9"), st, n))
    out += nine
    for k, kw in enumerate((dict(edges=("dirichlet",) * 4, bc="bounceback", v_rel=0.7, start=30.0),
                            dict(mode="kcrit", jc=12, K_C=KC), dict(mode=None),
                            dict(mode="prescribed", bc="macroscopic_edges", start=20.0, v_rel=0.5,
                                 edges=("dirichlet", "free", "free", "dirichlet")))):
        out.append((f"q9_{k}", dict(_strip(250, 110, **kw), lattice="D2Q9"), "f32", 50))
    out += [
        ("no_crack", _strip(300, 170, mode=None), "f32", 70),
        ("no_crack_edges", _strip(300, 170, mode=None, bc="macroscopic_edges"), "f32", 70),
        ("no_crack_small", _strip(33, 25, mode=None), "f64", 35),
        ("stationary_two", _strip(260, 90, mode="stationary", start=100.0, tip=180.0, two_tips=True), "f32", 40),
        ("crack_low", _strip(200, 120, mode="kcrit", jc=3, K_C=KC), "f32", 50),
        ("crack_high", _strip(200, 120, mode="prescribed", jc=117, v_rel=0.4), "f32", 50),
        ("dirichlet_all", _strip(270, 140, bc="bounceback", edges=("dirichlet",) * 4, v_rel=0.7, start=30.0), "f32", 50),
        ("edges_dirichlet_sides", _strip(250, 110, mode="prescribed", bc="macroscopic_edges", start=20.0, v_rel=0.5,
                                         edges=("dirichlet", "free", "free", "dirichlet")), "f32", 50),
        ("edge_crack_edges_f64", _strip(150, 90, mode="prescribed", bc="macroscopic_edges", v_rel=0.5), "f64", 33),
        ("clamped", _strip(200, 90, mode="prescribed", tip=180.0, v_rel=0.9), "f32", 100),
        ("wide_window", _strip(400, 90, mode="kcrit", K_C=KC, tip=150.0, fit_width=9.0, r0=3.0), "f32", 64),
        ("two_wide_windows", _strip(400, 90, mode="kcrit", K_C=KC, start=150.0, tip=158.0, two_tips=True, fit_width=5.0,
                                    r0=1.0), "f32", 64),
        ("far_window", _strip(400, 90, mode="kcrit", K_C=KC, tip=150.0, r_min=30.0), "f32", 64),
        ("many_tiles", _strip(3072, 1700, mode="kcrit", K_C=KC), "f32", 45),
        ("many_tiles_periodic", _strip(3001, 1777, bc="bounceback", v_rel=0.5, start=1000.0, tip=1200.0,
                                     edges=("periodic", "periodic", "dirichlet", "free")), "f32_f16", 41),
        ("many_tiles_no_crack", _strip(2900, 2000, mode=None), "f32_lf", 37),
        ("many_tiles_bf16", _strip(3500, 1500, v_rel=0.5), "f32_bf16", 26),
        ("tall", _strip(120, 1500, mode="kcrit", K_C=KC), "f32", 40),
        ("example", W.kcrit_centre_crack(), "f32", 200),
    ]
    for k, (nx, ny) in enumerate([(16, 20), (32, 25), (33, 31), (47, 60), (129, 128), (255, 257), (256, 256)]):   # FP64, one column a thread
        out.append((f"narrow_{nx}x{ny}", _strip(nx, ny, v_rel=0.7), "f64", 41 + k))
        out.append((f"narrow_rest_{nx}x{ny}", _strip(nx, ny, mode="stationary", bc="bounceback", start=nx * 0.3,
                                                     tip=nx * 0.6, two_tips=True), "f64", 40))
        out.append((f"narrow_bulk_{nx}x{ny}", _strip(nx, ny, mode=None), "f64", 43))
        out.append((f"narrow_periodic_{nx}x{ny}", _strip(nx, ny, bc="bounceback", v_rel=0.5, start=nx * 0.5, tip=nx * 0.8,
                                                         edges=("periodic", "periodic", "dirichlet", "free")), "f64", 45))
        out.append((f"narrow_kcrit_{nx}x{ny}", _strip(nx, ny, mode="kcrit", K_C=KC), "f64", 60))
    for tip in (110.2, 117.9, 119.5, 223.4):   # ends that a step moves over a tile boundary, towards either side
        out.append((f"over_{tip}", _strip(400, 80, v_rel=0.9, start=236.6 - tip / 2, tip=tip + 130, two_tips=True), "f32", 48))
        out.append((f"over_f64_{tip}", _strip(250, 80, v_rel=0.9, start=tip - 90, tip=tip, two_tips=True), "f64", 60))
    return out


@pytest.mark.parametrize("name,p,storage,n", cases(), ids=[c[0] for c in cases()])
def test_passes_equal_single_steps(gpu, name, p, storage, n):
    lbm = gpu
    w0, wd0 = W.random_state(p["nx"], p["ny"], 11)
    two = p["crack"].get("two_tips")
    got = []
    for chunks in ([n, 5, 19], [1] * (n + 24)):
        lat = lbm.Lattice(p, storage)
        lat.set_fields(w0, wd0)
        for c in chunks:
            lat.step(c)
        h = [lat.history(n + 24)] + ([lat.history_left(n + 24)] if two else [])
        st = [lat.crack_state()] + ([lat.crack_state_left()] if two else [])
        got.append((lat.fields(), lat.cut_mask("v"), h, st))
        lat.close()
    (f, m, h, st), (f1, m1, h1, st1) = got
    for a, b in zip(f, f1):
        np.testing.assert_array_equal(a, b)
    np.testing.assert_array_equal(m, m1)
    for a, b in zip(h, h1):
        for k in a:
            np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    assert st == st1


TAPES = ["macro_growth", "bb_growth", "bb_periodic", "all_dirichlet", "scaled_units", "no_crack", "wide_macro", "wide_bb"]


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("every", [0, 13])
@pytest.mark.parametrize("kind", TAPES)
def test_tape_passes_equal_single_steps(gpu, kind, every, storage):
    """The recording and the sweep in passes against single steps (a launch
    shape of the user's own keeps a lattice to those): the same losses and
    gradients, bit for bit (the load gradient's sum does not depend on the
    route)."""
    lbm = gpu
    T = 59
    p, loaded, w0, wd0, sens, tgt = W.adjoint_case(kind, T, seed=5, ns=23)
    got = []
    for rows in (0, 7):
        lat = lbm.Lattice(p, storage)
        lat.set_launch(rows)
        lat.set_fields(w0, wd0)
        tape = lbm.Tape(lat, sens, T, checkpoint_every=every)
        loss = tape.forward(tgt)
        mis = tape.misfits() if every == 0 else np.zeros(1)
        got.append((loss, mis, *tape.backward(device=False), *lat.fields(), lat.history(T)["K"]))
        tape.close()
        lat.close()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("storage", ["f32", "f32_bf16", "f32_f16", "f32_lf"])
def test_batch_passes_equal_single_steps(gpu, storage):
    """A batch of uneven lattices in passes (pairs of 8, 4 and 2 steps, then
    single ones) against the same lattices stepped alone, one step a call."""
    lbm = gpu
    probs = [_strip(97, 41, v_rel=0.6), _strip(300, 150, mode="kcrit", K_C=KC), _strip(33, 25, mode=None),
             _strip(500, 80, mode="kcrit", K_C=6e-5, start=200.0, tip=215.0, two_tips=True),
             _strip(260, 120, mode="kcrit", bc="macroscopic_edges", K_C=KC),
             _strip(240, 70, bc="bounceback", v_rel=0.5, edges=("periodic", "periodic", "dirichlet", "free"), start=150.0,
                    tip=200.0)]
    solo = [lbm.Lattice(p, storage) for p in probs]
    lats = [lbm.Lattice(p, storage) for p in probs]
    for k, (a, b) in enumerate(zip(solo, lats)):
        w0, wd0 = W.random_state(a.nx, a.ny, 30 + k)
        a.set_fields(w0, wd0)
        b.set_fields(w0, wd0)
    batch = lbm.Batch(lats)
    for n in (3, 16 + 8 + 4 + 3, 21):
        batch.step(n)
        for a in solo:
            for _ in range(n):
                a.step(1)
    for a, b in zip(solo, lats):
        for x, y in zip(a.fields(), b.fields()):
            np.testing.assert_array_equal(x, y)
        assert a.crack_state() == b.crack_state()
        ha, hb = a.history(60), b.history(60)
        for key in ha:
            np.testing.assert_array_equal(ha[key], hb[key])
    batch.close()

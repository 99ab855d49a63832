"""Passes, batches, row slabs and tapes against single steps where g, dt and dh
are no powers of two, so that every product of the update rounds: the roundings
of the update, the boundary rules and their adjoints are fixed in the source,
and the results agree bit for bit whatever kernel advances the lattice."""
import numpy as np
import pytest

from paper_2206_12412_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CS, RHO, DT, DH = 0.7, 1.3, 0.3, 0.5


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_12412_gb300 import lbm
    lbm.load_library()
    return lbm


def _strip(nx, ny, mode="prescribed", bc="macroscopic", edges=("free", "free", "dirichlet", "dirichlet"), tip=None,
           start=0.0, u0=1e-3, lattice="D2Q5", dh=DH, dt=DT, cs=CS, rho=RHO, **crack):
    p = W.base_problem(nx, ny, bc_mode=bc, edges=edges, cs=cs, rho=rho, dh=dh, dt=dt)
    p["hist_cap"] = 512
    if mode:
        crack = dict({"fit_width": dh, "r0": 2.0 * dh}, **crack)
        p = W.with_crack(p, mode=mode, y=(ny // 2) * dh, x_start=start * dh, x_tip=(nx / 4 if tip is None else tip) * dh,
                         **crack)
    p["loads"] = [{"edge": e, "kind": ("linear", "sin2", "halfsine", "const")[k], "amp": (-1) ** k * u0, "t": 25.0 * dt}
                  for k, e in enumerate(("left", "right", "bottom", "top")) if edges[k] == "dirichlet"]
    return dict(p, lattice=lattice)


KC = 2e-5
FORMS = {
    "prescribed": dict(v_rel=0.6),
    "kcrit": dict(mode="kcrit", K_C=KC),
    "two_pairs": dict(mode="kcrit", K_C=KC, fit_width=1.0),
    "two_ends": dict(mode="kcrit", K_C=KC, start=110.0, tip=131.0, two_tips=True),
    "periodic": dict(bc="bounceback", v_rel=0.5, edges=("periodic", "periodic", "dirichlet", "free"), start=200.0, tip=270.0),
    "edges": dict(mode="kcrit", bc="macroscopic_edges", K_C=KC),
    "edges_dirichlet": dict(bc="macroscopic_edges", v_rel=0.5, start=20.0, edges=("dirichlet", "free", "free", "dirichlet")),
    "no_crack_edges": dict(mode=None, bc="macroscopic_edges"),
}
STORAGES = ["f64", "f32", "f32_bf16", "f32_f16", "f32_lf"]


def cases():
    out = [(f"{nm}_{st}", _strip(*size, **kw), st, 47) for nm, kw in FORMS.items() for st in STORAGES
           for size in [(300, 150)]]
    out += [(f"{nm}_{st}_q9", _strip(300, 150, lattice="D2Q9", **kw), st, 47) for nm, kw in FORMS.items()
            for st in ("f64", "f32")]
    out += [(f"narrow_{nm}", _strip(130, 70, **FORMS[nm]), "f64", 47) for nm in ("prescribed", "kcrit", "edges")]
    out += [(f"wide_{st}", _strip(3001, 1201, **FORMS["kcrit"]), st, 30) for st in STORAGES[1:]]
    return out


def _state(lat, n, two):
    h = [lat.history(n)] + ([lat.history_left(n)] if two else [])
    st = [lat.crack_state()] + ([lat.crack_state_left()] if two else [])
    return lat.fields(), lat.cut_mask("v"), h, st


def _same(a, b):
    for x, y in zip(a[0], b[0]):
        np.testing.assert_array_equal(x, y)
    np.testing.assert_array_equal(a[1], b[1])
    for x, y in zip(a[2], b[2]):
        for k in x:
            np.testing.assert_array_equal(x[k], y[k], err_msg=k)
    assert a[3] == b[3]


def run_case(lbm, p, storage, chunks):
    w0, wd0 = W.random_state(p["nx"], p["ny"], 11)
    lat = lbm.Lattice(p, storage)
    lat.set_fields(w0, wd0)
    for c in chunks:
        lat.step(c)
    out = _state(lat, sum(chunks), p["crack"].get("two_tips"))
    lat.close()
    return out


@pytest.mark.parametrize("name,p,storage,n", cases(), ids=[c[0] for c in cases()])
def test_passes_equal_single_steps(gpu, name, p, storage, n):
    _same(run_case(gpu, p, storage, [n, 5]), run_case(gpu, p, storage, [1] * (n + 5)))


@pytest.mark.parametrize("storage", STORAGES)
def test_batch_equals_lattices_alone(gpu, storage):
    lbm = gpu
    probs = [_strip(300, 150, **FORMS[k]) for k in ("prescribed", "kcrit", "periodic", "edges")]
    solo, lats = ([lbm.Lattice(p, storage) for p in probs] for _ in range(2))
    for k, (a, b) in enumerate(zip(solo, lats)):
        w0, wd0 = W.random_state(a.nx, a.ny, 30 + k)
        a.set_fields(w0, wd0)
        b.set_fields(w0, wd0)
    batch = lbm.Batch(lats)
    for n in (3, 31):
        batch.step(n)
        for a in solo:
            for _ in range(n):
                a.step(1)
    for a, b in zip(solo, lats):
        _same(_state(a, 34, False), _state(b, 34, False))
    batch.close()


@pytest.mark.parametrize("storage", STORAGES)
def test_slabs_equal_lattice(gpu, storage):
    lbm = gpu
    p = _strip(300, 150, **FORMS["kcrit"])
    w0, wd0 = W.random_state(300, 150, 11)
    lat, dec = lbm.Lattice(p, storage), lbm.Decomp(p, 3, storage)
    for x in (lat, dec):
        x.set_fields(w0, wd0)
        x.step(30)
    for a, b in zip(lat.fields(), dec.fields()):
        np.testing.assert_array_equal(a, b)
    lat.close()
    dec.close()


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("kind", ["macro_growth", "bb_growth", "bb_periodic", "all_dirichlet", "no_crack", "wide_macro"])
def test_tape_passes_equal_single_steps(gpu, kind, storage):
    lbm = gpu
    T = 59
    p, _, w0, wd0, sens, tgt = W.adjoint_case(kind, T, seed=5, ns=23)
    p = dict(p, dt=0.7, mu=p["mu"] * 1.37, rho=p["rho"] * 0.9)
    got = []
    for rows in (0, 7):
        lat = lbm.Lattice(p, storage)
        lat.set_launch(rows)
        lat.set_fields(w0, wd0)
        tape = lbm.Tape(lat, sens, T)
        loss = tape.forward(tgt)
        got.append((loss, tape.misfits(), *tape.backward(device=False), *lat.fields(), lat.history(T)["K"]))
        tape.close()
        lat.close()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)

"""Field copies at shapes and addresses off the usual ones: every value comes
back as it was set, through host and device memory of the caller's."""
import numpy as np
import pytest

from paper_2206_12412_gb300 import _abi as A
from paper_2206_12412_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STORAGES = ["f64", "f32", "f32_bf16", "f32_f16", "f32_lf"]


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_12412_gb300 import lbm
    lbm.load_library()
    return lbm


def _values(ny, nx, storage, seed):
    """Small whole numbers, which every storage holds exactly (w and wdot: w - dt
    wdot is exact as well)."""
    return np.random.default_rng(seed).integers(-100, 101, (ny, nx)).astype(np.float64 if storage == "f64" else np.float32)


@pytest.mark.parametrize("storage", STORAGES)
def test_tall_lattice_round_trip(gpu, storage):
    """More rows than 65535 blocks of 16, the highest grid."""
    import torch
    nx, ny = 9, 65535 * 16 + 17
    lat = gpu.Lattice(W.base_problem(nx, ny, edges=("free",) * 4), storage)
    if storage == "f32_f16":
        gpu.lbm_set_wd_scale(lat.h, 1.0)
    for device in (True, False):
        w, wd = _values(ny, nx, storage, 1 + device), _values(ny, nx, storage, 3 + device)
        lat.set_fields(*((torch.from_numpy(a).cuda() for a in (w, wd)) if device else (w, wd)))
        for got, want in zip(lat.fields(), (w, wd)):
            np.testing.assert_array_equal(got, want)
        out = lat.fields_device()
        torch.cuda.synchronize()
        for got, want in zip(out, (w, wd)):
            np.testing.assert_array_equal(got.cpu().numpy(), want)
    lat.close()


@pytest.mark.parametrize("offset", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("nx", [64, 61])
@pytest.mark.parametrize("storage", STORAGES)
def test_device_memory_at_any_address(gpu, storage, nx, offset):
    """Device arrays that start `offset` bytes into an allocation, off the elements'
    alignment among them."""
    import torch
    ny = 33
    lat = gpu.Lattice(W.base_problem(nx, ny), storage)
    if storage == "f32_f16":
        gpu.lbm_set_wd_scale(lat.h, 1.0)
    want = [_values(ny, nx, storage, s) for s in (5, 6)]
    raw = torch.zeros(2, ny * nx * want[0].itemsize + 32, dtype=torch.uint8, device="cuda")
    size = want[0].nbytes
    for k, a in enumerate(want):
        raw[k, offset:offset + size] = torch.from_numpy(a.view(np.uint8).reshape(-1)).cuda()
    torch.cuda.synchronize()
    for k, which in enumerate(("w", "wdot")):
        gpu.lbm_set_fields(lat.h, A.FIELD[which], raw[k].data_ptr() + offset, True, lat.dtype_code)
    lat.sync()
    for got, a in zip(lat.fields(), want):
        np.testing.assert_array_equal(got, a)
    raw.zero_()
    torch.cuda.synchronize()
    for k, which in enumerate(("w", "wdot")):
        gpu.lbm_fields(lat.h, A.FIELD[which], raw[k].data_ptr() + offset, True, lat.dtype_code)
    lat.sync()
    back = raw.cpu().numpy()
    for k, a in enumerate(want):
        np.testing.assert_array_equal(back[k, offset:offset + size], a.view(np.uint8).reshape(-1))
        assert not back[k, :offset].any() and not back[k, offset + size:].any()
    lat.close()

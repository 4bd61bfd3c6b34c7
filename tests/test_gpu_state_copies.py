"""State import and export through device arrays: the kernels read and write the caller's arrays
themselves where they can reach them (aligned device memory), and through staging copies elsewhere
(host memory, arrays that are not aligned to their element size). Either way the same values arrive."""
import numpy as np
import pytest

from tests._pic import P, make_cfg

pytestmark = pytest.mark.gpu

REALS = ("ox", "oy", "oz", "dux", "duy", "duz", "w")


def _names(cfg):
    return [n for n in ("cell", "species", *REALS, "id") if (cfg.ndim == 3 or n != "oy") and (cfg.sigma_perp > 0 or n != "w")]


def _dtype(n, T):
    return np.uint32 if n == "id" else np.int32 if n in ("cell", "species") else T


def _on_device(a, shift):
    """A device copy of a, `shift` bytes past an aligned address, with its torch buffer."""
    import torch

    raw = torch.zeros(a.nbytes + 16, dtype=torch.uint8, device="cuda")
    raw[shift:shift + a.nbytes] = torch.from_numpy(a.view(np.uint8).reshape(-1).copy()).cuda()
    return raw


def _state(where, arrays, n, shift=0):
    s = P.make_state(where, None, None)
    s.np = n
    for k, a in arrays.items():
        setattr(s, k, a.ctypes.data if isinstance(a, np.ndarray) else a.data_ptr() + shift)
    return s


# sizes around the export's blocks of 256 cells: fewer, exactly one, one more, many; empty cells and bins
@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("ndim,nx,ny,nz", [(2, 7, 1, 9), (2, 16, 1, 16), (2, 257, 1, 3), (3, 12, 10, 14)])
@pytest.mark.parametrize("shift", [0, 2])
def test_state_through_device_arrays(ndim, nx, ny, nz, precision, shift):
    import torch

    cfg = make_cfg(ndim=ndim, nx=nx, ny=ny, nz=nz, precision=precision, ppc=4, sigma_perp=3.0 if ndim == 3 else 0.0)
    T = np.float32 if precision == 0 else np.float64
    rng = np.random.default_rng(3)
    ncell = nx * ny * nz
    counts = rng.integers(0, 9, size=(2, ncell))
    counts[:, ::5] = 0
    cell = np.concatenate([np.repeat(np.arange(ncell), c) for c in counts]).astype(np.int32)
    n = len(cell)
    a = {"cell": cell, "species": np.repeat([0, 1], counts.sum(axis=1)).astype(np.int32), "id": np.arange(n, dtype=np.uint32)}
    for k in REALS:
        a[k] = rng.uniform(0.0, 0.999, n).astype(T)
    a = {k: np.ascontiguousarray(a[k]) for k in _names(cfg)}
    perm = rng.permutation(n)  # any order may be imported
    h = P.pic_create(cfg)
    try:
        dev = {k: _on_device(v[perm], shift) for k, v in a.items()}
        torch.cuda.synchronize()
        P.pic_set_state(h, _state(P.PIC_DEVICE, dev, n, shift))
        host = {k: np.zeros(n + 5, dtype=_dtype(k, T)) for k in _names(cfg)}
        s = P.pic_get_state(h, _state(P.PIC_HOST, host, n + 5))
        assert s.np == n
        out = {k: _on_device(np.zeros(n, dtype=_dtype(k, T)), shift) for k in _names(cfg)}
        torch.cuda.synchronize()
        s = P.pic_get_state(h, _state(P.PIC_DEVICE, out, n, shift))
        assert s.np == n
        key = host["species"][:n].astype(np.int64) * ncell + host["cell"][:n]
        assert np.all(np.diff(key) >= 0)  # by species, then by cell
        order = np.argsort(host["id"][:n])
        for k in _names(cfg):
            got = out[k].cpu().numpy()[shift:shift + n * host[k].itemsize].copy().view(host[k].dtype)
            np.testing.assert_array_equal(got, host[k][:n], err_msg=k)
            np.testing.assert_array_equal(host[k][:n][order], a[k], err_msg=k)
        e = P.pic_energy(h)
        u0 = np.sqrt(cfg.gamma ** 2 - 1)
        u2 = a["dux"].astype(np.float64) ** 2 + a["duy"].astype(np.float64) ** 2 + (T(u0).astype(np.float64) + a["duz"].astype(np.float64)) ** 2
        w = a["w"].astype(np.float64) if "w" in a else float(T(0.3868 ** 2 / 8))
        assert abs(e["k"] - np.sum(w * (u2 / (1 + np.sqrt(1 + u2))))) <= 1e-13 * e["k"] + 1e-300
        assert e["np"] == n
    finally:
        P.pic_destroy(h)


# field arrays at every alignment the copy kernel distinguishes (16 bytes, the element, less: the plain copies),
# lengths with and without a remainder of its 16-byte units, one and many blocks; one array given for several fields
@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("nx,nz", [(3, 5), (7, 9), (64, 64), (301, 517)])
@pytest.mark.parametrize("shift", [0, 8, 4, 2])
def test_fields_through_device_arrays(nx, nz, precision, shift):
    import torch

    cfg = make_cfg(nx=nx, nz=nz, precision=precision, ppc=1, init_beam=0)
    T = np.float32 if precision == 0 else np.float64
    names = ("ex", "ey", "ez", "bx", "by", "bz")
    rng = np.random.default_rng(4)
    f = {n: rng.normal(size=nx * nz).astype(T) for n in names}
    dev = {n: _on_device(f[n], shift) for n in names}
    out = {n: _on_device(np.zeros_like(f[n]), shift) for n in names}
    h = P.pic_create(cfg)
    try:
        P.pic_set_state(h, _state(P.PIC_DEVICE, dev, -1, shift))
        P.pic_get_state(h, _state(P.PIC_DEVICE, out, 0, shift))
        for n in names:
            raw = out[n].cpu().numpy()
            assert raw[shift:shift + f[n].nbytes].tobytes() == f[n].tobytes(), n
            assert not raw[:shift].any() and not raw[shift + f[n].nbytes:].any(), n
        one = _on_device(np.zeros_like(f["ex"]), shift)
        P.pic_get_state(h, _state(P.PIC_DEVICE, {n: one for n in names}, 0, shift))
        torch.cuda.synchronize()
        assert one.cpu().numpy()[shift:shift + f["bz"].nbytes].tobytes() == f["bz"].tobytes()  # the last one stays
    finally:
        P.pic_destroy(h)

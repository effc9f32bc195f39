"""State import, export and macroscopic fields on device arrays: the
conversions between double and the storage types against numpy's, the integer
sums of the density and velocity against exactly rounded sums, and arrays on
the device against arrays on the host."""

import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TORCH_DT = {"fp64": "float64", "fp32": "float32", "fp16": "float16", "bf16": "bfloat16"}
NP_DT = {"fp64": np.float64, "fp32": np.float32, "fp16": np.float16}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g

    g.build()


def solver(storage, Q=19, dims=(37, 5, 7), bc_z=0, rho0=1.0, bufs=None, streaming="aa"):
    from paper_2502_20049_gb300 import psm

    nx, ny, nz = dims
    return psm.Solver(psm.SolverConfig(nx, ny, nz, Q=Q, storage=storage, streaming=streaming, bc_z=bc_z, rho0=rho0,
                                       u_in=(0.01, 0.0, 0.03)), buffers=bufs, keep=bufs is not None)


def awkward(n, dt, seed):
    """Doubles around every kind of rounding to dt: ties, near ties, subnormals, the largest values, zeros."""
    r = np.random.default_rng(seed)
    p = {np.float64: 52, np.float32: 23, np.float16: 10}[dt]
    lo, hi = {np.float64: (-300, 300), np.float32: (-152, 129), np.float16: (-27, 17)}[dt]
    m = 1.0 + r.integers(0, 1 << p, n) * 2.0 ** -p
    tail = r.choice([0.0, 0.5, 0.5 + 2.0 ** -8, 0.5 - 2.0 ** -8, 0.25, 0.75], n) * 2.0 ** -p
    x = np.ldexp(m + tail, r.integers(lo, hi, n)) * r.choice([-1.0, 1.0], n)
    x[r.random(n) < 0.05] = 0.0
    x[r.random(n) < 0.02] = -0.0
    x[:4] = [np.inf, -np.inf, np.nan, np.ldexp(1.0, hi)]
    return x


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("dims", [(37, 5, 7), (256, 3, 2)])
def test_import_rounds_and_export_widens_like_numpy(storage, dims):
    """With rho0 = 1e-300 the shift vanishes beside every value, so an imported
    double is stored as its rounding to the storage type and exported as it is."""
    import torch

    dt = NP_DT[storage]
    sol = solver(storage, dims=dims, rho0=1e-300)
    x = awkward(int(np.prod(sol.shape)), dt, 3).reshape(sol.shape)
    with np.errstate(over="ignore"):
        want = x.astype(dt)
    dev = torch.from_numpy(x).cuda()
    sol.set_state(dev)
    raw = torch.empty(sol.shape, dtype=getattr(torch, TORCH_DT[storage]), device="cuda")
    got = sol.get_pdfs(raw).cpu().numpy()
    nz = x != 0
    assert np.array_equal(got[nz], want[nz], equal_nan=True)
    assert np.all(np.abs(got[~nz].astype(np.float64)) <= 1e-300)
    out = torch.empty(sol.shape, dtype=torch.float64, device="cuda")
    back = sol.get_state(out).cpu().numpy()
    keep = np.isfinite(want) & (np.abs(want) > 1e-280)
    assert np.array_equal(back[keep], want[keep].astype(np.float64))
    # the staged path (host arrays) gives the same bits
    assert np.array_equal(sol.get_state(), back, equal_nan=True)
    assert np.array_equal(sol.get_pdfs(), got, equal_nan=True)
    sol.set_state(x)
    assert np.array_equal(sol.get_pdfs(), got, equal_nan=True)


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16", "fp64"])
@pytest.mark.parametrize("Q", [19, 27])
def test_macroscopic_against_exact_sums(storage, Q):
    """Density and velocity from exactly rounded sums (math.fsum): rho is one
    rounding from exact (below FP64 storage), u at most four: j rounded once,
    rho once, the quotient by less than two."""
    import torch

    r = np.random.default_rng(7)
    dims = (33, 9, 5)
    n = int(np.prod(dims))
    f = r.standard_normal((Q, n)) * 0.01
    f[:, n // 3:2 * n // 3] *= 2.0 ** r.integers(-18, 1, (Q, n // 3))          # wide ranges within a cell
    f[:, 2 * n // 3:] *= 2.0 ** r.integers(-13 if storage == "fp16" else -90, 4, (1, n - 2 * n // 3))  # across cells
    f[:, 5] = 0.0
    f[:, 7] = 0.0
    f[3, 7] = 0.25
    dt = getattr(torch, TORCH_DT[storage])
    buf = torch.from_numpy(f).to(dt).reshape(Q, dims[2], dims[1], dims[0]).cuda()
    sol = solver(storage, Q, dims, bufs=[buf])
    rho = torch.empty((dims[2], dims[1], dims[0]), dtype=torch.float64, device="cuda")
    u = torch.empty((dims[2], dims[1], dims[0], 3), dtype=torch.float64, device="cuda")
    sol.macroscopic(rho, u)
    rho, u = rho.cpu().numpy().reshape(-1), u.cpu().numpy().reshape(-1, 3)
    from paper_2502_20049_gb300 import psm

    c, _, _ = psm.lattice_velocities(Q)
    g = buf.cpu().double().numpy().reshape(Q, n)
    eps = 2.0 ** -53
    for k in range(n):
        wr = math.fsum([1.0] + list(g[:, k]))
        big = np.abs(g[:, k]).sum()
        # FP64 storage sums in FP64: Q roundings of partial sums at most `big` in size
        tr = 2 * eps * abs(wr) if storage != "fp64" else (2 * abs(wr) + Q * big) * eps
        assert abs(rho[k] - wr) <= tr, k
        for a in range(3):
            j = math.fsum(g[i, k] * c[i, a] for i in range(Q))
            tu = 4 * eps * abs(j / wr) if storage != "fp64" else (4 * abs(j / wr) + 2 * Q * big / wr) * eps
            assert abs(u[k, a] - j / wr) <= tu, (k, a)
    hr, hu = sol.macroscopic()
    assert np.array_equal(hr.reshape(-1), rho) and np.array_equal(hu.reshape(-1, 3), u)


def test_macroscopic_of_non_finite_and_extreme_cells():
    """Cells outside the integer sums' range take FP64 sums: infinities and NaN
    come out as such, subnormal and huge populations keep their values."""
    import torch

    dims, Q = (32, 2, 2), 19
    f = torch.full((Q, 2, 2, 32), 0.001, dtype=torch.float32)
    f[:, 0, 0, 0] = 0.0
    f[4, 0, 0, 0] = float("inf")
    f[:, 0, 0, 1] = float("nan")
    f[:, 0, 0, 2] = 1e-40
    f[:, 0, 0, 3] = 3e37
    sol = solver("fp32", Q, dims, bufs=[f.cuda()])
    rho, u = sol.macroscopic()
    assert np.isinf(rho[0, 0, 0]) and np.isnan(rho[0, 0, 1]) and np.isnan(u[0, 0, 1]).all()
    assert rho[0, 0, 2] == 1.0 and np.abs(u[0, 0, 2]).max() <= 1e-38
    assert abs(rho[0, 0, 3] / (19 * float(np.float32(3e37))) - 1) < 1e-14 and np.isfinite(u[0, 0, 3]).all()
    assert np.isfinite(rho[0, 0, 4:]).all() and np.isfinite(u[0, 0, 4:]).all()


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("dims,bc_z", [((37, 5, 7), 1), ((1, 1, 1), 1), ((3, 1, 2), 1), ((64, 8, 3), 0)])
@pytest.mark.parametrize("odd", [0, 1])
def test_uniform_state_equals_the_field_state(storage, dims, bc_z, odd):
    """The filled uniform equilibrium against the per-cell import of the same
    field, in both layouts of the AA pattern (odd: swapped)."""
    a, b = solver(storage, 27, dims, bc_z), solver(storage, 27, dims, bc_z)
    for s in (a, b):
        s.step(odd)
    a.init_equilibrium(1.02, (0.01, -0.02, 0.03))
    shape = a.shape[1:]
    b.init_equilibrium_field(np.full(shape, 1.02), np.tile(np.array([0.01, -0.02, 0.03]), shape + (1,)))
    assert np.array_equal(a.get_state(), b.get_state())


def test_arrays_that_overlap_the_state_are_staged():
    """Export into, and import from, the solver's own buffer."""
    import torch

    buf = torch.zeros((19, 6, 4, 32), dtype=torch.float64, device="cuda")
    sol = solver("fp64", 19, (32, 4, 6), bufs=[buf])
    x = 0.03 + 0.01 * np.random.default_rng(1).random(sol.shape)
    sol.set_state(x)
    want = sol.get_state()
    sol.get_state(buf)  # natural layout: the buffer now holds the unshifted values
    assert np.array_equal(buf.cpu().numpy(), want)
    sol.set_state(buf)
    assert np.array_equal(sol.get_state(), want)


def macro_cells(storage):
    """Populations [19, cells] whose momentum lies far below the largest population of the cell, and per
    cell and axis whether its FP64 sum is exact (at most one value that does not cancel with the next)."""
    Q = 19
    dt = {"fp32": np.float32, "bf16": np.float32}[storage]
    f, exact = [], []
    for e in range(-110, -30, 3):       # f_0 alone above values of 2^e; opposite pairs are (1, 2), (3, 4), (5, 6)
        m = 1.2345678 if storage == "fp32" else 1.2421875
        a = np.zeros(Q, dt)
        a[0], a[3] = 0.01, m * 2.0 ** e
        f.append(a)
        exact.append((True, True, True))
        a = a.copy()
        a[1] = a[2] = 0.0078125          # cancels exactly on x
        a[5] = -m * 2.0 ** (e - 7)
        f.append(a)
        exact.append((True, True, True))
        a = a.copy()
        a[7:15] = (1 + np.arange(8) / 8) * 2.0 ** (e + np.arange(8) % 5) * (-1.0) ** np.arange(8)
        f.append(a)
        exact.append((False, False, False))
    return np.array(f).T.copy(), exact


@pytest.mark.parametrize("storage", ["fp32", "bf16"])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 9])
def test_macroscopic_keeps_momentum_far_below_the_largest_population(storage, scale):
    """A momentum made of populations 2^-110 to 2^-30 of the cell's largest (a rest population, or a pair
    that cancels): no digit may be lost.  Where the FP64 sum is exact, u is four roundings from exact
    (density, quotient); elsewhere each of the Q additions may round at the size of the populations that
    carry momentum on the axis (2 Q eps sum |f_i c_i|)."""
    import torch
    from paper_2502_20049_gb300 import psm

    Q = 19
    f, exact = macro_cells(storage)
    f = f * np.float32(scale)            # a scale of 2^9 makes the largest population exceed 2
    n = f.shape[1]
    buf = torch.from_numpy(f).to(getattr(torch, TORCH_DT[storage])).reshape(Q, 1, 1, n).cuda()
    sol = solver(storage, Q, (n, 1, 1), bufs=[buf])
    rho, u = sol.macroscopic()
    rho, u = rho.reshape(-1), u.reshape(-1, 3)
    c, _, _ = psm.lattice_velocities(Q)
    g = buf.cpu().double().numpy().reshape(Q, n)
    eps = 2.0 ** -53
    for k in range(n):
        wr = math.fsum([1.0] + list(g[:, k]))
        assert abs(rho[k] - wr) <= (2 * abs(wr) + Q * np.abs(g[:, k]).sum()) * eps, k
        for a in range(3):
            terms = [g[i, k] * c[i, a] for i in range(Q)]
            want = math.fsum(terms) / wr
            tol = 4 * eps * abs(want)
            if not exact[k][a]:
                tol += 2 * Q * eps * sum(map(abs, terms)) / wr
            assert abs(u[k, a] - want) <= tol, (k, a, u[k, a], want)


@pytest.mark.parametrize("at", [0, 100, 2200])
def test_density_and_velocity_into_overlapping_arrays(at):
    """A caller that wants the velocity alone may let the density array lie
    anywhere in the velocity's: the velocity is what stays."""
    import torch

    dims = (37, 5, 7)
    n = int(np.prod(dims))
    sol = solver("fp32", dims=dims)
    z, y, x = np.meshgrid(np.arange(7), np.arange(5), np.arange(37), indexing="ij")
    sol.init_equilibrium_field(1.0 + 0.01 * np.sin(0.3 * x + y), 0.02 * np.stack([np.sin(0.5 * x), np.cos(y + z), 0.1 * z], -1))
    _, want = sol.macroscopic()
    u = torch.empty((7, 5, 37, 3), dtype=torch.float64, device="cuda")
    sol.macroscopic(u.view(-1)[at:at + n], u)
    assert np.array_equal(u.cpu().numpy(), want)


@pytest.mark.parametrize("kind", ["managed", "pinned"])
def test_arrays_in_managed_and_pinned_memory(kind):
    """Managed memory takes the direct kernels, pinned host memory the staging
    chunk: the bits of an array on the device."""
    import ctypes

    import torch

    dims = (37, 5, 7)
    sol = solver("fp32", dims=dims)
    sol.init_equilibrium(1.02, (0.01, -0.02, 0.03))
    want = sol.get_state(torch.empty(sol.shape, dtype=torch.float64, device="cuda")).cpu().numpy()
    n = want.size
    if kind == "pinned":
        a = torch.empty(sol.shape, dtype=torch.float64).pin_memory()
        sol.get_state(a)
        got = a.numpy()
        sol.init_equilibrium(1.0, (0.0, 0.0, 0.0))
        sol.set_state(a)
    else:
        from paper_2502_20049_gb300 import psm

        rt = ctypes.CDLL("/usr/local/cuda/lib64/libcudart.so")
        p = ctypes.c_void_p()
        assert rt.cudaMallocManaged(ctypes.byref(p), ctypes.c_size_t(8 * n), ctypes.c_uint(1)) == 0
        psm.check(psm.lib().psm_get_state(sol._h, p))
        got = np.ctypeslib.as_array(ctypes.cast(p, ctypes.POINTER(ctypes.c_double)), shape=(n,)).reshape(want.shape).copy()
        sol.init_equilibrium(1.0, (0.0, 0.0, 0.0))
        psm.check(psm.lib().psm_set_state(sol._h, p))
        sol.synchronize()
        assert rt.cudaFree(p) == 0
    assert np.array_equal(got, want)
    assert np.array_equal(sol.get_state(), want)

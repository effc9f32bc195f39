"""The step kernels at the edges of their work split: rows shorter and longer
than a warp's 32 cells, rows with a remainder, one cell, grids on either side of
the switch to small blocks, and one to four bodies in the load reduction."""

import numpy as np
import pytest

from paper_2502_20049_gb300 import workloads as W

from helpers import ft_err, perm_lib_to_oracle, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g

    g.build()


def case(dims, storage, streaming, Q=19, nb=2, fluid="trt", bc_z=1, steps=5, s=2):
    nx, ny, nz = dims
    m = min(dims)
    shapes = [(W.ELLIPSOID, (0.3 * m + 0.6, 0.2 * m + 0.5, 0.2 * m + 0.4), s), (W.SPHERE, (0.15 * m + 0.5,), 3),
              (W.BOX, (0.7, 0.6, 0.8), 1), (W.SPHERE, (0.9,), 0)]
    bodies = [W.BodyCase(k, p, sd, (nx * (0.3 + 0.15 * i), ny * 0.5 + 0.1, nz * (0.6 - 0.1 * i)),
                         omega=(0.01, 0.02, 0.03 * (-1) ** i), v=(0.03, 0.0, 0.0)) for i, (k, p, sd) in enumerate(shapes[:nb])]
    return W.Case("shapes", nx, ny, nz, Q=Q, storage=storage, streaming=streaming, fluid=fluid, tau=0.65, solid=1,
                  weighting=1, bc_z=bc_z, u_in=(0.02, -0.01, 0.03), steps=steps, bodies=bodies)


@pytest.mark.parametrize("dims", [(1, 1, 1), (1, 5, 3), (31, 3, 4), (32, 4, 3), (33, 5, 7), (63, 2, 9), (65, 6, 5),
                                  (203, 7, 5), (300, 3, 4), (40, 40, 40)])
@pytest.mark.parametrize("streaming,bc_z", [("aa", 1), ("aa", 0), ("twogrid", 1)])
def test_ragged_rows_fp64_match_the_oracle(dims, streaming, bc_z):
    c = case(dims, "fp64", streaming, bc_z=bc_z, nb=1 + sum(dims) % 4)
    g, o = run_gpu(c), run_oracle(c)
    assert np.abs(g["f"] - o["f"][perm_lib_to_oracle(19)]).max() <= 1e-13
    assert ft_err(g, o) <= 1e-10


@pytest.mark.parametrize("dims", [(32, 32, 38), (64, 64, 9), (33, 31, 36), (95, 20, 20)])
@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("Q,streaming", [(19, "aa"), (27, "aa"), (19, "twogrid")])
def test_small_blocks_equal_whole_blocks(dims, storage, Q, streaming):
    """Small grids take blocks of 64 by themselves; forced plain loads keep blocks
    of 256.  The same cells in the same warps: states bit for bit, loads to the
    rounding of the FP64 sums' order."""
    from paper_2502_20049_gb300 import psm

    c = case(dims, storage, streaming, Q=Q, nb=4, steps=6)
    a, b = psm.Solver.from_case(c), psm.Solver.from_case(c)
    b.set_kernel_variant("plain")
    a.step(c.steps)
    b.step(c.steps)
    assert np.array_equal(a.get_state(), b.get_state())
    for k in range(4):
        fa, fb = a.force_torque(k), b.force_torque(k)
        # at most nwarps additions of partials whose sizes sum to at most nwarps times the largest total
        assert np.abs(fa - fb).max() <= 1e-12 * max(1.0, np.abs(fb).max())


@pytest.mark.parametrize("storage,streaming,dims", [("fp32", "aa", (64, 8, 12)), ("fp16", "twogrid", (33, 9, 7)),
                                                    ("fp64", "aa", (20, 11, 9))])
@pytest.mark.parametrize("n", [2, 15, 16, 17, 33])
def test_loads_of_many_steps_equal_those_of_single_steps(storage, streaming, dims, n):
    """A call of n steps sums its steps' loads together, a call of one in the step
    kernel: the same sums bit for bit, around the number of steps summed at once."""
    from paper_2502_20049_gb300 import psm

    c = case(dims, storage, streaming, nb=3)
    a, b = psm.Solver.from_case(c), psm.Solver.from_case(c)
    a.step(n)
    for _ in range(n):
        b.step(1)
    for k in range(3):
        fa = a.force_torque(k)
        assert np.abs(fa).max() > 0
        assert np.array_equal(fa, b.force_torque(k))


@pytest.mark.parametrize("dims", [(256, 16, 20), (64, 64, 40), (512, 6, 12), (128, 32, 24)])
@pytest.mark.parametrize("storage,fluid,Q", [("fp16", "cumulant", 19), ("bf16", "cumulant", 19), ("fp16", "trt", 19),
                                             ("bf16", "bgk", 27), ("fp16", "bgk", 27)])
@pytest.mark.parametrize("streaming", ["aa", "twogrid"])
def test_pairs_of_a_varying_flow_equal_plain_bitwise(dims, storage, fluid, Q, streaming):
    """x-neighbour pairs (packed arithmetic among them) against one cell per
    thread on a flow that differs in every cell, over more tiles than a block
    keeps in flight, with row ends and ghost planes: the same states bit for bit."""
    from paper_2502_20049_gb300 import psm

    c = case(dims, storage, streaming, Q=Q, fluid=fluid, nb=2, steps=5)
    nx, ny, nz = dims
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    rho = 1.0 + 0.01 * np.sin(0.37 * x + 0.21 * y - 0.5 * z)
    u = 0.03 * np.stack([np.sin(0.3 * x + 0.7 * y), np.cos(0.2 * y - 0.4 * z), np.sin(0.6 * z + 0.1 * x)], -1)
    a, b = psm.Solver.from_case(c), psm.Solver.from_case(c)
    a.set_kernel_variant("tma")
    b.set_kernel_variant("plain")
    for s in (a, b):
        s.init_equilibrium_field(rho, u)
        s.step(c.steps)
    assert np.array_equal(a.get_state(), b.get_state())


@pytest.mark.parametrize("dims,auto", [((32, 32, 32), "plain"), ((64, 64, 64), "tma"), ((37, 23, 19), "plain")])
def test_variant_names_the_kernel_that_runs_fp64(dims, auto):
    """FP64 grids of at most 256 cells per SM take plain loads under AUTO, larger
    ones of a TMA shape the TMA-staged kernel; forced variants are what was forced."""
    from paper_2502_20049_gb300 import psm

    s = psm.Solver(psm.SolverConfig(*dims, storage="fp64"))
    assert s.kernel_variant == auto
    s.set_kernel_variant("plain")
    assert s.kernel_variant == "plain"
    if dims[0] != 37:
        s.set_kernel_variant("tma")
        assert s.kernel_variant == "tma"
    s.set_kernel_variant("auto")
    assert s.kernel_variant == auto


@pytest.mark.parametrize("streaming", ["aa", "twogrid"])
def test_small_fp64_grid_with_the_tma_kernel_matches_the_oracle(streaming):
    """The TMA-staged FP64 kernel on a grid where AUTO takes plain loads; 17 steps: more than one sum of loads."""
    from paper_2502_20049_gb300 import psm

    c = case((64, 16, 12), "fp64", streaming, nb=3, steps=17)
    s = psm.Solver.from_case(c)
    s.set_kernel_variant("tma")
    s.step(c.steps)
    g = dict(f=s.get_state(), ft=np.stack([s.force_torque(b) for b in range(3)], axis=1))
    o = run_oracle(c)
    assert np.abs(g["f"] - o["f"][perm_lib_to_oracle(19)]).max() <= 1e-13
    assert ft_err(g, o) <= 1e-10


@pytest.mark.parametrize("storage,dims", [("fp32", (64, 16, 12)), ("fp16", (256, 8, 12)), ("fp64", (33, 12, 9))])
def test_steps_between_a_callers_kernels_on_its_stream(storage, dims):
    """psm_step on a side stream, its launches overlapped, between kernels of the
    caller on the same stream that write the PDF buffer before and read it after
    each call, without a synchronisation: as on the default stream with one."""
    import torch
    from paper_2502_20049_gb300 import psm

    c = case(dims, storage, "aa", nb=2)
    cfg = psm.SolverConfig(*dims, storage=storage, fluid="trt", tau=0.65, u_in=(0.02, -0.01, 0.03))
    dt = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16}[storage]
    fields = [(psm.voxelize(b.kind, b.params, b.s), b) for b in c.bodies]
    start = (0.01 * torch.rand((19,) + dims[::-1], generator=torch.Generator().manual_seed(3))).to(dt).cuda()

    def run(stream, wait):
        with torch.cuda.stream(stream):
            f = torch.zeros_like(start)
            sol = psm.Solver(cfg, buffers=[f], keep=True)
            for k, (g, b) in enumerate(fields):
                sol.set_geometry(k, g, np.array(b.Q0), b.R0, b.omega, b.v)
            seen = []
            for n in (1, 2, 3, 18):
                f.copy_(start + f * 0.5)
                if wait:
                    torch.cuda.synchronize()
                sol.step(n)
                seen.append(f.clone())
                if wait:
                    torch.cuda.synchronize()
            return [x.cpu() for x in seen], [sol.force_torque(k) for k in range(2)]

    a, fa = run(torch.cuda.Stream(), False)
    b, fb = run(torch.cuda.default_stream(), True)
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    for x, y in zip(fa, fb):
        assert np.array_equal(x, y)

"""The mesh voxeliser's work split: dense and sparse tiles, rows of several
passes, the crossing limit, and its argument checks on the GPU."""

import numpy as np
import pytest

from paper_2502_20049_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g

    g.build()


@pytest.mark.parametrize("s", [0, 1, 2, 3])
def test_dense_tiles_equal_oracle(oracle_mod, s):
    """Hundreds of triangles per tile: one thread per triangle."""
    from paper_2502_20049_gb300 import psm

    v, t = W.icosphere(3.3, 4, centre=(0.13, -0.07, 0.21))  # 5,120 triangles
    g = psm.voxelize_mesh(v, t, s)
    sub, lo = oracle_mod.voxelize_mesh(v, t, s)
    assert np.array_equal(g.lo, lo) and np.array_equal(g.subcells(), sub) and sub.sum() > 0


@pytest.mark.parametrize("length,s", [(31.0, 2), (127.0, 3), (130.0, 3), (300.0, 2), (700.0, 3)])
def test_long_rows_against_the_half_open_box(length, s):
    """A box is the sub-cells with centres in (x0, x1] x [y0, y1) x [z0, z1):
    rows from below one pass (1,024 sub-cells) to six."""
    from paper_2502_20049_gb300 import psm

    lo, hi = np.array([0.3, 0.45, 0.2]), np.array([0.3 + length, 3.4, 2.7])
    v, t = W.box_mesh(lo, hi)
    g = psm.voxelize_mesh(v, t, s)
    sub = g.subcells()
    n = 1 << s
    c = [g.lo[k] + (np.arange(sub.shape[2 - k]) + 0.5) / n for k in range(3)]
    q = [(x > np.float32(a)) & (x < np.float32(b)) for x, a, b in zip(c, lo, hi)]  # no centre on a face
    want = q[2][:, None, None] & q[1][None, :, None] & q[0][None, None, :]
    assert np.array_equal(sub.astype(bool), want)


@pytest.mark.parametrize("boxes,ok", [(128, True), (129, False)])
def test_crossing_limit(boxes, ok):
    """256 crossings along a row are counted, more are refused."""
    from paper_2502_20049_gb300 import psm

    v, t = W.merge_meshes(*[W.box_mesh((2.0 * i + 0.2, 0.1, 0.1), (2.0 * i + 1.1, 2.0, 2.0)) for i in range(boxes)])
    if ok:
        assert psm.voxelize_mesh(v, t, 0).subcells().sum() == boxes * 4
    else:
        with pytest.raises(psm.PSMError) as ei:
            psm.voxelize_mesh(v, t, 0)
        assert ei.value.code == -6


def test_bad_meshes_are_refused_on_the_gpu():
    from paper_2502_20049_gb300 import psm

    v, t = W.box_mesh((0, 0, 0), (2, 2, 2))

    def refused(v, t, text, s=1):
        with pytest.raises(psm.PSMError) as ei:
            psm.voxelize_mesh(v, t, s)
        assert ei.value.code == -1 and text in str(ei.value), str(ei.value)

    refused(v, t[:-1], "not closed")
    bad = t.copy()
    bad[3, 1] = 8
    refused(v, bad, "index out of range")
    bad[3, 1] = -1
    refused(v, bad, "index out of range")
    bad = t.copy()
    bad[0, 1] = bad[0, 0]
    refused(v, bad, "degenerate")
    for x in (np.nan, np.inf):
        w = v.copy()
        w[2, 1] = x
        refused(w, t, "non-finite")
    refused(v * np.float32(1e6), t, "extent")
    # an edge shared four times is even: two boxes joined along an edge
    a, b = W.box_mesh((0, 0, 0), (1.3, 1.2, 1.1)), W.box_mesh((1.3, 1.2, 0), (2.4, 2.3, 1.1))
    vv, tt = W.merge_meshes(a, b)
    uniq, inv = np.unique(vv, axis=0, return_inverse=True)
    assert psm.voxelize_mesh(uniq.astype(np.float32), inv.reshape(-1)[tt].astype(np.int32), 2).subcells().sum() > 0


def test_loose_triangles_are_refused_at_once_whatever_their_number():
    """Triangles without a common edge have three distinct edges each; 349,525
    of them are one edge short of 2^20, a power of two that a table of the edges
    must not be filled to (262,144 leave a quarter of it free)."""
    import time

    from paper_2502_20049_gb300 import psm

    def refuse(nt):
        v = np.random.default_rng(5).random((3 * nt, 3), dtype=np.float32)
        t = np.arange(3 * nt, dtype=np.int32).reshape(-1, 3)
        best = np.inf
        for _ in range(3):
            t0 = time.perf_counter()
            with pytest.raises(psm.PSMError, match="not closed"):
                psm.voxelize_mesh(v, t, 1)
            best = min(best, time.perf_counter() - t0)
        return best

    few, many = refuse(262144), refuse(349525)
    assert many <= 10 * few, (few, many)


@pytest.mark.parametrize("side", [1446, 1450])
def test_grids_of_many_tiles(side):
    """A thin box on either side of 2^17 tiles (362^2 and 363^2; more take their
    counts from an allocation of their own): faces on cell faces, so whole cells
    are inside or outside."""
    from paper_2502_20049_gb300 import psm

    v, t = W.box_mesh((0, 0, 0), (1, side, side))
    g = psm.voxelize_mesh(v, t, 2)
    w = g.words().reshape(side + 2, side + 2, 3)
    want = np.zeros_like(w)
    want[1:-1, 1:-1, 1] = np.iinfo(w.dtype).max
    assert np.array_equal(w, want)


def test_calls_that_grow_the_heap_take_about_as_long():
    """Results that are kept and freed in turn make the heap grow and shrink
    under the field; a call must not pay several times its own time for that."""
    import time

    from paper_2502_20049_gb300 import psm

    v, t = W.icosphere(60.0, 6)  # 81,920 triangles, a field of 123^3 words at s = 2
    held, took = [], []
    for k in range(16):
        t0 = time.perf_counter()
        g = psm.voxelize_mesh(v * np.float32(1 - 0.0005 * k), t, 2)
        took.append(time.perf_counter() - t0)
        held = (held + [g, g.words()])[-4:]
    took = sorted(took[4:])
    assert took[-1] <= 4 * took[len(took) // 2], took

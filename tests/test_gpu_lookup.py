"""Leaf lookup at its edges: leaves of levels 17 to 21, where the walk's
position is rarely certain and the mirrored frame meets lattice points, against
the oracle; and the coarse table in 64-bit entries (2^26 leaves or more)
against the search of all keys."""
import ctypes as C

import numpy as np
import pytest

import synth
from test_gpu_parity import _check_case
from tinytrees import D, leaf_boxes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_09882_gb300 as rt
    return rt


def _nested(targets, max_level, root_level=1):
    """Octree whose cells that hold a target (integer depth-21 points) are split down to max_level."""
    n = 1 << root_level
    todo = [(root_level, x, y, z, targets) for z in range(n) for y in range(n) for x in range(n)]
    leaves = []
    while todo:
        lev, x, y, z, t = todo.pop()
        sh = D - lev
        t = t[((t >> sh) == np.array([x, y, z])).all(axis=1)]
        if lev < max_level and t.shape[0]:
            todo += [(lev + 1, 2 * x + dx, 2 * y + dy, 2 * z + dz, t) for dz in (0, 1) for dy in (0, 1) for dx in (0, 1)]
        else:
            leaves.append((lev, x << sh, y << sh, z << sh))
    a = np.array(leaves, dtype=np.uint64)
    keys = synth.interleave(a[:, 1], a[:, 2], a[:, 3])
    order = np.argsort(keys)
    return keys[order], a[order, 0].astype(np.uint8)


@pytest.mark.parametrize("max_level", [17, 19, 20, 21])
@pytest.mark.parametrize("where", ["inside", "corner", "middle"])
def test_deepest_leaves(rt, max_level, where):
    """A cluster of leaves of the deepest level, inside the box, at its corners
    (first and last lattice cells) and around its centre planes; sources at
    leaf centres, corners, on faces and anywhere in the leaves."""
    rng = np.random.default_rng(3000 + max_level)
    at = {"inside": [[1234567, 700001, 1999999]], "corner": [[0, 0, 0], [(1 << D) - 200] * 3, [0, (1 << D) - 200, 0]],
          "middle": [[(1 << (D - 1)) - 100] * 3]}[where]
    targets = np.concatenate([np.array(p) + rng.integers(0, 200, size=(24, 3)) for p in at])
    keys, lev = _nested(targets, max_level)
    lo, hi = leaf_boxes(keys, lev)
    deep = np.flatnonzero(lev >= max_level - 2)
    pick = rng.choice(deep, size=min(48, deep.size), replace=False)
    mid = 0.5 * (lo[pick] + hi[pick])
    some = lo[pick] + (hi[pick] - lo[pick]) * rng.random((pick.size, 3))
    src = np.concatenate([mid, lo[pick], some, np.column_stack([lo[pick, 0], mid[:, 1], some[:, 2]]), rng.random((16, 3))])
    dens = rng.uniform(0.1, 10.0, size=(keys.shape[0], 2)).astype(np.float32)
    for nside in (1, 4):
        _check_case(rt, keys, lev, dens, src, nside, label=f"{where} {max_level} nside{nside}")


def test_wide_table(rt):
    """A box of 200^3 level-8 cells in leaves of level 9, some split to level 10
    and a few of those to 11: more than 2^26 leaves, single-level, mixed and outside
    cells, at the table level the build chooses and at shallower ones.  Columns
    bit for bit those of the call that searches all keys."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(9)
    g = torch.arange(400, device="cuda")
    cells = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), dim=-1).reshape(-1, 3)

    def spread(v):
        for s, m in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F), (4, 0x10C30C30C30C30C3),
                     (2, 0x1249249249249249)):
            v = (v | (v << s)) & m
        return v

    off = torch.tensor([[x, y, z] for z in (0, 1) for y in (0, 1) for x in (0, 1)], device="cuda")
    keys, levels = [], []
    for lev, share in ((9, 0.02), (10, 0.01), (11, 0.0)):
        split = torch.rand(cells.shape[0], generator=gen, device="cuda") < share
        c = cells[~split] << (D - lev)
        keys.append(spread(c[:, 0]) | (spread(c[:, 1]) << 1) | (spread(c[:, 2]) << 2))
        levels.append(torch.full((c.shape[0],), lev, dtype=torch.uint8, device="cuda"))
        cells = (2 * cells[split][:, None, :] + off).reshape(-1, 3)
    keys, order = torch.sort(torch.cat(keys))
    levels = torch.cat(levels)[order]
    assert keys.numel() >= 1 << 26
    del c, cells, order
    ext = (200 << (D - 8),) * 3
    dens = torch.rand((keys.numel(), 2), generator=gen, device="cuda")
    src = torch.rand((1500, 3), generator=gen, device="cuda", dtype=torch.float64) * (200 / 256)
    f = rt._lib.rt_trace_columns_noalloc
    P = C.c_void_p
    f.argtypes = [P, P, C.c_int64, P, C.c_int, P, C.c_int64, C.c_int, P, C.c_int, C.c_int, C.c_int, P, C.POINTER(rt.Stats), P]
    want = {}
    for mode in (rt.MODE_FP64, rt.MODE_F32_KAHAN):
        want[mode] = torch.empty((1500, 12, 2), device="cuda", dtype=torch.float64 if mode == rt.MODE_FP64 else torch.float32)
        st = rt.Stats()
        assert f(keys.data_ptr(), levels.data_ptr(), keys.numel(), (C.c_int32 * 3)(*ext), 11, src.data_ptr(), 1500, 1, dens.data_ptr(),
                 2, rt.F32, mode, want[mode].data_ptr(), C.byref(st), P(torch.cuda.current_stream().cuda_stream)) == 0
        assert st.status == 0
    try:
        for cap in (-1, 8, 6):
            rt.set_table_cap(cap)
            tree = rt.Octree(keys, levels, extent=ext)
            for mode, w in want.items():
                assert torch.equal(rt.trace_columns(tree, src, 1, dens, mode), w), (cap, mode)
            assert tree.stats()["status"] == 0
            tree.close()
    finally:
        rt.set_table_cap(-1)

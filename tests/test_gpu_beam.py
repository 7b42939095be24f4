"""Sources at one offset in consecutive leaves of a cube: the columns come from
per-direction step tables instead of a walk, and must be bit for bit those of
the walk, as must the statistics.

The walk is what the same call does for fewer than a sixteenth of the leaves,
so the reference traces the sources in slices."""
import numpy as np
import pytest

import synth
from tinytrees import uniform_octree

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_09882_gb300 as rt
    return rt


def _dev(a):
    import torch
    a = np.ascontiguousarray(a)
    return torch.from_numpy(a.view(np.int64) if a.dtype == np.uint64 else a).cuda()


def _stats(tree):
    st = tree.stats()
    assert st["status"] == 0, st
    return st["rays"], st["segments"], st["exit_fallbacks"]


def _sources(keys, lev, how, rng):
    c = synth.leaf_centres(synth.Cloud(keys, lev, np.zeros((keys.shape[0], 1)), (1 << 21,) * 3))
    n = c.shape[0]
    h = 2.0 ** -int(lev[0])
    if how == "offset":          # off the centre, off the depth-21 lattice
        return c + (np.array([7 / 32, -11 / 32, 3 / 64]) + np.array([3, 5, -7]) * 2.0 ** -35) * h
    if how == "range":           # part of the leaves: ragged, not aligned to a block of any kind
        return c[n // 5 + 3:n // 2 + 18]
    if how == "most":            # ragged at both ends, few leaves outside
        return c[n // 50 + 3:n - n // 40 - 11]
    if how == "some_moved":      # some sources elsewhere, the first among them: the walk traces those
        idx = np.concatenate([[0, 1, 33, n - 1], rng.integers(0, n, n // 40)])
        c[idx] += (rng.random((idx.size, 3)) - 0.5) * 0.9 * h
        return c
    if how == "many_moved":      # too many: the walk traces all
        idx = rng.integers(0, n, n // 4)
        c[idx] += (rng.random((idx.size, 3)) - 0.5) * 0.9 * h
        return c
    if how == "last_place":      # one unit in the last place below the centre in some leaves
        c[::11] = np.nextafter(c[::11], 0.0)
        return c
    return c


@pytest.mark.parametrize("level,S,nside,dens,how", [
    (5, 1, 1, "f32", "centres"), (5, 4, 2, "f32", "centres"), (5, 8, 1, "f64", "centres"), (5, 3, 1, "f32", "offset"),
    (5, 2, 2, "f64", "range"), (6, 4, 1, "f32", "range"), (5, 4, 1, "f32", "some_moved"), (5, 2, 1, "f32", "many_moved"),
    (6, 1, 2, "f32", "last_place"), (5, 5, 4, "f32", "centres")])
@pytest.mark.parametrize("mode", ["f32k", "fp64"])
def test_columns_equal_the_walk(rt, level, S, nside, dens, how, mode):
    import torch
    rng = np.random.default_rng(1200 + 10 * level + S)
    keys, lev = uniform_octree(level)
    src = _dev(_sources(keys, lev, how, rng))
    n = rng.lognormal(0.0, 2.0, size=(keys.shape[0], S)).astype(np.float32 if dens == "f32" else np.float64)
    tree, d = rt.Octree(_dev(keys), _dev(lev)), _dev(n)
    cut = keys.shape[0] // 16 - 32
    tree.reset_stats()
    want = torch.cat([rt.trace_columns(tree, s, nside, d, mode) for s in src.split(cut)])
    want_st = _stats(tree)
    for again in range(2):  # the second call finds the first one's tables
        tree.reset_stats()
        got = rt.trace_columns(tree, src, nside, d, mode)
        assert _stats(tree) == want_st
        assert torch.equal(got, want), float((got - want).abs().max())
    # another offset on the same handle, then the first again
    moved = src + 2.0 ** -20
    w2 = torch.cat([rt.trace_columns(tree, s, nside, d, mode) for s in moved.split(cut)])
    assert torch.equal(rt.trace_columns(tree, moved, nside, d, mode), w2)
    assert torch.equal(rt.trace_columns(tree, src, nside, d, mode), want)
    # epilogues: nd terms per source in another order, each within 2^-53 of the
    # sum of non-negative terms; A_V,eff takes a logarithm of it
    for kind in ("av_eff", "beta", "attenuation"):
        e = rt.trace_epilogue(tree, src, nside, d, kind, [1.0] * S, 0.05, mode=mode)
        r = torch.cat([rt.trace_epilogue(tree, s, nside, d, kind, [1.0] * S, 0.05, mode=mode) for s in src.split(cut)])
        torch.testing.assert_close(e, r, rtol=1e-13, atol=1e-13)
    tree.close()


@pytest.mark.parametrize("level,S,nside,dens,how", [
    (5, 1, 2, "f64", "centres"), (5, 2, 2, "f32", "offset"), (5, 3, 2, "f32", "some_moved"), (5, 8, 2, "f64", "last_place"),
    (6, 1, 1, "f32", "most"), (6, 2, 1, "f32", "most"), (6, 4, 1, "f64", "most"), (6, 6, 2, "f32", "most")])
@pytest.mark.parametrize("mode", ["f32k", "fp64"])
def test_larger_columns_equal_the_walk(rt, level, S, nside, dens, how, mode):
    """Calls large enough for the form (a quarter million rays, few leaves
    computed in vain), ragged ranges among them."""
    test_columns_equal_the_walk(rt, level, S, nside, dens, how, mode)


@pytest.mark.parametrize("level,S,n_src,mode", [(5, 1, 32768, "f32k"), (5, 4, 32768, "fp64"), (6, 4, 200000, "f32k"), (6, 3, 190011, "f32k")])
def test_scattered_sources(rt, level, S, n_src, mode):
    """Sources at no common offset are walked: the same columns and statistics as
    the call without the form (a lowered step cap, which no ray reaches, turns it
    off), and about its time, the least of thirty calls of each in turn.  The
    form's checks take 12 to 16 us, whatever the walk takes; a vote that lets the
    tables be walked and a walk that waits for it took 160 at 64^3."""
    import torch
    rng = np.random.default_rng(1300 + level)
    keys, lev = uniform_octree(level)
    tree = rt.Octree(_dev(keys), _dev(lev))
    c = rng.random((n_src, 3))
    cell = (c * (1 << level)).astype(np.int64)
    order = np.argsort(sum(((cell[:, b] >> i) & 1) << (3 * i + b) for b in range(3) for i in range(level)), kind="stable")
    sets = [_dev(c[order]), _dev(np.nextafter(c[order], 0.0))]  # another call's tables must not help
    d = torch.rand((keys.shape[0], S), device="cuda")
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    least, out, st = {}, {}, {}
    for i in range(30):
        for cap in (0, 3 * (1 << level) + 2):
            tree.set_step_cap(cap)
            tree.reset_stats()
            torch.cuda.synchronize()
            ev[0].record()
            out[cap] = rt.trace_columns(tree, sets[i % 2], 1, d, mode, out=out.get(cap))
            ev[1].record()
            torch.cuda.synchronize()
            least[cap] = min(least.get(cap, 1e9), ev[0].elapsed_time(ev[1]))
            st[cap] = _stats(tree)
    (a, b), (x, y) = out.values(), st.values()
    assert torch.equal(a, b) and x == y
    on, off = least.values()
    assert on < off + 0.1, (on, off)  # ms
    tree.close()


def test_captured_call_walks(rt):
    """Under stream capture the call takes the walk (its scratch could move
    before a replay) and replays to the same columns."""
    import torch
    keys, lev = uniform_octree(5)
    src = _dev(_sources(keys, lev, "centres", None))
    d = torch.rand((keys.shape[0], 4), device="cuda")
    tree = rt.Octree(_dev(keys), _dev(lev))
    want = rt.trace_columns(tree, src, 1, d)
    out = torch.zeros_like(want)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        rt.trace_columns(tree, src, 1, d, out=out)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    tree.close()


@pytest.mark.parametrize("S", [1, 2, 4])
def test_paired_walk(rt, S):
    """Two rays per lane: a walked call of more than 2^24 rays of leaf centres (a step
    cap no ray reaches turns the form off).  Bit for bit the form's columns, with
    the same statistics, also with some sources off the centres and a ragged end;
    under a cap that stops most rays, the finished ones keep their columns."""
    import torch
    level = 7
    rng = np.random.default_rng(1500 + S)
    keys, lev = uniform_octree(level)
    tree = rt.Octree(_dev(keys), _dev(lev))
    src = _dev(_sources(keys, lev, "some_moved", rng)[:-37])
    d = torch.rand((keys.shape[0], S), device="cuda")
    tree.reset_stats()
    want = rt.trace_columns(tree, src, 1, d)
    st = _stats(tree)
    tree.set_step_cap(3 * (1 << level) + 2)
    tree.reset_stats()
    assert torch.equal(rt.trace_columns(tree, src, 1, d), want) and _stats(tree) == st
    nseg, _ = rt.trace_paths(tree, src, 1)
    tree.set_step_cap(40)
    tree.reset_stats()
    got = rt.trace_columns(tree, src, 1, d)
    short = tree.stats()
    done = nseg <= 40
    assert bool(done.any()) and not bool(done.all())
    assert short["status"] == 6  # RT_ERR_STEP_LIMIT
    assert short["segments"] == int(nseg.clamp(max=40).sum(dtype=torch.int64))
    assert torch.equal(got[done], want[done]) and not bool(got[~done].any())
    tree.close()


@pytest.mark.parametrize("how", ["centres", "scattered"])
def test_memory_between_calls(rt, how):
    """A handle that has traced keeps its tables, not the row copies of the
    densities (two of 134 MB here): an allocation of all that is free and
    half of them besides fits, and the next call still gives the same columns."""
    import torch
    keys, lev = uniform_octree(7)
    tree = rt.Octree(_dev(keys), _dev(lev))
    src = _dev(_sources(keys, lev, "centres", None) if how == "centres" else np.random.default_rng(5).random((keys.shape[0], 3)))
    d = torch.rand((keys.shape[0], 8), device="cuda", dtype=torch.float64)
    out = rt.trace_columns(tree, src, 1, d, "fp64")
    want = out.clone()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = torch.empty(torch.cuda.mem_get_info()[0] + (128 << 20), dtype=torch.uint8, device="cuda")
    del held
    torch.cuda.empty_cache()
    assert torch.equal(rt.trace_columns(tree, src, 1, d, "fp64", out=out), want)
    tree.close()


def test_first_call_beside_a_capture(rt):
    """A handle's first call, and one that needs larger tables, on a stream of its
    own while another stream is captured in the default mode: the capture stands
    and both results are right."""
    import torch
    keys, lev = uniform_octree(5)
    src = _dev(_sources(keys, lev, "centres", None))
    d = torch.rand((keys.shape[0], 4), device="cuda")
    other = rt.Octree(_dev(keys), _dev(lev))  # loads the kernels and the directions
    want = [rt.trace_columns(other, src, ns, d) for ns in (1, 2)]
    tree = rt.Octree(_dev(keys), _dev(lev))
    out = [torch.zeros_like(w) for w in want]
    x = torch.zeros(1000, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        x += 1
        for ns in (1, 2):
            rt.trace_columns(tree, src, ns, d, out=out[ns - 1], stream=side)
        x += 1
    g.replay()
    torch.cuda.synchronize()
    assert bool((x == 2).all())
    assert all(torch.equal(a, b) for a, b in zip(out, want))
    tree.close()
    other.close()


@pytest.mark.parametrize("n_src,nside", [(1, 1), (1, 8), (7, 4), (31, 2), (33, 1), (100, 2)])
@pytest.mark.parametrize("mode", ["f32k", "fp64"])
def test_few_rays_equal_many(rt, n_src, nside, mode):
    """A call of few rays gives each warp fewer than 32 of them; the columns,
    the gradient's terms and the paths are those of the same sources among many."""
    import torch
    from tinytrees import random_octree
    rng = np.random.default_rng(77)
    keys, lev, _ = random_octree(rng, 1, 6, 0.35)
    tree = rt.Octree(_dev(keys), _dev(lev))
    dens = _dev(rng.random((keys.shape[0], 3)).astype(np.float32))
    many = _dev(rng.random((6000, 3)))
    few = many[:n_src]
    want = rt.trace_columns(tree, many, nside, dens, mode)[:n_src]
    assert torch.equal(rt.trace_columns(tree, few, nside, dens, mode), want)
    for a, b in zip(rt.trace_paths(tree, few, nside, mode), rt.trace_paths(tree, many, nside, mode)):
        assert torch.equal(a, b[:n_src])
    # the transpose of the columns: <g, A n> = <A^T g, n>, FP64 sums of
    # non-negative terms against FP32 columns within their 1e-5
    g = torch.rand(want.shape, device="cuda", dtype=want.dtype)
    grad = rt.trace_columns_adjoint(tree, few, nside, g, mode)
    lhs, rhs = (g.double() * want.double()).sum(), (grad * dens.double()).sum()
    torch.testing.assert_close(lhs, rhs, rtol=1e-12 if mode == "fp64" else 1e-5, atol=0)
    tree.close()


@pytest.mark.parametrize("n_src,nside", [(1, 2), (3, 8), (31, 2), (33, 1), (100, 2)])
@pytest.mark.parametrize("mode", ["f32k", "fp64"])
@pytest.mark.parametrize("grid", ["octree", "cube"])
def test_few_rays_epilogue(rt, n_src, nside, mode, grid):
    """The epilogues of a call of few rays: each ray's term is that of the same
    ray among many, and a source's sum of them within a rounding a direction."""
    import torch
    from tinytrees import random_octree
    rng = np.random.default_rng(78)
    keys, lev = uniform_octree(4) if grid == "cube" else random_octree(rng, 1, 6, 0.35)[:2]
    tree = rt.Octree(_dev(keys), _dev(lev))
    dens = _dev(rng.random((keys.shape[0], 3)).astype(np.float32))
    many = _dev(rng.random((6000, 3)))
    for kind in ("attenuation", "av_eff", "beta"):
        few, all_ = (rt.trace_epilogue(tree, s, nside, dens, kind, [1.0, 2.0, 0.5], 0.7, mode=mode) for s in (many[:n_src], many))
        if kind == "attenuation":
            assert torch.equal(few, all_[:n_src])
        else:  # A_V,eff takes the logarithm of a mean of at least exp(-3.02 * 0.7 * 3.5 sqrt(3))
            torch.testing.assert_close(few, all_[:n_src], rtol=12 * nside * nside * 2.0 ** -52, atol=12 * nside * nside * 2.0 ** -52)
    tree.close()

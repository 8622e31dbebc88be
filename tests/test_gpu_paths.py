"""Which path a call takes and what it leaves behind, against the CPU oracle: shared lanes of the bit-sliced mixing, launches
that follow one another on different kernels."""
import numpy as np
import pytest

from paper_2203_08680_gb300 import gom
from paper_2203_08680_gb300 import instances as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from test_gpu_bs_items import _windows  # noqa: E402
from test_gpu_parity import _assert_same_state, _assert_same_stats, _gpu_state  # noqa: E402


def _few_rows(oracle, g, p, rows, seed):
    """A population of `rows` distinct rows, its cut weights and the best one's index."""
    rng = np.random.default_rng(seed)
    base = rng.integers(0, 2, (rows, g.n), dtype=np.uint8)
    pop = base[rng.integers(0, rows, p)]
    f = np.array([oracle.cut_value(g, x) for x in pop], dtype=np.int64)
    return pop, f, int(f.argmax())


def _load(P, run, pop, f, best):
    P.set_population(torch.from_numpy(pop).cuda(), torch.from_numpy(pop[best]).cuda(), int(f[best]), 0)
    run.load(pop, f, pop[best], int(f[best]), 0)


def _steps(P, run, gens, generation=None):
    """`gens` generations of both, every one compared."""
    for gen in range(gens):
        stats = generation(1) if generation else P.generation(1)[0]
        _assert_same_stats(stats[0], run.generation())
        _assert_same_state(_gpu_state(P), run.get(), f"generation {gen}")
    assert np.array_equal(P.fitness().cpu().numpy(), run.get()["f"])


@pytest.mark.parametrize("s,degree", [(5, 12), (12, 8), (24, 6)])
@pytest.mark.parametrize("p", [4, 33, 150])
def test_lanes_of_a_pair_share_its_corrected_flips(oracle, s, degree, p):
    """Groups of a few elements with many edges, so that up to 32 lanes share a pair, and populations of two rows,
    where individuals often are the run start that their own search falls through to: the pair's first lane corrects
    the flip planes that all its lanes have stored."""
    g = I.random_regular(60, degree, seed=s + p, wmin=-20, wmax=100)
    ep, ev = _windows(g.n, s)
    P = gom.Population(g, p, 3, fos=gom.gom_fos_create(g.n, ep, ev), bitsliced=True)
    k, co = oracle.color(g, ep, ev)
    run = oracle.Run(g, ep, ev, co, k, p, 3)
    _load(P, run, *_few_rows(oracle, g, p, 2, 7 * s + p))
    _steps(P, run, 10)


@pytest.mark.parametrize("bound,side,p", [(0, 40, 96), (10, 30, 70), (64, 30, 300)])
def test_captured_launch_replayed_between_other_paths(oracle, bound, side, p):
    """A generation captured on the default path and replayed after, before and between generations of the per-lane
    path, whose persistent kernel has another grid: each path's barrier counter stays a multiple of its own grid."""
    g = I.torus2d(side, seed=bound + p)
    stream = torch.cuda.Stream()
    fos = gom.gom_build_fos(g, gom.GOM_FOS_BFLT, bound) if bound else None
    ep, ev = oracle.build_bflt(g, bound) if bound else oracle.build_fos(g)
    k, co = oracle.color(g, ep, ev)
    run = oracle.Run(g, ep, ev, co, k, p, 5)
    with torch.cuda.stream(stream):
        P = gom.Population(g, p, 5, fos=fos, stream=stream, persistent=True)
        if not bound:
            gom.gom_set_option(P.ctx, gom.GOM_OPT_BITSLICED, 1)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        P.generation(1, want_stats=False)
    gom.gom_set_option(P.ctx, gom.GOM_OPT_BITSLICED, 0)
    with torch.cuda.stream(stream):
        for step in "drdrrddr":
            if step == "r":
                graph.replay()
            else:
                P.generation(1, want_stats=False)
            run.generation()
            assert P.generation_counter() == run.get()["g"]  # (an error word here is a barrier that gave up)
            _assert_same_state(_gpu_state(P), run.get(), step)


@pytest.mark.parametrize("bound,side,p,wmax,late", [(0, 60, 96, 255, 1), (0, 60, 96, 3000, 1), (0, 60, 96, 65535, 1),
                                                    (64, 30, 512, 100, 1), (100, 24, 40, 100, 1), (100, 24, 40, 2000, 1),
                                                    (0, 8, 16, 3000, 0)])
def test_mixing_option_reads_and_restores_the_path(oracle, bound, side, p, wmax, late):
    """GOM_OPT_BITSLICED reads the path in force for every model that runs on bit-planes (`late`: the default), writing
    back what was read changes nothing, and each value can be set again; the same generations on either path."""
    g = I.torus2d(side, seed=side + wmax, wmin=-wmax // 2, wmax=wmax)
    fos = gom.gom_build_fos(g, gom.GOM_FOS_BFLT, bound) if bound else None
    ep, ev = oracle.build_bflt(g, bound) if bound else oracle.build_fos(g)
    k, co = oracle.color(g, ep, ev)
    run = oracle.Run(g, ep, ev, co, k, p, 4)
    P = gom.Population(g, p, 4, fos=fos)
    assert gom.gom_get_option(P.ctx, gom.GOM_OPT_BITSLICED) == late
    gom.gom_set_option(P.ctx, gom.GOM_OPT_BITSLICED, late)
    for value in (late, 0, 1, 0, 1):
        gom.gom_set_option(P.ctx, gom.GOM_OPT_BITSLICED, value)
        assert gom.gom_get_option(P.ctx, gom.GOM_OPT_BITSLICED) == value
        _steps(P, run, 1)


def test_mixing_option_refused_past_every_width():
    """Weights past 65,535: no bit-planes, 1 is refused and 0 stands."""
    P = gom.Population(I.torus2d(12, seed=1, wmin=1, wmax=70000), 40, 1)
    assert gom.gom_get_option(P.ctx, gom.GOM_OPT_BITSLICED) == 0
    with pytest.raises(gom.GomError) as ei:
        gom.gom_set_option(P.ctx, gom.GOM_OPT_BITSLICED, 1)
    assert ei.value.code == -7
    gom.gom_set_option(P.ctx, gom.GOM_OPT_BITSLICED, 0)


@pytest.mark.parametrize("bound,p", [(0, 32), (24, 32), (100, 32), (24, 512), (100, 300)])
@pytest.mark.parametrize("dynamic", [True, False])
def test_item_schedule_of_the_bit_sliced_paths(oracle, bound, p, dynamic):
    """GOM_OPT_DYNAMIC on one-warp tiles (a one-word population) and, by element class, on tiles of several warps:
    claims leave their marks in the groups' counters, which stand behind the group order in the workspace, the static
    stride leaves them zero; equal generations."""
    g = I.torus2d(24, seed=bound)
    fos = gom.gom_build_fos(g, gom.GOM_FOS_BFLT, bound) if bound else None
    ep, ev = oracle.build_bflt(g, bound) if bound else oracle.build_fos(g)
    k, co = oracle.color(g, ep, ev)
    run = oracle.Run(g, ep, ev, co, k, p, 6)
    P = gom.Population(g, p, 6, fos=fos, persistent=True, dynamic=dynamic, bitsliced=True)
    _steps(P, run, 3)
    raw = P.workspace.cpu().numpy()[(-P.workspace.data_ptr()) % 256:]
    words = raw[:len(raw) // 256 * 256].view(np.int32).reshape(-1, 64)
    rows, order = (k + 63) // 64, oracle.group_order(6, k, 2)
    at = [r for r in range(len(words) - rows) if np.array_equal(words[r:r + rows].ravel()[:k], order)]
    assert len(at) == 1
    claims = words[at[0] + rows:at[0] + 2 * rows].ravel()[:k]
    assert claims.all() if dynamic else not claims.any()


def test_batch_counters_after_an_import_of_an_earlier_generation(oracle):
    """A batch made generations 3 to 7, then one instance is set back to generation 0: it has no counters of a call
    until the next one."""
    g = I.torus2d(12, seed=3)
    P = gom.Population(g, 40, 2)
    pop, _, fe = P.population()
    xe, _ = P.elite()
    P.generation(3)
    ws = torch.empty(gom.gom_batch_workspace_bytes(1) + 256, dtype=torch.uint8, device="cuda")
    batch = gom.gom_batch_create([P.ctx], None, ws[(-ws.data_ptr()) % 256:])
    gom.gom_batch_generation(batch, 4)
    assert [s["generation"] for s in gom.gom_batch_stats(batch, 0, 8)] == [3, 4, 5, 6]
    P.set_population(pop, xe, fe, 0)
    assert gom.gom_batch_stats(batch, 0, 8) == []
    gom.gom_batch_generation(batch, 2)
    ep, ev = oracle.build_fos(g)
    k, co = oracle.color(g, ep, ev)
    want = oracle.Run(g, ep, ev, co, k, 40, 2).run(2)
    for a, o in zip(gom.gom_batch_stats(batch, 0, 8), want):
        _assert_same_stats(a, o)


@pytest.mark.parametrize("bound,kind,side,p,late", [
    (0, 0, 100, 64, 1), (0, 0, 100, 32, 0), (0, 0, 10, 16, 0), (0, 0, 50, 128, 1), (0, 1, 50, 64, 0), (0, 1, 33, 128, 0),
    (14, 0, 50, 64, 0), (10, 0, 50, 300, 1), (24, 0, 50, 64, 0), (24, 0, 50, 128, 0), (48, 0, 33, 128, 0),
    (48, 0, 33, 256, 1), (24, 0, 100, 128, 1), (64, 0, 150, 64, 1), (100, 0, 22, 64, 1), (128, 0, 30, 1024, 1)])
def test_default_mixing_path(bound, kind, side, p, late):
    """The default on either side of the lines where one path was measured as the faster."""
    g = I.torus2d(side, seed=1)
    fos = gom.gom_build_fos(g, gom.GOM_FOS_BFLT, bound) if bound else None
    P = gom.Population(g, p, 1, kind=gom.GOM_FOS_SINGLETON if kind else gom.GOM_FOS_NEIGHBOURHOOD, fos=fos)
    assert gom.gom_get_option(P.ctx, gom.GOM_OPT_BITSLICED) == late


@pytest.mark.parametrize("bound,side,p", [(0, 30, 32), (0, 40, 96), (10, 20, 200), (24, 30, 300), (64, 20, 200), (100, 16, 40)])
@pytest.mark.parametrize("persistent", [True, False])
def test_forced_improvement_on_the_default_path(oracle, bound, side, p, persistent):
    """Forced Improvement where the mixing option was never set: per lane, bit-sliced, and by element class, until
    individuals have entered it (in the oracle's runs too)."""
    from test_gpu_fi import KEYS, _same, _state
    g = I.torus2d(side, seed=bound + p)
    fos = gom.gom_build_fos(g, gom.GOM_FOS_BFLT, bound) if bound else None
    ep, ev = oracle.build_bflt(g, bound) if bound else oracle.build_fos(g)
    k, co = oracle.color(g, ep, ev)
    run = oracle.Run(g, ep, ev, co, k, p, 8)
    run.set_fi(True, 2)
    P = gom.Population(g, p, 8, fos=fos, persistent=persistent, forced_improvement=True, fi_nis=2)
    seen = 0
    for gen in range(18):
        want = run.generation()
        got = P.generation(1)[0][0]
        seen += want["fi_individuals"]
        for gk, ok in KEYS:
            assert got[gk] == want[ok], (gen, gk, got, want)
        _same(_state(P), run.get(), f"gen {gen}")
    assert seen > 0


def test_batch_of_per_lane_instances_takes_no_room_for_bit_planes(oracle):
    """60 small linkage trees, whose shares of the warps leave them per lane: the launch has more than the one block
    of eight warps per SM that the regions of the element classes would leave, and the trees' generations are their
    own; with few instances the same trees are on bit-planes."""
    ws = torch.empty(gom.gom_batch_workspace_bytes(60) + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:]
    graphs = [I.torus2d(14, seed=i) for i in range(60)]
    pops = [gom.Population(g, 32, i, fos=gom.gom_build_fos(g, gom.GOM_FOS_BFLT, 128)) for i, g in enumerate(graphs)]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for part, config in ((pops, (8, 2, 0, 300)), (pops[:2], (8, 2, 2, 300))):
        batch = gom.gom_batch_create([P.ctx for P in part], config, ws)
        grid = gom.gom_batch_layout(batch, 0)[2]
        assert grid > sms if len(part) == 60 else grid == 2
        gom.gom_batch_generation(batch, 3)
        del batch
    for i in (0, 1, 59):
        ep, ev = oracle.build_bflt(graphs[i], 128)
        k, co = oracle.color(graphs[i], ep, ev)
        run = oracle.Run(graphs[i], ep, ev, co, k, 32, i)
        run.run(6 if i < 2 else 3)
        _assert_same_state(_gpu_state(pops[i]), run.get(), f"instance {i}")


def _batch_of(P, config):
    ws = torch.empty(gom.gom_batch_workspace_bytes(1) + 256, dtype=torch.uint8, device="cuda")
    batch = gom.gom_batch_create([P.ctx], config, ws[(-ws.data_ptr()) % 256:])

    def generation(num):
        gom.gom_batch_generation(batch, num)
        return gom.gom_batch_stats(batch, 0, num)
    return generation


@pytest.mark.parametrize("degree,wmax", [(4, 1000), (6, 1000), (7, 500), (9, 700), (12, 300), (15, 280),
                                         (4, 65535), (6, 20000), (7, 20000), (9, 10000), (12, 6000), (15, 4000),
                                         (20, 2000)])
@pytest.mark.parametrize("path", ["persistent", "graph", "batch"])
def test_wide_weights_on_bit_planes(oracle, degree, wmax, path):
    """Weights of 9 to 12 bits with sums below 2^16 (but the last row), then of up to 16 bits with sums below 2^20, in
    every element class; on bit-planes by request, the batch on one warp, whose fitness planes fill up between
    flushes."""
    g = I.random_regular(240, degree, seed=degree + wmax, wmin=-wmax, wmax=wmax)
    g.weight[:] = np.where(np.abs(g.weight) > wmax * 9 // 10, np.sign(g.weight) * wmax, g.weight)
    P = gom.Population(g, 70, 5, persistent=path != "graph", bitsliced=True)
    assert gom.gom_get_option(P.ctx, gom.GOM_OPT_BITSLICED) == 1
    ep, ev = oracle.build_fos(g)
    k, co = oracle.color(g, ep, ev)
    run = oracle.Run(g, ep, ev, co, k, 70, 5)
    _steps(P, run, 5, _batch_of(P, (1, 2, 1, 300)) if path == "batch" else None)


@pytest.mark.parametrize("bound,p,wmax", [(17, 64, 3000), (24, 300, 300), (40, 65, 3000), (64, 512, 3000), (100, 70, 300),
                                          (128, 1024, 2000), (128, 32, 2000)])
@pytest.mark.parametrize("path", ["persistent", "batch"])
def test_wide_weights_by_element_class(oracle, bound, p, wmax, path):
    """Linkage trees with 9- to 12-bit weights of either sign, by element class: the persistent kernel and one block of
    a batch, whose warps pass the sixteen items between two flushes of 20-bit sums."""
    g = I.torus2d(20, seed=bound + p, wmin=-wmax, wmax=wmax)
    ep, ev = oracle.build_bflt(g, bound)
    P = gom.Population(g, p, 9, fos=gom.gom_build_fos(g, gom.GOM_FOS_BFLT, bound), bitsliced=True)
    assert gom.gom_get_option(P.ctx, gom.GOM_OPT_BITSLICED) == 1
    k, co = oracle.color(g, ep, ev)
    run = oracle.Run(g, ep, ev, co, k, p, 9)
    _load(P, run, *_few_rows(oracle, g, p, 5, bound))
    _steps(P, run, 4, _batch_of(P, (4, 2, 1, 300)) if path == "batch" else None)


@pytest.mark.parametrize("n,p,shift", [(28003, 101, 1), (28003, 101, 0), (30001, 100, 2), (12003, 1024, 3), (20004, 100, 0),
                                       (20004, 100, 3), (9001, 700, 1), (9001, 300, 0), (100, 64, 0), (101, 64, 1)])
def test_rows_out_on_either_side_of_the_size_rule(n, p, shift):
    """The export in whole lines (the larger sizes: ragged tiles, rows and buffers off the 4-byte words) and one byte a
    thread."""
    P = gom.Population(I.empty_graph(n), p, 3, kind=gom.GOM_FOS_SINGLETON)
    pop = torch.from_numpy(np.random.default_rng(n + p).integers(0, 2, (p, n), dtype=np.uint8)).cuda()
    P.set_population(pop, pop[0].clone(), 0, 0)
    out = torch.full((p * n + 8,), 9, dtype=torch.uint8, device="cuda")
    gom.gom_get_population(P.ctx, out[shift:shift + p * n])
    assert torch.equal(out[shift:shift + p * n].view(p, n), pop)
    assert (out[:shift] == 9).all() and (out[shift + p * n:] == 9).all()

"""The bit-sliced mixing against the CPU oracle at the sizes where its donor
tables can go wrong: largest elements at the edges of the element classes (8,
16 and 32 variables), population words filled by one individual or all, and
populations of few distinct rows (long runs of equal patterns, searches that
fall through to the parent's own column)."""
import numpy as np
import pytest

from paper_2203_08680_gb300 import gom
from paper_2203_08680_gb300 import instances as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from test_gpu_parity import _assert_same_state, _assert_same_stats, _gpu_state  # noqa: E402


def _windows(n, s):
    """Singletons and windows of 2 .. s consecutive variables (mixed sizes, overlapping)."""
    sets = [[v] for v in range(n)]
    sets += [list(range(v, min(n, v + 1 + (v // s) % s))) for v in range(0, n, s)]
    sets += [list(range(v, v + s)) for v in range(0, n - s + 1, 2 * s)]
    return np.cumsum([0] + [len(x) for x in sets]).astype(np.int64), np.concatenate(sets).astype(np.int32)


@pytest.mark.parametrize("s,p", [(1, 2), (1, 33), (5, 32), (8, 3), (8, 257), (9, 31), (9, 64), (16, 100), (16, 512),
                                 (17, 65), (32, 40), (32, 1024)])
@pytest.mark.parametrize("rows", [0, 3])
def test_bit_sliced_items(oracle, s, p, rows):
    """`rows` distinct rows in the population (0: random), six generations, every one compared."""
    g = I.torus2d(9, seed=s + p, wmin=-20, wmax=100)
    ep, ev = _windows(g.n, s)
    P = gom.Population(g, p, 7, fos=gom.gom_fos_create(g.n, ep, ev), bitsliced=True)
    k, co = oracle.color(g, ep, ev)
    run = oracle.Run(g, ep, ev, co, k, p, 7)
    if rows:
        rng = np.random.default_rng(s * 1000 + p)
        base = rng.integers(0, 2, (rows, g.n), dtype=np.uint8)
        pop = base[rng.integers(0, rows, p)]
        f = np.array([oracle.cut_value(g, x) for x in pop], dtype=np.int64)
        best = int(f.argmax())
        P.set_population(torch.from_numpy(pop).cuda(), torch.from_numpy(pop[best]).cuda(), int(f[best]), 0)
        run.load(pop, f, pop[best], int(f[best]), 0)
    for gen in range(6):
        stats, _ = P.generation(1)
        _assert_same_stats(stats[0], run.generation())
        _assert_same_state(_gpu_state(P), run.get(), f"generation {gen}")


@pytest.mark.parametrize("wmax,degree", [(255, 4), (256, 4), (4095, 4), (4096, 6), (65535, 4), (65535, 9)])
@pytest.mark.parametrize("path", ["persistent", "graph", "batch"])
def test_wide_weights(oracle, wmax, degree, path):
    """Weights up to every plane width's bound, of either sign (65,535 on 90-edge elements: sums past the widest
    planes, the per-lane path)."""
    g = I.random_regular(600, degree, seed=wmax % 97, wmin=-wmax, wmax=wmax)
    g.weight[:] = np.where(np.abs(g.weight) > wmax * 9 // 10, np.sign(g.weight) * wmax, g.weight)
    P = gom.Population(g, 70, 5, persistent=path != "graph")
    ep, ev = oracle.build_fos(g)
    k, co = oracle.color(g, ep, ev)
    run = oracle.Run(g, ep, ev, co, k, 70, 5)
    if path == "batch":
        ws = torch.empty(gom.gom_batch_workspace_bytes(1) + 256, dtype=torch.uint8, device="cuda")
        batch = gom.gom_batch_create([P.ctx], (4, 2, 8, 300), ws[(-ws.data_ptr()) % 256:])
    for gen in range(5):
        if path == "batch":
            gom.gom_batch_generation(batch, 1)
            stats = gom.gom_batch_stats(batch, 0, 1)
        else:
            stats, _ = P.generation(1)
        _assert_same_stats(stats[0], run.generation())
        _assert_same_state(_gpu_state(P), run.get(), f"generation {gen}")
    assert np.array_equal(P.fitness().cpu().numpy(), run.get()["f"])


@pytest.mark.parametrize("bound,p", [(10, 300), (16, 33), (17, 64), (40, 65), (64, 512), (100, 70), (128, 1024), (128, 32)])
@pytest.mark.parametrize("path", ["persistent", "batch", "wide"])
def test_linkage_trees_by_class(oracle, bound, p, path):
    """Elements of 1 to `bound` variables in one model: the small classes' items and the blocks' large elements
    (33 to 128 variables) on the default path, batched, and with 16-bit weights; a few distinct rows at first, so
    that long runs and self-hits occur."""
    wmax = 30000 if path == "wide" else 100
    g = I.torus2d(22, seed=bound + p, wmin=-wmax // 3, wmax=wmax)
    ep, ev = oracle.build_bflt(g, bound)
    P = gom.Population(g, p, 9, fos=gom.gom_build_fos(g, gom.GOM_FOS_BFLT, bound))
    k, co = oracle.color(g, ep, ev)
    run = oracle.Run(g, ep, ev, co, k, p, 9)
    rng = np.random.default_rng(bound * 7 + p)
    base = rng.integers(0, 2, (5, g.n), dtype=np.uint8)
    pop = base[rng.integers(0, 5, p)]
    f = np.array([oracle.cut_value(g, x) for x in pop], dtype=np.int64)
    best = int(f.argmax())
    P.set_population(torch.from_numpy(pop).cuda(), torch.from_numpy(pop[best]).cuda(), int(f[best]), 0)
    run.load(pop, f, pop[best], int(f[best]), 0)
    if path == "batch":
        ws = torch.empty(gom.gom_batch_workspace_bytes(1) + 256, dtype=torch.uint8, device="cuda")
        batch = gom.gom_batch_create([P.ctx], (4, 2, 2, 300), ws[(-ws.data_ptr()) % 256:])
    for gen in range(4):
        if path == "batch":
            gom.gom_batch_generation(batch, 1)
            stats = gom.gom_batch_stats(batch, 0, 1)
        else:
            stats, _ = P.generation(1)
        _assert_same_stats(stats[0], run.generation())
        _assert_same_state(_gpu_state(P), run.get(), f"generation {gen}")

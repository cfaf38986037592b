"""GPU: what the low-order equations take from a step, with few groups on many cells: right at the edges of the blocks, and no
slower than one thread per cell or face."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def plan(n, G, faces=False):
    import paper_2305_11998_gb300 as molc
    return molc.Plan.from_workload(synth.Workload("few", n, n, 1.0, G, 0.01, 10.0, 1, 4, 1, 1), faces=faces)


def time_us(f, n=20):
    """The least time of a launch in replays of a graph of n."""
    f()
    torch.cuda.synchronize()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        for _ in range(n):
            f()
    best = float("inf")
    for _ in range(6):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        g.replay()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / n)
    return best


def moments(n, G, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return {k: torch.rand(G, n * n, dtype=torch.float64, device="cuda", generator=gen) + 0.01
            for k in ("E", "Fx", "Fy", "Nxx", "Nxy", "Nyy")}


@pytest.mark.parametrize("n,G", [(1, 1), (16, 2), (37, 1), (37, 2), (37, 3)])
def test_closure(n, G):
    P, m, c = plan(n, G), moments(n, G, 3), 3.0
    f = P.closure(m, c, grey=True)
    for j, (k, x) in enumerate((("fxx", "Nxx"), ("fxy", "Nxy"), ("fyy", "Nyy"))):
        want = m[x] / (c * m["E"])
        assert bool(((f[k] - want).abs() <= 4 * U * want).all()), k
        mean = m[x].sum(0) / (c * m["E"].sum(0))
        assert bool(((f["grey"][j] - mean).abs() <= 2 * (G + 4) * U * mean).all()), k
    P.close()


# half-way between 21.5 us in blocks of cells x groups and 13.7 us with one thread per cell; 17.9 and 15.1 with 2 groups
@pytest.mark.parametrize("n,G,most", [(512, 1, 17.6), (400, 2, 16.5)])
def test_closure_time(n, G, most):
    P, m = plan(n, G), moments(n, G, 3)
    assert time_us(lambda: P.closure(m, 3.0, grey=True)) <= most
    P.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n,G", [(3, 1), (60, 1), (200, 1), (120, 2), (90, 5), (70, 33)])
def test_face_moments_of_each_group_alone(n, G, prec):
    """Face moments of all groups against those of each group's own plan: the same sums, FP64 reductions in another order."""
    gen = torch.Generator(device="cuda").manual_seed(5)
    kappa, B = (torch.rand(G, n * n, dtype=torch.float64, device="cuda", generator=gen) + 0.2 for _ in range(2))
    bnd = torch.rand(4, G, dtype=torch.float64, device="cuda", generator=gen) + 0.2

    def faces(groups):
        P = plan(n, len(groups), faces=True)
        I = P.new_intensity(prec)
        k, b, e = kappa[groups].contiguous(), B[groups].contiguous(), bnd[:, groups].contiguous()
        P.intensity_init(prec, I, b)
        P.sweep(prec, k, b, 1.0, 0.3, I, e)
        out = P.face_moments(prec, I, 1.0)
        torch.cuda.synchronize()
        P.close()
        return out

    whole = faces(list(range(G)))
    for g in sorted({0, G // 2, G - 1}):
        part = faces([g])
        # a face takes fewer than 100 terms, none larger than its E c; FP32 states of B in [0.2, 1.2] share one scale
        for k, x in part.items():
            assert float((whole[k][g] - x[0]).abs().max()) <= 200 * U * float(whole["E"].max()), k


# half-way between 156 and 23.6 us, 55.2 and 46.3 us: 16 faces a block whatever the groups, one thread per (face, group)
@pytest.mark.parametrize("n,G,most", [(512, 1, 89.8), (256, 8, 50.7)])
def test_face_moments_time(n, G, most):
    P = plan(n, G, faces=True)
    B = torch.ones(G, n * n, dtype=torch.float64, device="cuda")
    I = P.new_intensity("fp32")
    P.intensity_init("fp32", I, B)
    P.sweep("fp32", B, B, 1.0, 0.3, I, torch.ones(4, G, dtype=torch.float64, device="cuda"))
    assert time_us(lambda: P.face_moments("fp32", I, 1.0)) <= most
    P.close()

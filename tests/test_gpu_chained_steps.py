"""GPU: steps whose kernels follow one another by programmatic dependent launch.  Where the walks are few but the kernels
around the sweep are not, a step takes no longer than the same work launched plainly; and a chained step of either
precision can be captured in a CUDA graph and replayed."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def molc():
    import paper_2305_11998_gb300 as m
    m.load()
    return m


def problem(molc, prec, n, G, npol, naz, div):
    wl = synth.Workload("chain", n, n, 6.0, G, 0.001, 100.0, npol, naz, div, 1)
    d = wl.inputs(5)
    P = molc.Plan.from_workload(wl)
    dev = {k: torch.tensor(d[k], dtype=torch.float64, device="cuda") for k in ("kappa", "B", "bnd")}
    I = P.new_intensity(prec).zero_()
    P.intensity_init(prec, I, dev["B"])
    return P, dev, d, I


def time_us(step, n=30):
    """The least mean of five runs of n steps."""
    best = float("inf")
    for _ in range(6):   # the first warms up
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        for _ in range(n):
            step()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / n)
    return best


# few walks (at most 152 x 128), many cells: the batch of one instance launches the same kernels plainly
@pytest.mark.parametrize("n,npol,naz", [(400, 1, 12), (216, 6, 20), (200, 8, 32)])
def test_few_walks_on_many_cells_not_slower_than_plain_launches(molc, n, npol, naz):
    P, dev, d, I = problem(molc, "fp32", n, 1, npol, naz, 2)
    assert 2 * P.info.n_tracks <= 152 * 128
    out = P.new_moments()
    chained = time_us(lambda: P.sweep("fp32", dev["kappa"], dev["B"], d["c"], d["dt"], I, dev["bnd"], out=out))
    batch = molc.Batch([P])
    batch.bind([dict(dev, I=I, c=d["c"], dt=d["dt"], out=out)])
    plain = time_us(batch.sweep)
    batch.close()
    assert chained <= 1.15 * plain, (chained, plain)
    P.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("shape", [(16, 4, 2, 16, 2), (64, 2, 5, 8, 2), (24, 17, 4, 8, 2)], ids=lambda s: "n%d_g%d_p%d" % s[:3])
def test_captured_chained_steps_replay(molc, prec, shape):
    P, dev, d, I = problem(molc, prec, *shape)
    J = I.clone()
    out, ref = P.new_moments(), P.new_moments()
    step = lambda state, m: P.sweep(prec, dev["kappa"], dev["B"], d["c"], d["dt"], state, dev["bnd"], out=m)  # noqa: E731
    for _ in range(5):
        step(J, ref)
    step(I, out)   # loads the kernels before the capture
    torch.cuda.synchronize()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        step(I, out)
        step(I, out)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(I, J)   # the state depends on no order of additions
    for k in ref:
        if prec == "fp32":
            assert torch.equal(out[k], ref[k]), k
        else:   # FP64 atomics: the order of at most a few hundred terms, of the size of c E
            size = d["c"] * ref["E"].abs()
            assert torch.all((out[k] - ref[k]).abs() <= 1e-12 * torch.clamp(size if k != "E" else ref["E"].abs(), min=1e-30 * size.max())), k
    assert P.device_status() == 0
    P.close()

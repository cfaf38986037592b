"""GPU: an instance whose gather needs much shared memory for a single cell does not slow down the others of its batch, whose
blocks would otherwise be given as much; and the results stay those of single steps."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def instance(molc, n, G, npol, naz, div):
    wl = synth.Workload("cls", n, n, 6.0, G, 0.001, 100.0, npol, naz, div, 1)
    d = wl.inputs(4)
    P = molc.Plan.from_workload(wl)
    a = {k: torch.tensor(d[k], dtype=torch.float64, device="cuda") for k in ("kappa", "B", "bnd")}
    I = P.new_intensity("fp32").zero_()
    P.intensity_init("fp32", I, a["B"])
    return P, dict(a, I=I, c=d["c"], dt=d["dt"], out=P.new_moments())


def batch_us(molc, ones):
    batch = molc.Batch([P for P, _ in ones])
    batch.bind([a for _, a in ones])
    best = float("inf")
    for _ in range(6):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        e[0].record()
        for _ in range(5):
            batch.sweep()
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]) * 1e3 / 5)
    batch.close()
    return best


def test_one_large_unit_among_others():
    import paper_2305_11998_gb300 as molc
    ones = [instance(molc, 192, 17, 3, 40, 2) for _ in range(2)]
    alone = batch_us(molc, ones)
    # 100 azimuth pairs with one segment or two of each cell, 32 groups: units of about 128 segments, 50 KB and more
    small = instance(molc, 6, 32, 3, 200, 1)
    together = batch_us(molc, ones + [small])
    assert together <= 1.1 * alone, (together, alone)


def test_results():
    import paper_2305_11998_gb300 as molc
    shapes = [(24, 17, 3, 24, 2), (6, 32, 3, 200, 1), (8, 32, 3, 96, 1), (6, 32, 4, 200, 1)]
    ones = [instance(molc, *s) for s in shapes]
    single = [instance(molc, *s) for s in shapes]
    batch = molc.Batch([P for P, _ in ones])
    batch.bind([a for _, a in ones])
    for _ in range(2):
        batch.sweep()
        for P, a in single:
            P.sweep("fp32", a["kappa"], a["B"], a["c"], a["dt"], a["I"], a["bnd"], out=a["out"])
    torch.cuda.synchronize()
    for (P, a), (_, b) in zip(ones, single):
        assert torch.equal(a["I"], b["I"])
        for k in a["out"]:
            assert torch.equal(a["out"][k], b["out"][k]), k
    batch.close()

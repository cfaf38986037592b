"""GPU: the moment gather at the edges of its work split: one segment a cell, runs of exactly four and one over, units
of more than 128 segments (a split cell), a last chunk of few groups, one to eight polar cosines.  Against the binary128
oracle through the parity gate; and the same bits from a batch, which shares its blocks out otherwise."""
import pytest

import oracle
import parity
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# cells a side, groups, polar cosines, azimuths, rays a cell
SHAPES = [(2, 1, 1, 4, 1), (7, 33, 3, 12, 4), (6, 32, 8, 8, 5), (5, 17, 7, 12, 9), (4, 37, 2, 16, 33), (3, 32, 5, 12, 64),
          (40, 3, 6, 8, 2), (70, 2, 4, 8, 3)]


@pytest.mark.parametrize("n,G,npol,naz,div", SHAPES)
def test_moments_at_split_edges(n, G, npol, naz, div):
    import paper_2305_11998_gb300 as molc
    wl = synth.Workload("runs", n, n, 6.0, G, 0.001, 100.0, npol, naz, div, 1)
    d = wl.inputs(3)
    P = molc.Plan.from_workload(wl)
    dev = {k: torch.tensor(d[k], dtype=torch.float64, device="cuda") for k in ("kappa", "B", "bnd")}
    states = [P.new_intensity("fp32").zero_() for _ in range(2)]   # whole buffers are compared
    for I in states:
        P.intensity_init("fp32", I, dev["B"])
    got = P.sweep("fp32", dev["kappa"], dev["B"], d["c"], d["dt"], states[0], dev["bnd"])
    out = {k: torch.empty_like(x) for k, x in got.items()}
    batch = molc.Batch([P])
    batch.bind([dict(dev, I=states[1], c=d["c"], dt=d["dt"], out=out)])
    batch.sweep()
    torch.cuda.synchronize()
    assert torch.equal(states[0], states[1])
    for k in got:
        assert torch.equal(got[k], out[k]), k
    ref = parity.reference(oracle.Geometry.from_workload(wl), d, "fp32", npol)
    parity.compare({k: x.cpu().numpy() for k, x in got.items()}, ref, "fp32", d["c"])
    assert P.device_status() == 0
    batch.close()
    P.close()

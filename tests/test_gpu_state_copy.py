"""GPU: writing segment averages into a state and reading them back, over the state's layouts: every polar count of the
FP32 bundles, group ranges inside, across and beyond a chunk of 32 groups, more groups than a block has threads, and
FP64 rows.  The expected values are formed on the host to the last bit: the state keeps Ibar - B in its own precision."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [("fp32", n, 5, 0, 5) for n in range(1, 9)] + [("fp32", 3, 37, 0, 37), ("fp32", 4, 37, 30, 5),
                                                      ("fp32", 2, 37, 33, 1), ("fp32", 1, 150, 1, 147),
                                                      ("fp64", 3, 37, 0, 37), ("fp64", 9, 5, 2, 3),
                                                      ("fp64", 2, 150, 0, 150)]


@pytest.mark.parametrize("prec,NP,G,g0,count", CASES)
def test_import_then_export(prec, NP, G, g0, count):
    import paper_2305_11998_gb300 as molc
    wl = synth.Workload("copy", 7, 5, 1.0, G, 0.01, 10.0, NP, 12, 3, 1)
    P = molc.Plan.from_workload(wl)
    rng = np.random.default_rng(NP * 1000 + G)
    ns, cell = P.info.n_segments, P.tracks()["cell"]
    B = torch.tensor(rng.uniform(0.5, 2.0, (G, 35)))
    Bseg = B[:, cell].T.contiguous()
    delta = torch.tensor(rng.uniform(-1.0, 1.0, (ns, G)) * 10.0 ** rng.uniform(-6, 0, (ns, G)))
    delta[::7] = 0.0
    canon = Bseg + delta
    I = P.new_intensity(prec)
    P.intensity_init(prec, I, B.cuda())
    sub = canon[:, g0:g0 + count].contiguous()
    P.intensity_import(prec, I, sub.cuda(), B.cuda(), g_begin=g0)
    kept = canon - Bseg
    want = Bseg + (kept.float().double() if prec == "fp32" else kept)
    want[:, :g0] = Bseg[:, :g0]
    want[:, g0 + count:] = Bseg[:, g0 + count:]
    assert torch.equal(P.intensity_export(prec, I).cpu(), want)
    assert torch.equal(P.intensity_export(prec, I, g0, count).cpu(), want[:, g0:g0 + count])
    P.close()

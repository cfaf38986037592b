"""GPU: the moment gather keeps its rate (state bytes read over the kernel's time) away from the production shape: one, two,
five and seven polar cosines.  The floors lie half-way between the rates of a cut tuned for 4 polar cosines alone (1.76, 2.87,
3.06 and 2.48 TB/s) and those of the library's cut (2.00, 3.10, 3.73 and 4.12 TB/s)."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# cells a side, groups, polar cosines, azimuths, rays a cell, bytes per second
SHAPES = [(248, 17, 1, 48, 4, 1.88e12), (256, 17, 2, 56, 2, 2.98e12), (243, 8, 5, 60, 2, 3.39e12),
          (128, 17, 7, 48, 2, 3.30e12)]


@pytest.mark.parametrize("n,G,npol,naz,div,floor", SHAPES)
def test_gather_rate(n, G, npol, naz, div, floor):
    import paper_2305_11998_gb300 as molc
    wl = synth.Workload("rate", n, n, 6.0, G, 0.001, 100.0, npol, naz, div, 1)
    d = wl.inputs(3)
    P = molc.Plan.from_workload(wl)
    dev = {k: torch.tensor(d[k], dtype=torch.float64, device="cuda") for k in ("kappa", "B", "bnd")}
    I = P.new_intensity("fp32")
    P.intensity_init("fp32", I, dev["B"])
    out = P.new_moments()
    P.kernel_timing(True)
    best = float("inf")
    for _ in range(8):   # the first warms up
        P.sweep("fp32", dev["kappa"], dev["B"], d["c"], d["dt"], I, dev["bnd"], out=out)
        ms, steps = P.kernel_time_parts()
        best = min(best, ms["moments"] / steps)
    P.kernel_timing(False)
    assert 4 * P.info.n_updates / (best * 1e-3) >= floor
    P.close()

"""GPU: the FP64 sweep forming its cell entries from the inputs.  molc_sweep reads them from a table; molc_sweep_static_scratch
does so only while accumulators and table together fit its 64 MiB (80 bytes per cell and group), and between that and the
limit of the accumulators alone (48 bytes) the sweep forms them on the fly."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,G,npol", [(256, 17, 2), (224, 18, 1), (200, 30, 3)])
def test_entries_on_the_fly(n, G, npol):
    import paper_2305_11998_gb300 as molc
    assert 48 * n * n * G <= 64 << 20 < 80 * n * n * G
    wl = synth.Workload("fly", n, n, 6.0, G, 0.01, 10.0, npol, 8, 1, 1)
    d = wl.inputs(7)
    P = molc.Plan.from_workload(wl)
    dev = {k: torch.tensor(d[k], dtype=torch.float64, device="cuda") for k in ("kappa", "B", "bnd")}
    outs, states = [], []
    for sweep in (P.sweep, P.sweep_static_scratch):
        I = P.new_intensity("fp64").zero_()
        P.intensity_init("fp64", I, dev["B"])
        for _ in range(2):
            out = sweep("fp64", dev["kappa"], dev["B"], d["c"], d["dt"], I, dev["bnd"])
        outs.append(out)
        states.append(I)
    torch.cuda.synchronize()
    assert torch.equal(states[0], states[1])
    cE = d["c"] * outs[0]["E"].abs()
    for k in outs[0]:   # FP64 reductions in any order
        size = outs[0]["E"].abs() if k == "E" else cE
        assert bool(((outs[0][k] - outs[1][k]).abs() <= 1e-12 * torch.clamp(size, min=1e-30 * float(size.max()))).all()), k
    assert P.device_status() == 0
    P.close()

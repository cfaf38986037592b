"""GPU: an FP64 state that starts 8 bytes past a 16-byte boundary is swept like an aligned one."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# polar cosines in pairs and fours a thread, and 6, which an unaligned state takes in threes
@pytest.mark.parametrize("npol", [2, 4, 6, 8])
def test_state_at_an_odd_multiple_of_8_bytes(npol):
    import paper_2305_11998_gb300 as molc
    wl = synth.Workload("odd", 17, 17, 1.0, 24, 0.01, 10.0, npol, 24, 16, 1)
    d = wl.inputs(3)
    P = molc.Plan.from_workload(wl)
    dev = {k: torch.tensor(d[k], dtype=torch.float64, device="cuda") for k in ("kappa", "B", "bnd")}
    whole = [torch.zeros(P.intensity_bytes("fp64") + 16, dtype=torch.uint8, device="cuda") for _ in range(2)]
    assert whole[0].data_ptr() % 16 == 0
    states = [whole[0][:-16], whole[1][8:-8]]
    outs = []
    for I in states:
        P.intensity_init("fp64", I, dev["B"])
        for _ in range(2):
            out = P.sweep("fp64", dev["kappa"], dev["B"], d["c"], d["dt"], I, dev["bnd"])
        outs.append(out)
    torch.cuda.synchronize()
    n = 8 * P.intensity_count()
    assert torch.equal(states[0][:n], states[1][:n])   # the segment averages depend on no order of additions
    cE = d["c"] * outs[0]["E"].abs()
    for k in outs[0]:
        size = outs[0]["E"].abs() if k == "E" else cE
        assert bool(((outs[0][k] - outs[1][k]).abs() <= 1e-12 * torch.clamp(size, min=1e-30 * float(size.max()))).all()), k
    assert P.device_status() == 0
    P.close()

"""GPU: molc_grey_coefficients reads all groups of a cell before it writes that cell's six results, so that the output may lie
over an input's first six groups."""
import ctypes as C

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,G", [(9, 6), (16, 17), (45, 33), (69, 9), (70, 6), (75, 17)])   # up to 69^2 cells shared out by groups too
@pytest.mark.parametrize("over", ["kappa", "B", "E", "Fx", "Fy"])
def test_output_over_an_input(n, G, over):
    import paper_2305_11998_gb300 as molc
    P = molc.Plan.from_workload(synth.Workload("grey", n, n, 1.0, G, 0.01, 10.0, 1, 4, 1, 1))
    g = torch.Generator(device="cuda").manual_seed(n * G)
    a = {k: torch.rand(G, n * n, dtype=torch.float64, device="cuda", generator=g)
         for k in ("kappa", "B", "E", "Fx", "Fy", "Nxx", "Nxy", "Nyy")}
    a["Fx"] -= 0.5
    m = {k: a[k] for k in molc.molc.MOMENTS}
    want = torch.stack(list(P.grey_coefficients(m, a["kappa"], a["B"]).values()))
    ptr = lambda t: C.c_void_p(t.data_ptr())  # noqa: E731
    moments = molc.molc._Moments(*[ptr(m[k]).value for k in molc.molc.MOMENTS])
    rc = molc.load().molc_grey_coefficients(P._h, C.byref(moments), ptr(a["kappa"]), ptr(a["B"]), ptr(a[over]),
                                            C.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    assert rc == 0
    assert torch.equal(a[over].reshape(-1)[: 6 * n * n].reshape(6, -1), want)
    P.close()

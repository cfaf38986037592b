"""GPU: two host threads, each with its own plan and stream, whose moment gathers take different amounts of shared memory above
the default limit of 48 KB: the limit is the process's, and neither thread may lower it under the other's launch."""
import threading

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_two_threads_with_large_gathers():
    import paper_2305_11998_gb300 as molc
    n, G, sweeps, errors = 4, 32, 2000, []
    gate = threading.Barrier(2)

    def work(naz):
        try:
            q = synth.product_quadrature(1, naz)
            # rays 1.5 cells apart: at most one segment of a cell and azimuth pair, so that a cell's list is all runs
            P = molc.Plan(n, n, 1.0, 1.0, q.mu, q.cos_phi, q.sin_phi, q.w, G, 1.5 / n, renorm=False)
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                B = torch.ones(G, n * n, dtype=torch.float64, device="cuda")
                bnd = torch.ones(4, G, dtype=torch.float64, device="cuda")
                I = P.new_intensity("fp32")
                P.intensity_init("fp32", I, B)
                out = P.new_moments()
                P.sweep("fp32", B, B, 1.0, 0.5, I, bnd, out=out)
                first = out["E"].clone()
                stream.synchronize()
                gate.wait(timeout=60)
                for _ in range(sweeps):
                    P.sweep("fp32", B, B, 1.0, 0.5, I, bnd, out=out)
                stream.synchronize()
                assert torch.equal(out["E"], first)   # B = boundary = 1 everywhere: a step changes nothing
            P.close()
        except BaseException as e:  # noqa: BLE001
            errors.append(e)
            gate.abort()

    threads = [threading.Thread(target=work, args=(naz,)) for naz in (400, 240)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors

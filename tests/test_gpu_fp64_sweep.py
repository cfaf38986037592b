"""GPU: the FP64 sweep's ways of cutting its work (polar cosines per thread, partial chunks, few and many characteristics,
cell entries formed ahead or on the fly) against the binary128 oracle, with the tolerances of the parity gate."""
import numpy as np
import pytest

import oracle
import parity
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def molc():
    import paper_2305_11998_gb300 as m
    m.load()
    return m


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def inputs(n, G, seed):
    """Optical depths of a cell from 1e-10 to 1e4 side by side, B over six decades, boundaries of order one."""
    rng = np.random.default_rng(seed)
    return dict(kappa=np.exp(rng.uniform(np.log(1e-9), np.log(1e5), (G, n))),
                B=np.exp(rng.uniform(np.log(1e-6), 0.0, (G, n))), bnd=rng.uniform(0, 1, (4, G)), c=1.0, dt=0.7)


# (cells a side, polar cosines, groups, azimuths, spacing divisor): 1 to 8 polar cosines in one thread, with the many
# characteristics that takes; the same counts with few characteristics, one polar cosine a thread; and counts above 8
# cut into 3, 5 and 1 a thread
SHAPES = [(17, n, 24, 24, 16) for n in (2, 3, 4, 5, 6, 7, 8)] + [(9, n, 2, 8, 2) for n in (1, 2, 3, 5, 8)] + [
    (17, 9, 10, 24, 16), (17, 10, 17, 24, 16), (9, 11, 5, 8, 3)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "n%d_p%d_g%d_a%d_s%d" % s)
def test_polar_chunks_vs_binary128(molc, shape):
    n, NP, G, na, div = shape
    wl = synth.Workload("fp64", n, n, 1.0, G, 0.01, 10.0, NP, na, div, 1)
    d = inputs(n * n, G, 17 * NP + G)
    P = molc.Plan.from_workload(wl)
    k, B, bnd = dev(d["kappa"]), dev(d["B"]), dev(d["bnd"])
    I = P.new_intensity("fp64")
    P.intensity_init("fp64", I, B)
    geom = oracle.Geometry.from_workload(wl)
    groups = [0, G - 1]
    I_prev = I_err = None
    for step in range(2):
        out = (P.sweep if step else P.sweep_static_scratch)("fp64", k, B, d["c"], d["dt"], I, bnd)
        ref = parity.reference(geom, d, "fp64", NP, groups=groups, I_prev=I_prev, I_err=I_err, want_I=True)
        I_prev, I_err = ref["I"], ref["I_err"]
        got = {kk: v.cpu().numpy()[groups] for kk, v in out.items()}
        parity.compare(got, ref, "fp64", d["c"])
    assert P.device_status() == 0
    P.close()


@pytest.mark.parametrize("NP", [3, 4, 7])
def test_face_sums_vs_binary128(molc, NP):
    """The face sums of the FP64 sweep for more than two polar cosines against binary128."""
    wl = synth.Workload("faces", 9, 9, 1.0, 9, 0.01, 10.0, NP, 16, 8, 1)
    d = inputs(81, 9, NP)
    P = molc.Plan.from_workload(wl, faces=True)
    I = P.new_intensity("fp64")
    B = dev(d["B"])
    P.intensity_init("fp64", I, B)
    P.sweep("fp64", dev(d["kappa"]), B, d["c"], d["dt"], I, dev(d["bnd"]))
    got = {k: v.cpu().numpy() for k, v in P.face_moments("fp64", I, d["c"]).items()}
    r = oracle.sweep(oracle.Geometry.from_workload(wl), d["kappa"], d["B"], d["c"], d["dt"], d["bnd"],
                     precision="quad", want_faces=True, groups=[0, 8])
    for k in ("E", "Nxx", "Nyy"):
        ref = r["face_" + k]
        assert np.max(np.abs(got[k][[0, 8]] - ref) / np.maximum(np.abs(ref), 1e-30 * np.abs(ref).max())) <= 1e-12, k
    cE = d["c"] * np.abs(r["face_E"])
    for k in ("Fx", "Fy", "Nxy"):
        assert np.max(np.abs(got[k][[0, 8]] - r["face_" + k]) / cE) <= 1e-12, k
    P.close()


@pytest.mark.parametrize("kappa", [0.0, 1e-300, 1e-12, 1e300])
def test_extreme_opacities(molc, kappa):
    """Opacities whose optical depth leaves the fixed-point range (or nearly vanishes) against the FP64 closed form of a
    one-cell characteristic set: every characteristic enters at 1 and I^{n-1} = B = 0."""
    q = synth.product_quadrature(3, 8)
    P = molc.Plan(1, 1, 1.0, 1.0, q.mu, q.cos_phi, q.sin_phi, q.w, 1, 0.05)
    k, B, bnd = dev([[kappa]]), dev([[0.0]]), dev(np.ones((4, 1)))
    I = P.new_intensity("fp64")
    P.intensity_init("fp64", I, B)
    c, dt = 1.0, 1e290 if kappa < 1e-290 else 1e250
    out = {n: v.cpu().numpy().item() for n, v in P.sweep("fp64", k, B, c, dt, I, bnd).items()}
    tr = P.tracks()
    m = np.repeat(np.arange(q.n), np.diff(tr["dir_ray_off"]))        # one segment a characteristic
    tau = (kappa + 1 / (c * dt)) * tr["len"] / np.sqrt(1 - q.mu[m] ** 2)
    mean = np.where(tau < 1e-8, 1 - tau / 2, -np.expm1(-tau) / tau)   # (1 - e^-tau)/tau
    E = np.sum(q.w[m] * tr["area"] * mean) / c
    assert out["E"] == pytest.approx(E, rel=1e-13)
    assert P.device_status() == 0
    P.close()

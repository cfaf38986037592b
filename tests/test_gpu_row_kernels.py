"""GPU: the closure, the grey coefficients and the face moments at the edges of their blocks (cells, groups and faces that
do not fill the last one).  The first two on moments made up here, against torch in FP64 within the rounding of two sums of
G terms; the face moments of many groups against those of plans of few (the same sums, added in any order)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def plan(nx, ny, G, faces=False):
    import paper_2305_11998_gb300 as molc
    q = synth.product_quadrature(2, 8)
    return molc.Plan(nx, ny, 1.0, ny / nx, q.mu, q.cos_phi, q.sin_phi, q.w, G, 0.5 / nx, "uniform", True, faces=faces)


@pytest.mark.parametrize("nx,ny,G", [(1, 1, 1), (8, 4, 8), (11, 3, 7), (13, 5, 9), (9, 9, 40)])
def test_closure_and_grey_coefficients(nx, ny, G):
    P = plan(nx, ny, G)
    gen = torch.Generator(device="cuda").manual_seed(7)
    rand = lambda lo=0.0: torch.rand(G, nx * ny, generator=gen, device="cuda", dtype=torch.float64) * (1 - lo) + lo  # noqa: E731
    m = {k: rand(-1.0) if k in ("Fx", "Fy", "Nxy") else rand(0.01) for k in ("E", "Fx", "Fy", "Nxx", "Nxy", "Nyy")}
    kappa, B, c = rand(0.01) * 50, rand(0.01), 3.0
    for x in (*m.values(), B):
        x[:, 0] = 0.0            # a cell without radiation
    f = P.closure(m, c, grey=True)
    got = P.grey_coefficients(m, kappa, B)
    tol = 2 * (G + 4) * U
    quot = lambda a, b: torch.where(b > 0, a / b, 0.0)  # noqa: E731
    for k, n in (("fxx", "Nxx"), ("fxy", "Nxy"), ("fyy", "Nyy")):
        want = quot(m[n], c * m["E"])
        assert bool(((f[k] - want).abs() <= 4 * U * want.abs()).all()), k
    Es = m["E"].sum(0)
    for j, n in enumerate(("Nxx", "Nxy", "Nyy")):
        assert bool(((f["grey"][j] - quot(m[n].sum(0), c * Es)).abs() <= tol * quot(m[n].abs().sum(0), c * Es)).all()), n
    want = {"kappa_E": (m["E"], None), "kappa_B": (B, None), "KRx": (m["Fx"].abs(), "eta_x"), "KRy": (m["Fy"].abs(), "eta_y")}
    for k, (w, eta) in want.items():
        mean = quot((kappa * w).sum(0), w.sum(0))
        assert bool(((got[k] - mean).abs() <= 2 * tol * mean).all()), k
        if eta:
            F = m["Fx"] if eta == "eta_x" else m["Fy"]
            bound = quot(((kappa + mean) * F.abs()).sum(0), Es)
            assert bool(((got[eta] - quot(((kappa - mean) * F).sum(0), Es)).abs() <= 4 * tol * bound).all()), eta
    P.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_face_moments_of_many_groups(prec):
    nx, ny, G = 5, 3, 40
    rng = np.random.default_rng(5)
    t = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    kappa, B, bnd = rng.uniform(0.1, 9.0, (G, nx * ny)), rng.uniform(0.2, 1.0, (G, nx * ny)), rng.uniform(0.2, 1.0, (4, G))
    def faces(g):
        P = plan(nx, ny, kappa[g].shape[0], faces=True)
        I = P.new_intensity(prec)
        P.intensity_init(prec, I, t(B[g]))
        P.sweep(prec, t(kappa[g]), t(B[g]), 1.0, 0.3, I, t(bnd[:, g]))
        out = P.face_moments(prec, I, 1.0)
        torch.cuda.synchronize()
        P.close()
        return out
    whole = faces(slice(0, G))
    for g0 in range(0, G, 8):
        part = faces(slice(g0, g0 + 8))
        # a face takes fewer than 100 terms, none larger than its E c; FP32 states of B in [0.2, 1] share one scale
        for k, x in part.items():
            assert float((whole[k][g0:g0 + 8] - x).abs().max()) <= 200 * U * float(whole["E"].max()), k

"""The rounding of the HLLC flux of the non-compact schemes (csrc/k1d_nc.cu): gks_flux
against HLLC in extended precision from the interface states that
geno_reconstruct returns (the same states to the bit), on a smooth state.

Bar: as accurate as plain FP64 with a division per quotient, evaluated here on the
same states: root mean square error of each flux no larger, with 1% for the sample
of 2 10^5 faces and the order of the operations.  (Products with a reciprocal in
place of the divisions are 2% to 3% further off.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2507_20461_gb300 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _hllc(L, R, g):
    """subsonic HLLC (Toro, Davis bounds), in the precision of L and R"""
    one, half = L.dtype.type(1), L.dtype.type(0.5)
    (rl, ml, El), (rr, mr, Er) = L, R
    ul, ur = ml / rl, mr / rr
    pl, pr = (g - one) * (El - half * rl * ul * ul), (g - one) * (Er - half * rr * ur * ur)
    cl, cr = np.sqrt(g * pl / rl), np.sqrt(g * pr / rr)
    SL, SR = np.minimum(ul - cl, ur - cr), np.maximum(ul + cl, ur + cr)
    Ss = (pr - pl + rl * ul * (SL - ul) - rr * ur * (SR - ur)) / (rl * (SL - ul) - rr * (SR - ur))
    assert (SL < 0).all() and (SR > 0).all()

    def side(r, u, p, E, S, W):
        k = r * (S - u) / (S - Ss)
        U = [k, k * Ss, k * (E / r + (Ss - u) * (Ss + p / (r * (S - u))))]
        F = [r * u, r * u * u + p, u * (E + p)]
        return np.array([F[v] + S * (U[v] - W[v]) for v in range(3)])

    return np.where(Ss >= 0, side(rl, ul, pl, El, SL, L), side(rr, ur, pr, Er, SR, R))


@pytest.mark.skipif(np.finfo(np.longdouble).nmant <= 52, reason="no extended precision")
@pytest.mark.parametrize("order", [5, 6])
@pytest.mark.parametrize("speed", [0.4, -0.4])
def test_flux_is_as_accurate_as_with_divisions(order, speed):
    n = 200003
    rng = np.random.default_rng(order)
    x = (np.arange(n) + 0.5) / n
    rho = 1.0 + 0.2 * np.sin(2 * np.pi * x + rng.uniform(0, 6))
    u = speed + 0.1 * np.cos(2 * np.pi * x)
    p = 1.0 + 0.1 * np.sin(4 * np.pi * x)
    W = np.array([rho, rho * u, p / 0.4 + 0.5 * rho * u * u])
    s = B.Solver((n,), bc=B.BC_PERIODIC, precision=0, order=order, limiter=1)
    s.set_state(torch.from_numpy(W).to(DEV), torch.zeros((1,) + W.shape, dtype=torch.float64, device=DEV))
    st = torch.empty(2 * 3 * 2 * (n + 1), dtype=torch.float64, device=DEV)
    s.reconstruct(st)
    out = torch.empty(3 * 3 * (n + 1), dtype=torch.float64, device=DEV)
    s.flux(1e-6, out)
    s.close()
    L, R = st.cpu().numpy().reshape(2, 3, 2, n + 1)[:, :, 0]
    got = out.cpu().numpy().reshape(3, 3, n + 1)[0]
    wide = np.longdouble
    exact = _hllc(L.astype(wide), R.astype(wide), wide(1.4))
    plain = _hllc(L, R, np.float64(1.4))

    def rms(f):
        return np.sqrt(((f - exact) ** 2).mean(axis=1))

    assert (rms(got) <= 1.01 * rms(plain)).all(), (rms(got) / rms(plain)).astype(float)

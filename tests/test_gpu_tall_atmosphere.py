"""The correction tables of an atmosphere so tall that not all of its pieces
between breakpoints are tabulated: vertical columns against the closed form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_columns_through_pieces_of_either_kind():
    pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    h = np.array([0.0, 5e3, 9e6, 9.002e6, 1.2e7])   # 16 points per 2 km: the third piece and up are not tabulated
    delta = np.array([2.9e-4, 2e-4, 1e-5, 9e-6, 1e-7])
    atm = B.Atmosphere(kind=B.CS_ATM_TABLE, table=dict(h=h, delta=delta), refraction=True, transmission=True,
                       table_dh=2e4, table_nw=2)
    tab, info = atm.table()
    k = np.log(delta[1:] / delta[:-1]) / np.diff(h)
    for j in (0, 1, 100, 449, 450, 451, 500, 598):
        top = 2000.0 + j * info["dh"]
        want = 0.0
        for i in range(4):   # 100 rho dh, rho = 1.225e-3 delta / kappa [g/cm^3], exponential in each piece
            lo, hi = max(h[i], 2000.0), min(h[i + 1], top)
            if hi > lo:
                want += 100 * 1.225e-3 / 2.9e-4 * delta[i] * (np.exp(k[i] * (hi - h[i])) - np.exp(k[i] * (lo - h[i]))) / k[i]
        assert abs(float(tab[j, 0, 0, 2]) - want) <= 2e-6 * want, (j, float(tab[j, 0, 0, 2]), want)   # (stored in FP32)

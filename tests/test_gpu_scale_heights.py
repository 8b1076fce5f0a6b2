"""Scale heights without a usable reciprocal.  An infinite aerosol scale height
is an aerosol density that does not fall with height, an infinite layer scale
an empty layer; a denormal one an aerosol that ends at once.  The tables equal
those of a merely very large or very small one, whose quotients h / H round to
the same exponentials."""
import numpy as np
import pytest

from paper_2405_04229_gb300 import binding as B
from paper_2405_04229_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _table(aer_H=1200.0, layer_c=None, spherical=False):
    layered = dict(synth.US_STANDARD)
    if layer_c is not None:
        layered["c"] = [layer_c if i == 1 else c for i, c in enumerate(layered["c"])]
    atm = B.Atmosphere(layered=layered, refraction=True, transmission=True, transmission_params=dict(aer_H=aer_H),
                       spherical=spherical)
    tab = atm.table()[0]
    atm.close()
    return tab


@pytest.mark.parametrize("spherical", [False, True])
@pytest.mark.parametrize("kw,like", [(dict(aer_H=np.inf), dict(aer_H=1e60)), (dict(aer_H=1e-310), dict(aer_H=1e-60)),
                                     (dict(layer_c=np.inf), dict(layer_c=1e60))])
def test_tables_like_those_of_an_ordinary_number(kw, like, spherical):
    got, ref = _table(spherical=spherical, **kw), _table(spherical=spherical, **like)
    assert np.isfinite(ref).all()
    assert np.array_equal(got, ref)

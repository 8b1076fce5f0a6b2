"""Device memory of the telescope search's lists for an array of few spheres
far apart, which is mostly empty cells."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spherical", [False, True])
def test_sparse_array_takes_no_more_than_one_list_of_4e6_cells_a_level(spherical):
    torch = pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    rng = np.random.default_rng(3)
    tel = np.concatenate([rng.uniform(-10e3, 10e3, (2000, 2)), np.full((2000, 1), 2000.0), np.full((2000, 1), 6.0)], axis=1)
    B.Detector(tel=tel[:1], spherical=spherical).close()   # (the context is up)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    det = B.Detector(tel=tel, spherical=spherical)
    used = free - torch.cuda.mem_get_info()[0]
    det.close()
    # three levels of 4e6 cells of 8 bytes; 25 cells of 20 bytes a sphere and level; allocations of 2 MB
    assert used <= 3 * (4e6 * 8 + 2000 * 25 * 20) + (2 << 20)

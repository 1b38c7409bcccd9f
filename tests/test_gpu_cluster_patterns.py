"""GPU cluster histograms of ordered lattices against the oracle: columns, diagonals and
rows of single sites, columns joined at one end, a snake through the whole lattice -- the
longest chains and the most contacts a word can have.  Exact integers."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1309_4349_gb300 as klmc  # noqa: E402

klmc.build()


def patterns(Lx, Ly):
    y, x = np.divmod(np.arange(Lx * Ly), Lx)
    yield x % 2 == 0
    yield (x + y) % 2 == 0
    yield (x - y) % 2 == 0
    yield y % 2 == 0
    yield (x % 2 == 0) | (y == Ly // 2)
    yield x % 8 < 4
    yield (y % 4 == 0) | ((x == 0) & (y % 8 < 4)) | ((x == Lx - 2) & (y % 8 >= 4))


@pytest.mark.parametrize("packing", [klmc.PACK_BIT, klmc.PACK_BYTE])
@pytest.mark.parametrize("Lx,Ly,boundary", [
    (64, 64, 0), (33, 40, 0), (256, 128, 0), (4, 4, 0), (300, 300, 0), (257, 65, 0), (4, 1500, 0), (2000, 33, 0),
    (402, 63, 1), (66, 35, 1)])
def test_ordered_lattices(Lx, Ly, boundary, packing):
    for geometry in ([klmc.TRI6] if boundary else [klmc.TRI6, klmc.SQ4]):
        lat = klmc.Lattice(Lx, Ly, geometry=geometry, boundary=boundary, packing=packing, n_A=Lx, seed=1)
        for t in patterns(Lx, Ly):
            t = t.astype(np.uint8)
            lat.set_lattice(t)
            for species in (1, 0):
                s, c = lat.cluster_histogram(species)
                rs, rc = oracle.cluster_histogram(Lx, Ly, geometry, t, species, boundary=boundary)
                assert np.array_equal(s, rs) and np.array_equal(c, rc)
        lat.close()

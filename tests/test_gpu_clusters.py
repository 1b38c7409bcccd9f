"""GPU cluster histograms against the oracle at the sizes where the tiled labelling can go
wrong: one CTA's lattices (up to 8 words by 1024 words in all) and just beyond, tiles of 32
rows by 256 sites with remainders of one row, one word and one site, both boundaries.
Exact integers."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1309_4349_gb300 as klmc  # noqa: E402

klmc.build()

SIZES = [(4, 4, 0), (5, 33, 0), (33, 5, 0), (64, 64, 0), (256, 128, 0), (256, 129, 0), (257, 32, 0), (257, 33, 0),
         (289, 97, 0), (512, 64, 0), (513, 65, 0), (4, 2000, 0), (2000, 4, 0),
         (10, 7, 1), (24, 21, 1), (262, 7, 1), (402, 63, 1)]


def lattices(Lx, Ly, rng):
    """Random sites at several densities, and domains with a little noise."""
    for f in (0.05, 0.5, 0.65, 1.0):
        yield (rng.random(Lx * Ly) < f).astype(np.uint8)
    coarse = np.kron(rng.random((Ly // 9 + 1, Lx // 9 + 1)) < 0.45, np.ones((9, 9)))[:Ly, :Lx] > 0
    yield (coarse ^ (rng.random((Ly, Lx)) < 0.03)).astype(np.uint8).reshape(-1)


@pytest.mark.parametrize("packing", [klmc.PACK_BIT, klmc.PACK_BYTE])
@pytest.mark.parametrize("Lx,Ly,boundary", SIZES)
def test_tiled_cluster_histogram(Lx, Ly, boundary, packing):
    rng = np.random.default_rng(Lx * 7919 + Ly)
    for geometry in ([klmc.TRI6] if boundary else [klmc.TRI6, klmc.SQ4]):
        lat = klmc.Lattice(Lx, Ly, geometry=geometry, boundary=boundary, packing=packing, n_A=Lx * Ly // 2, seed=1)
        for t in lattices(Lx, Ly, rng):
            lat.set_lattice(t)
            for species in (1, 0):
                s, c = lat.cluster_histogram(species)
                rs, rc = oracle.cluster_histogram(Lx, Ly, geometry, t, species, boundary=boundary)
                assert np.array_equal(s, rs) and np.array_equal(c, rc)
        lat.close()

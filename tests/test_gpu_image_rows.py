"""Snapshots whose CTAs take 1, 2, 4 and 8 image rows, with rows left over, against the
oracle.  Exact integers."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1309_4349_gb300 as klmc  # noqa: E402

klmc.build()


@pytest.mark.parametrize("S", [2, 5])
@pytest.mark.parametrize("W,H", [(3000, 31), (3000, 111), (3000, 250), (3000, 405)])
def test_snapshot_rows(W, H, S):
    Lx, Ly = 257, 190
    t = (np.random.default_rng(W + H).random(Lx * Ly) < 0.5).astype(np.uint8)
    for packing in (klmc.PACK_BIT, klmc.PACK_BYTE):
        lat = klmc.Lattice(Lx, Ly, n_A=10, seed=9, packing=packing)
        lat.set_lattice(t)
        image, mask = lat.snapshot(W, H, S)
        want, want_mask = oracle.snapshot(Lx, Ly, t, W, H, S)
        assert np.array_equal(image.cpu().numpy(), want) and np.array_equal(mask.cpu().numpy(), want_mask)
        lat.close()

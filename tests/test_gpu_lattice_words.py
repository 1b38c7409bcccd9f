"""The word-at-a-time lattice operations against the oracle at the sizes where they can go
wrong: rows of one word and of several with a last word of 1, 31 and 32 sites, rows that
start at any byte and site offset, buffers off 16-byte boundaries, both boundaries and
stores; images at sample counts with and without a specialised kernel.  Exact integers."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1309_4349_gb300 as klmc  # noqa: E402

klmc.build()

SIZES = [(4, 4, 0), (31, 9, 0), (32, 8, 0), (33, 7, 0), (65, 40, 0), (63, 17, 0), (130, 33, 0), (256, 16, 0),
         (400, 330, 0), (10, 7, 1), (33 + 5, 14, 1), (66, 35, 1), (402, 63, 1)]


@pytest.mark.parametrize("packing", [klmc.PACK_BIT, klmc.PACK_BYTE])
@pytest.mark.parametrize("Lx,Ly,boundary", SIZES)
def test_word_operations(Lx, Ly, boundary, packing):
    N, seed = Lx * Ly, 1000 + Lx + Ly
    rng = np.random.default_rng(seed)
    for geometry in ([klmc.TRI6] if boundary else [klmc.TRI6, klmc.SQ4]):
        for nA in (1, N // 3, N - 1):
            lat = klmc.Lattice(Lx, Ly, geometry=geometry, boundary=boundary, packing=packing, n_A=nA, seed=seed)
            assert np.array_equal(lat.get_lattice(), oracle.init(Lx, Ly, nA, seed))
            offset = int(rng.integers(0, 17))
            t = (rng.random(N) < 0.4).astype(np.uint8)
            buf = torch.zeros(N + 32, dtype=torch.uint8, device="cuda")
            buf[offset:offset + N] = torch.from_numpy(t).cuda()
            lat.set_lattice_device(buf[offset:offset + N], 2)
            assert np.array_equal(lat.get_lattice(), t)
            assert lat.n_A == int(t.sum())
            want = oracle.n_unlike(Lx, Ly, geometry, t, boundary=boundary)
            assert lat.energy()[0] == want == lat.energy_recount()
            for sample in (0, (1 << 32) + 5):
                assert round(lat.ffn(sample)[0] * N) == oracle.ffn_count(Lx, Ly, geometry, t, seed, sample,
                                                                         boundary=boundary)
            lat.close()


@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 64])
def test_image_samples(S):
    Lx, Ly, seed = 131, 70, 9
    t = (np.random.default_rng(S).random(Lx * Ly) < 0.5).astype(np.uint8)
    lat = klmc.Lattice(Lx, Ly, n_A=10, seed=seed)
    lat.set_lattice(t)
    for W, H in ((1, 1), (7, 9), (257, 8), (300, 123)):
        image, mask = lat.snapshot(W, H, S)
        want, want_mask = oracle.snapshot(Lx, Ly, t, W, H, S)
        assert np.array_equal(image.cpu().numpy(), want) and np.array_equal(mask.cpu().numpy(), want_mask)
        assert tuple(lat.image_ffn(image, mask, 35, S)) == tuple(oracle.image_ffn(want, want_mask, 35, seed, S))
    lat.close()

"""The sweep kernels' branches against the oracle at the sizes where they can go wrong:
rows whose last word holds one site (windows that reach past it), rows of 97 words and
more (inner words apart from row ends), tiled blocks of 8 phases, splits that leave words
of a phase to a second pass, and draw thresholds at both ends of their range (0, just
above, 2^32).  Exact integers."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1309_4349_gb300 as klmc  # noqa: E402

klmc.build()


def check(Lx, Ly, geometry, bw, cluster, threads=0, steps=(5, 4), plan=None, boundary=0, packing=klmc.PACK_BIT):
    seed, nA = 3 + Lx + Ly, Lx * Ly * 2 // 5
    lat = klmc.Lattice(Lx, Ly, geometry=geometry, packing=packing, n_A=nA, omega_over_kT=bw, seed=seed,
                       cluster=cluster, threads=threads, boundary=boundary)
    if plan is not None:
        assert lat.plan() == plan
    for n in steps:
        lat.sweep(n)
    t0 = oracle.init(Lx, Ly, nA, seed)
    ref = oracle.run_mpkk(Lx, Ly, bw, seed, t0, 0, sum(steps)) if boundary else \
        oracle.run(Lx, Ly, geometry, bw, seed, t0, 0, sum(steps))
    assert np.array_equal(lat.get_lattice(), ref.lattice)
    c = lat.counters()
    assert (c["attempts"], c["unlike"], c["draws"], c["accepts"]) == ref.counters()
    assert lat.energy()[0] == ref.n_unlike == lat.energy_recount()
    lat.close()


BOTH = [klmc.TRI6, klmc.SQ4]


@pytest.mark.parametrize("geometry", BOTH)
@pytest.mark.parametrize("Lx,Ly,cluster,threads", [
    (33, 64, 1, 128), (33, 64, 2, 256), (65, 48, 4, 512), (97, 80, 8, 128), (129, 130, 16, 256), (257, 100, 4, 256),
    (63, 64, 2, 256), (95, 70, 4, 512), (1025, 90, 4, 512), (34, 72, 3, 256), (65, 40, -1, 0), (993, 30, -1, 0)])
def test_last_word_of_a_row(geometry, Lx, Ly, cluster, threads):
    for bw in (0.7, -0.7):
        check(Lx, Ly, geometry, bw, cluster, threads)


@pytest.mark.parametrize("Lx,Ly", [(129, 70), (66, 84), (101, 105), (325, 112), (66, 28), (129, 21)])
def test_last_word_helical(Lx, Ly):
    assert oracle.helical_valid(Lx, Ly)
    for bw in (0.7, -0.7):
        check(Lx, Ly, klmc.TRI6, bw, 0, boundary=klmc.HELICAL)


@pytest.mark.parametrize("geometry", BOTH)
@pytest.mark.parametrize("Lx", [3040, 3072, 3073, 3103, 3104, 3105, 6177])
def test_wide_rows(geometry, Lx):
    """Rows of 95 (no inner words apart), 96, 97, 98 and 194 words."""
    check(Lx, 40, geometry, 0.7, -1, steps=(3, 2))
    check(Lx, 41, geometry, -0.4, -1, steps=(2,), packing=klmc.PACK_BYTE)


@pytest.mark.parametrize("geometry", BOTH)
@pytest.mark.parametrize("Lx,Ly,K", [(1024, 768, 8), (1024, 767, 4), (1017, 1023, 8), (1025, 1537, 8), (500, 2100, 8)])
def test_tiled_blocks_of_eight(geometry, Lx, Ly, K):
    """Blocks of 8 phases from 786432 sites on, below it 4; odd and even numbers of
    blocks (which of the two buffers holds the result)."""
    check(Lx, Ly, geometry, 0.8, -1, steps=(1, 2, 3), plan=K)


@pytest.mark.parametrize("geometry", BOTH)
@pytest.mark.parametrize("bw", [200.0, -200.0, 30.0, 22.0, -22.5, 1e-12, -1e-12, 3e-10])
def test_thresholds_at_both_ends(geometry, bw):
    check(70, 64, geometry, bw, 2, 256)
    check(65, 64, geometry, bw, -1)
    if geometry == klmc.TRI6:
        check(66, 56, geometry, bw, 0, boundary=klmc.HELICAL)


@pytest.mark.parametrize("geometry", BOTH)
@pytest.mark.parametrize("Lx,Ly,cluster,threads", [
    (400, 130, 8, 128), (400, 130, 5, 256), (640, 66, 4, 256), (960, 130, 8, 512), (350, 48, 1, 512), (700, 48, 2, 256)])
def test_second_pass_of_a_phase(geometry, Lx, Ly, cluster, threads):
    """Phases with fewer, as many and more words than a CTA has threads with tasks, and
    with words left over after whole passes (split between threads where they fit)."""
    check(Lx, Ly, geometry, 0.6, cluster, threads)

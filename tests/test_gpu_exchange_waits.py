"""The bounded wait of the resident sweeps' halo exchange: made to run out through the
test hook (the CTAs withhold their stores), the launch ends, klmc_energy and
klmc_get_counters report KLMC_ETIMEOUT, and the device context stays usable (a new
handle's sweeps match the oracle bit for bit)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1309_4349_gb300 as klmc  # noqa: E402

klmc.build()
KLMC_ETIMEOUT = 4


@pytest.mark.parametrize("Lx,Ly,cluster,threads,boundary", [
    (200, 160, 4, 512, 0), (100, 64, 2, 256, 0), (257, 300, 16, 128, 0), (402, 399, 0, 0, 1)])
def test_exchange_wait_gives_up_and_reports(Lx, Ly, cluster, threads, boundary):
    nA, bw, seed = Lx * Ly // 3, 0.9, 5
    kw = dict(n_A=nA, omega_over_kT=bw, seed=seed, cluster=cluster, threads=threads, boundary=boundary)
    lat = klmc.Lattice(Lx, Ly, **kw)
    try:
        assert lat.launch_shape()[0] > 1 and lat.plan() > 1  # blocks of phases between exchanges
        lat.test_copy_shortfall(16)
        lat.sweep(3)
        for call in (lat.energy, lat.counters):
            with pytest.raises(klmc.KlmcError) as err:
                call()
            assert err.value.status == KLMC_ETIMEOUT
    finally:
        lat.close()
    fresh = klmc.Lattice(Lx, Ly, **kw)
    try:
        fresh.sweep(3)
        t0 = oracle.init(Lx, Ly, nA, seed)
        ref = oracle.run_mpkk(Lx, Ly, bw, seed, t0, 0, 3) if boundary else \
            oracle.run(Lx, Ly, oracle.TRI6, bw, seed, t0, 0, 3)
        assert np.array_equal(fresh.get_lattice(), ref.lattice)
        assert fresh.energy()[0] == ref.n_unlike
    finally:
        fresh.close()

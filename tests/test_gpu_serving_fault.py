"""A served job whose launch gave up a bounded wait: its fault slot, set here from the
host while the job is resident (its memory comes from the test's allocator), makes the
job finish with KLMC_ETIMEOUT and without results; the job beside it is untouched."""
import time

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1309_4349_gb300 as klmc  # noqa: E402

klmc.build()
KLMC_ETIMEOUT, KLMC_ESTATE = 4, 7
STATE_SLOTS, FAULT_SLOT = 13, 12


class TensorAllocator:
    """Device memory from tensors that the test can write."""

    def __init__(self):
        self.held = {}

        def _alloc(nbytes, stream, user):
            t = torch.zeros(int(nbytes), dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            self.held[t.data_ptr()] = t
            return t.data_ptr()

        def _free(ptr, nbytes, stream, user):
            self.held.pop(ptr)

        self.alloc = klmc.ALLOC_FN(_alloc)
        self.free = klmc.FREE_FN(_free)

    def state(self):
        (t,) = [t for t in self.held.values() if t.numel() == 8 * STATE_SLOTS]
        return t.view(torch.int64)


def test_job_that_gave_up_is_no_success():
    srv, mem = klmc.Server(1 << 30), TensorAllocator()
    # about a second of sweeps, several hundred rounds
    bad = srv.submit(400, 400, n_mcs=100000, hist_every=50000, keep_lattice=True, n_A=48000, omega_over_kT=0.6, seed=3,
                     allocator=mem)
    deadline = time.time() + 30
    while srv.stats()["rounds"] < 2:  # placed, and its state no longer cleared
        assert time.time() < deadline
        time.sleep(0.001)
    good = srv.submit(48, 40, n_mcs=20, keep_lattice=True, n_A=500, omega_over_kT=0.6, seed=31)
    mem.state()[FAULT_SLOT] = 1
    torch.cuda.synchronize()
    assert srv.poll(bad) is None  # still running
    srv.drain(120.0)
    assert srv.poll(bad)["status"] == KLMC_ETIMEOUT
    assert srv.histogram(bad)[0].size == 0
    with pytest.raises(klmc.KlmcError) as e:
        srv.lattice(bad, 400 * 400)
    assert e.value.status == KLMC_ESTATE
    assert not mem.held
    r = srv.poll(good)
    assert r["status"] == 0 and srv.stats()["attempts"] == r["attempts"]
    ref = oracle.run(48, 40, klmc.TRI6, 0.6, 31, oracle.init(48, 40, 500, 31), 0, 20)
    assert np.array_equal(srv.lattice(good, 48 * 40), ref.lattice)
    srv.close()

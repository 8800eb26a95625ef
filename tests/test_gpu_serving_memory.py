"""Device memory of a job whose batches are scheduled faster than they are applied (needs
a GPU: -m gpu)."""
import numpy as np
import pytest

from paper_2307_04890_gb300 import synth
from test_zz_no_alloc import _cudart, _pool_reset_and_read

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2307_04890_gb300 as tn
    from paper_2307_04890_gb300.build import build_library

    build_library()


def test_plans_in_flight_stay_near_the_charge():
    """Nine batches at once: eight plans wait for their update.  The charge is 160 bytes
    per event of one batch; by the buffers' sizes a job holds at most 53 for the batch
    being scheduled, 8 x 12 for the plans in flight, 16 for the copy in and 32 for
    held-back events and their concatenation (buffers grow by doubling): 197."""
    n, batch, parts = 2000, 200_000, 9
    u, v, t = synth.uniform_events(n, batch * parts, t_range=8 * batch * parts, seed=4)
    rt = _cudart()
    with tn.Server(max_active=1, workers=2) as server:
        # a first job, so that the slot and its buffers are there
        server.submit(0, n, u[:1000], v[:1000], t[:1000], np.array([0, 1000], np.uint64))
        while not server.poll(wait_ms=1000):
            pass
        torch.cuda.synchronize()
        used, _ = _pool_reset_and_read(rt, reset=True)
        server.submit(1, n, u, v, t, np.arange(parts + 1, dtype=np.uint64) * batch)
        records = []
        while not records:
            records = server.poll(wait_ms=1000)
        assert records[0]["status"] == tn.TN_OK
        _, high = _pool_reset_and_read(rt, reset=False)
        sizes, _ = server.results[1]
    charge = tn.tn_server_job_bytes(n, batch)
    assert high - used <= 1.5 * charge, ((high - used) / batch, charge / batch)
    want, _ = tn.tn_out_component_sizes_host(u, v, t, n)
    assert np.array_equal(sizes, want)

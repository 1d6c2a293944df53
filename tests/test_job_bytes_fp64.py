"""Device memory of FP64 contexts with a given tau batch (counted on the host by gw_job_bytes): the digits of the
tensor-core products share the batch's memory, they do not come on top of it."""
import pytest

from paper_2406_18479_gb300 import gw


@pytest.mark.parametrize("nk3,nao,naux", [((2, 2, 2), 52, 208), ((1, 1, 1), 120, 480), ((3, 3, 3), 40, 160), ((2, 1, 1), 60, 90)])
def test_tau_batch_bounds_the_memory(nk3, nao, naux):
    """From 4 to 12 nodes a context grows by at most 8 nodes of intermediates (2 nk naux nao^2 complex each), one
    more for the division into whole nodes, and the 64 MiB every FP64 context may use for digits."""
    nk = nk3[0] * nk3[1] * nk3[2]
    per_node = 2 * nk * naux * nao * nao * 16
    size = lambda c: gw.gw_job_bytes(gw.make_config(nk3, nao, naux, 24, 50.0, tau_chunk=c))      # noqa: E731
    assert size(12) - size(4) <= 9 * per_node + (64 << 20)
    # a batch of every node needs no more than the same memory as an automatic batch of that size
    assert size(24) <= size(4) + 21 * per_node + (64 << 20)

"""Which pivoted QRs of a batch wait for the end of the work list: a few long
ones do (a cluster of 8 SMs each), as many as there are SMs do not (together
they would take several rounds of clusters where one CTA each takes one)."""
import pytest
import torch

from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,n,k,l,launches", [(4, 512, 60, 70, 3), (150, 100, 30, 40, 1)])
def test_launches_of_a_run(count, n, k, l, launches):
    from paper_1905_13257_gb300 import IdBatch, load
    A = gaussian_matrix(1024, n, seed=n, dtype=torch.float32, device="cuda")
    bt = IdBatch([dict(A=A, k=k, l=l, seed=i) for i in range(count)])
    bt.run()
    bt.wait()
    before = load().id_kernel_launches()
    bt.run()
    assert load().id_kernel_launches() - before == launches
    assert all(kout == k for _, _, kout in bt.wait())
    bt.close()

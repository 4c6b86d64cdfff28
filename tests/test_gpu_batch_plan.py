"""Every lattice of a batch is swept whatever the mix of sizes: lattices worth
less than one CTA each next to large ones."""
import numpy as np
import pytest

from paper_1010_4834_gb300 import Batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("block_size", [256, 512])
def test_small_lattices_beside_large_ones_are_swept(prec, block_size):
    dims = [(4, 4, 4, 4)] * 40 + [(16, 16, 16, 8)] * 5 + [(4, 4, 4, 4)] * 40
    betas = [2.0 + 0.005 * i for i in range(len(dims))]
    a = Batch(dims, betas, seed=5, start="hot", prec=prec)
    a.block_size = block_size
    assert a.groups == len(dims)
    b = Batch(dims, betas, seed=5, start="hot", prec=prec)
    b.groups = 1                      # one group: one lattice after another on every CTA
    start = [a.get_links(i) for i in range(len(dims))]
    hist = a.sweep_measure(2)
    a.sweep(1)
    b.sweep(3)
    for i in range(len(dims)):
        got = a.get_links(i)
        assert np.array_equal(got, b.get_links(i)), i
        assert (got != start[i]).any(axis=(1, 2)).all(), i
    assert (hist[:, :, 0] != 0).all()

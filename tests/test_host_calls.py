"""What the library's host code does around its kernels, on a CUDA runtime of
host memory (host_runtime.cpp): which buffers outlive which work, what a failed
allocation leaves behind, what a call reports."""
import numpy as np
import pytest

import host_runtime


@pytest.fixture()
def rc(tmp_path):
    return host_runtime.load(tmp_path)


def tile(H, W, value=9):
    """(mask, marker, descriptor); the stand-in reconstruction sets the marker to the mask."""
    I, J = np.full((H, W), value, np.uint8), np.zeros((H, W), np.uint8)
    return I, J, (I.ctypes.data, J.ctypes.data, H, W, W, 8)


def done(tiles):
    return all((J == I).all() for I, J, _ in tiles)


def test_graph_is_not_replayed_from_a_staging_buffer_that_is_gone(rc):
    """An explicit schedule is replayed as a graph that copies from the staging
    buffer; a larger batch on the other engine in between replaces that buffer."""
    c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    one, many = tile(10, 12), [tile(5, 5) for _ in range(40)]
    for _ in range(3):
        one[1][:] = 0
        assert rc.recon_batch_ex(c, [one[2]], [1], [0]) == rc.RECON_OK and done([one])
        assert rc.recon_batch(c, [t[2] for t in many]) == rc.RECON_OK and done(many)
    assert rc.lib().ht_faults() == 0
    assert host_runtime.counts(rc)["graph"] == 3
    rc.recon_free(c)

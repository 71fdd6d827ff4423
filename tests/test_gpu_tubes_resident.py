"""GPU test of the tube batch's resident form (a tube per block in shared
memory) against the streamed form, bit for bit: lengths around the pair chunks
of its block sizes (128, 256, 512 threads, two nodes each), the shortest and the
longest tube that it takes, few and many tubes, steps split over calls, and a
tube that goes unphysical on the way."""
import numpy as np
import pytest

from test_gpu_tubes import _batch, _fields

pytestmark = pytest.mark.gpu

LENGTHS = [2, 3, 4, 127, 128, 129, 255, 256, 257, 258, 385, 511, 512, 513, 767, 1023, 1024, 1025,
           1537, 2047, 2048, 2049, 3600]


def _run(B, chunks, streamed):
    from paper_0908_3749_gb300 import lbm
    b = lbm.lbm_batch_create(B["nx"], B["dx"], B["dt"], B["s"], B["left"], B["right"])
    try:
        if streamed:
            lbm.lbm_batch_set_tiling(b, 512, 128)
        lbm.lbm_batch_set_init(b, *_fields(B))
        for n in chunks:
            lbm.lbm_batch_step(b, n)
        out = [np.empty(lbm.lbm_batch_total_nodes(b)) for _ in range(4)]
        lbm.lbm_batch_moments(b, *out)
        return out, lbm.lbm_batch_status(b, len(B["nx"])), lbm.lbm_batch_step_count(b)
    finally:
        lbm.lbm_batch_destroy(b)


def _same(a, b):
    for x, y in zip(a[0], b[0]):
        np.testing.assert_array_equal(x, y)
    assert a[1][0] == b[1][0] == 0 and a[1][2:] == b[1][2:] and a[2] == b[2]
    np.testing.assert_array_equal(a[1][1], b[1][1])


@pytest.mark.parametrize("copies,chunks", [(1, [20]), (10, [2, 17, 1]), (1, [1, 1, 18])])
def test_resident_equals_streamed(copies, chunks):
    B = _batch(LENGTHS * copies, seed=11)
    _same(_run(B, chunks, False), _run(B, [sum(chunks)], True))


def test_one_tube_too_long_for_shared_memory():
    B = _batch([200, 3700, 40], seed=12)
    _same(_run(B, [15], False), _run(B, [15], True))


def test_first_bad_level_of_an_unphysical_tube():
    import workloads as W
    B = _batch([200, 150, 600], seed=13)
    B["s"][0, :] = 1e5                       # all rates 1e5: the Sod tube fails near level 1122
    B["dx"][0] = 0.005
    B["left"][0], B["right"][0] = W.SOD_L, W.SOD_R
    a, b = _run(B, [700, 600], False), _run(B, [1300], True)
    _same(a, b)
    assert a[1][1][0] > 0 and a[1][1][1] == -1 and a[1][1][2] == -1

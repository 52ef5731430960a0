"""Host model of the copies that bring a misaligned row chunk to shared memory (vstream.cu: vs_span, vs_copy_tail): every
copy starts on 16 bytes, is a multiple of 16 bytes, stays inside its tensor and its slot region, and with the elements
copied one by one covers exactly what the sums and the draw read."""
import pytest

CHUNK = 4096   # bytes of a row chunk


def span(total, e0, nel, vw):
    m = e0 % vw
    n = -(-(m + nel) // vw) * vw
    tail = 0
    if e0 - m + n > total:
        n -= vw
        tail = m + nel - n
    return m, e0 - m, n, tail


@pytest.mark.parametrize("size,chunk_size", [(4, 4), (2, 2), (4, 2)])   # element, and the element that counts a chunk's ids
@pytest.mark.parametrize("V", [1, 3, 5, 8, 1023, 1025, 2047, 2049, 4099])
def test_copies_stay_inside_and_cover_the_ids(V, size, chunk_size):
    vw, el, rows = 16 // size, CHUNK // chunk_size, 7
    region = el * size + 32
    for row in range(rows):
        for c in range(-(-V // el)):
            e0, nel = row * V + c * el, min(el, V - c * el)
            assert (row * V + c * el) % vw == row * V % vw   # a row's chunks share its misalignment
            m, src, n, tail = span(rows * V, e0, nel, vw)
            assert src % vw == 0 and n % vw == 0 and n >= 0 and 0 <= tail < vw
            assert src >= 0 and src + n <= rows * V and src + n + tail <= rows * V
            assert (n + tail) * size <= region
            assert n + tail >= m + nel                     # the ids m .. m + nel - 1 are all there

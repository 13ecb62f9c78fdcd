"""The bytes bench.py divides by the time of its request classes: what a request cannot
do without, its cube written once. (Rows out of the PSF's reach of any particle are
neither written nor read before the convolution, so a count of passes over the
cube can exceed what is moved, and a rate the memory's.)"""
import bench


def test_request_class_bytes():
    assert bench.request_class_bytes(24, 300) == 24 * 300 * 300 * 3721 * 4

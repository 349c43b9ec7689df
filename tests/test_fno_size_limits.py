"""The sizes that fh_fno_create refuses, before it asks for device memory: the set of the
former shared-memory bound, 64 width^2 + 128 max_batch width <= 227 KB (and the transforms'
n^2, n and n modes terms, which no admissible size reaches), and the ranges."""
import pytest

import paper_1701_04685_gb300 as fh


def status(*size):
    try:
        fh.FNO(*size[:6], max_batch=size[6]).close()
    except fh.FhError as e:
        return e.status
    return 0


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1701_04685_gb300 import build
    build.build()


@pytest.mark.parametrize("width,batch", [(64, 1), (60, 1), (59, 2), (59, 1), (32, 40), (32, 41), (8, 64), (28, 50), (24, 64), (23, 64), (48, 13), (48, 14)])
def test_width_and_batch(width, batch):
    refused = 8 * 8 * width * width + 2 * batch * 8 * width * 8 > 227 * 1024
    got = status(4, 1, 1, width, 1, 1, batch)
    assert (got == -8) == refused   # FH_ERR_UNSUPPORTED; elsewhere success, or no device on a host without one


def test_no_grid_reaches_the_former_transform_bound():
    assert 128 * 128 * 4 + 128 * 8 + 128 * 64 * 8 <= 227 * 1024


@pytest.mark.parametrize("size", [(3, 1, 1, 4, 1, 1, 1), (129, 1, 1, 4, 1, 1, 1), (8, 0, 1, 4, 1, 1, 1), (8, 1, 65, 4, 1, 1, 1), (8, 1, 1, 4, 5, 1, 1),
                                  (8, 1, 1, 4, 1, 9, 1), (8, 1, 1, 4, 1, 1, 65)])
def test_ranges(size):
    assert status(*size) == -1

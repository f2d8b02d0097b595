"""GPU parity at the edges of the reduce_by_index * vjp's coefficient table in shared memory: fp32, 96 KB < table <=
200 KB and n >= 256 m; inputs, reference and tolerance are those of test_gpu_hist_tables.py."""
import numpy as np
import pytest

from paper_2310_03568_gb300 import adcomb
from tests import test_gpu_hist_tables as tables
from tests._gpu import ensure_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    ensure_lib()
    yield
    adcomb.debug_force_hist_strategy(-1)


@pytest.mark.parametrize("m,n", [(24_576, 256 * 24_576), (24_577, 256 * 24_577), (24_577, 256 * 24_577 - 1),
                                 (24_578, 256 * 24_578 + 3), (51_200, 256 * 51_200 + 1)])
def test_table_in_shared_memory(m, n):
    tables.test_hist_mul_tables(np.float32, m, n)

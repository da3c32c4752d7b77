"""Device allocations made to fail on the host (kc_test_fail_alloc: no memory is
filled): a call either reports KC_ERR_OOM_DEVICE and works when it is made again,
or gives the result it gives with memory to spare."""
import ctypes

import pytest

import paper_1712_03254_gb300 as kc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kc.lib()


@pytest.fixture
def fail_alloc():
    """fail_alloc(skip, fails): of this thread's allocations the `fails` after the next `skip` fail;
    returns how many there were since the last call."""
    f = kc.lib().kc_test_fail_alloc
    f.restype, f.argtypes = ctypes.c_uint64, (ctypes.c_uint64, ctypes.c_uint64)
    yield f
    f(0, 0)


@pytest.mark.parametrize("n", [0, 1])
def test_batch_object_that_cannot_be_made(fail_alloc, n):
    """kc_batch_create reports the failed allocation and returns (its clean-up once
    waited for a lock that the call itself held)."""
    fail_alloc(n, 1)
    with pytest.raises(kc.KcError) as e:
        kc.KcBatch()
    assert e.value.name == "KC_ERR_OOM_DEVICE"
    fail_alloc(0, 0)
    kc.KcBatch()

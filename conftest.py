"""Between tests: free what the last one left in reference cycles (tensors that
an expected error's traceback holds), so that the collector does not free it in
the middle of a test that counts torch's memory."""
import gc

import pytest


@pytest.fixture(autouse=True)
def young_garbage_collected():
    gc.collect(1)

import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a)")
    config.addinivalue_line("markers", "slow: long-running CPU test")


@pytest.fixture(scope="session")
def orc():
    import oracle

    oracle.build()
    return oracle


@pytest.fixture(autouse=True)
def _collect_after_gpu_tests(request):
    # the traceback that pytest.raises keeps holds the test's device tensors in
    # a cycle; collected in a later test, they would change the allocator's
    # figures while that test watches them
    yield
    if request.node.get_closest_marker("gpu"):
        import gc

        gc.collect()

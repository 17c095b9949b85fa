import os
import sys

import pytest

# One thread for numpy's BLAS.  Its idle threads spin for some 30 ms behind every
# norm of a longer vector, one on each core: a test that follows had its main
# thread preempted for 4 to 6 ms at a time (scheduler delay of the thread), longer
# than a small batch's whole solve.  Before numpy is first imported.
os.environ.setdefault("OPENBLAS_NUM_THREADS", "1")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a) and the built CUDA library")
    config.addinivalue_line("markers", "slow: larger CPU case (still within minutes)")


@pytest.fixture(scope="session")
def golden_dir():
    return os.path.join(ROOT, "tests", "golden")

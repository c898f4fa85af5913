import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

# Threads of the oracle's linear algebra sleep between calls instead of spinning on their cores: for
# milliseconds after a call they kept the serving runtime's workers from waking up, which the
# look-ahead test takes for a wrong admission order.  (Read when numpy is loaded.)
os.environ.setdefault("OPENBLAS_THREAD_TIMEOUT", "4")


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (GB300) and the built library")
    config.addinivalue_line("markers", "slow: CPU test that takes more than ~20 s")

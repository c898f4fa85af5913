import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

# Threads of the oracle's linear algebra sleep 2^18 cycles after a call (the library's default is 2^26):
# while they spin on their cores, the serving runtime's workers wake up milliseconds late, which the
# look-ahead test takes for a wrong admission order.  (Much less, and the oracle itself takes twice as
# long.  Read when numpy is loaded.)
os.environ.setdefault("OPENBLAS_THREAD_TIMEOUT", "18")


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (GB300) and the built library")
    config.addinivalue_line("markers", "slow: CPU test that takes more than ~20 s")

import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (GB300) and the built library")
    config.addinivalue_line("markers", "slow: takes more than a few seconds")


@pytest.fixture(autouse=True)
def tuning_as_before():
    """A test that tunes the matcher leaves the tuning it found to the next one."""
    tm = sys.modules.get("paper_1810_00980_gb300.tm")
    before = tm.get_tuning() if tm is not None and tm._LIB is not None else None
    yield
    if before is not None:
        tm.set_tuning(**before)


@pytest.fixture(scope="session")
def oracle_mod():
    import oracle
    oracle.core.build()
    return oracle

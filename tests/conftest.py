import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a) and the built library")
    config.addinivalue_line("markers", "slow: full-size parity case")


@pytest.fixture(autouse=True)
def no_tile_shape_set():
    """Every test starts with the library's own choice of tile shapes, whatever the last one set."""
    crys = sys.modules.get("paper_2003_01178_gb300")
    if crys is not None and crys._lib is not None:
        for op in range(crys.NUM_OPS):
            crys.crys_reset_tile(op)


@pytest.fixture(scope="session")
def orc():
    import oracle
    oracle.build()
    return oracle

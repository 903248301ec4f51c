"""lks_workspace_bytes / lks_set_workspace reject NULL handles before any device work."""
import pytest

from paper_2112_13930_gb300 import build, lks


@pytest.fixture(scope="module")
def lib():
    build.build()
    return lks.load()


def test_null_handle(lib):
    assert lib.lks_workspace_bytes(None) == 0
    assert lib.lks_set_workspace(None, None, 0) == lks.LKS_EINVAL

"""The binding's mirror of mhc_forward_path has the layout of include/mhc.h (as test_abi_layout), and
mhc_forward_info refuses what it cannot answer without a GPU."""
import ctypes
import os
import shutil

import pytest

from paper_1411_3691_gb300 import build, mhc
from test_abi_layout import _c_layout


@pytest.mark.skipif(shutil.which("gcc") is None, reason="no host C compiler")
def test_layout(tmp_path):
    fields = [name for name, _ in mhc.ForwardPath._fields_]
    got = _c_layout(tmp_path, "mhc_forward_path", fields)
    assert got["size"] == ctypes.sizeof(mhc.ForwardPath)
    assert all(got[f] == getattr(mhc.ForwardPath, f).offset for f in fields)


def test_null_arguments():
    if not os.path.exists(mhc.LIB_PATH):
        build.build()
    assert mhc.lib().mhc_forward_info(None, None, None) == mhc.MHC_EINVAL

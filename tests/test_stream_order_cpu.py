"""Transfers to the device against the kernels that read them.  The library's
streams do not wait for the legacy stream, and a blocking copy from pageable
memory runs on that and may return before its data has arrived, as a blocking
memset may.  So the sources write device memory with the forms that name a
stream, and use the blocking forms for device to host copies only."""
import os
import re

import pytest

from paper_2007_00558_gb300 import build


def _code(path):
    s = re.sub(r"//[^\n]*", "", open(path).read())
    return re.sub(r"/\*.*?\*/", "", s, flags=re.S)


@pytest.mark.parametrize("path", build.sources(), ids=os.path.basename)
def test_device_writes_name_their_stream(path):
    for call in re.findall(r"\bcuda(?:Memset|Memcpy)(?:2D|3D|ToSymbol)?\s*\(.*?;", _code(path), flags=re.S):
        assert call.startswith("cudaMemcpy") and "cudaMemcpyDeviceToHost" in call, call

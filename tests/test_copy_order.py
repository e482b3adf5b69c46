"""Copies and fills that the host asks for and kernels on non-blocking streams read.
cudaMemcpy from pageable memory and cudaMemset may return before the data is in place, and
a non-blocking stream does not wait for the legacy stream they run on: every such call in
the sources is followed, in its function, by a wait for that stream or for the device."""
import glob
import os
import re

import pytest

from paper_2412_03489_gb300 import build as hb

CALL = re.compile(r"\bcudaMemset\(|\bcudaMemcpy\((?:[^;]*?)cudaMemcpyHostToDevice")
WAIT = re.compile(r"cudaStreamSynchronize\(cudaStreamLegacy\)|cudaDeviceSynchronize\(\)")


@pytest.mark.parametrize("name", sorted(os.path.basename(f) for f in glob.glob(os.path.join(hb.CSRC, "*.cu"))))
def test_copies_are_waited_for(name):
    with open(os.path.join(hb.CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    for m in CALL.finditer(text):
        end = text.index("\n}\n", m.end())   # of the function
        assert WAIT.search(text, m.end(), end), f"{name}: {text[m.start():m.start() + 80]!r}"

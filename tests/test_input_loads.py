"""How the product kernels read their inputs. A product is launched before the
previous kernel on its stream has ended, and that kernel may write x, X or gu.
So they are read by coherent loads that stay behind griddepcontrol.wait, never
by read-only loads (__ldg, ld.global.nc), which need data that is constant over
the whole kernel. CPU only (source text)."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_02893_gb300", "csrc")


@pytest.mark.parametrize("name", ["vbq_gemm.cu", "vbq_gemv.cu", "vbq_device.cuh"])
def test_inputs_are_read_coherently(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    assert not re.search(r"__ldg|__ldcs|__ldlu|ld\.global\.nc", text)
    if name == "vbq_device.cuh":
        loads = re.findall(r"\bldg_input_\w+\([^)]*\)\s*\{(.*?)\n\}", text, re.S)
        assert len(loads) == 3 and all("asm volatile" in b and '"memory"' in b for b in loads)
    else:
        assert "ldg_input_" in text
        # nothing else goes through the input pointers
        assert not re.search(r"reinterpret_cast<const \w+\*>\((?:x|X|gu|xg|src)\b[^;]*\)\s*\[", text)
        assert not re.search(r"\*reinterpret_cast<const \w+\*>\((?:x|X|gu|xg|src)\b", text)

"""vibe_get_wavefronts only copies: it must work whichever device is current.

Device-to-host copies do; an allocation or a kernel of its own would land on the current device with pointers
of the handle's device, an illegal access where the two differ. One GPU cannot show that (and no test may cause
it), so the function's text is held to the one CUDA call it may make. Its results are compared with the
definition in test_gpu_parity.py.
"""
import os
import re

from paper_2508_15743_gb300 import build as B


def body(name):
    text = open(os.path.join(B.CSRC, "vibe_api.cu")).read()
    text = re.sub(r"//[^\n]*", "", text)
    start = text.index("{", text.index(f"int {name}("))
    depth = 0
    for i in range(start, len(text)):
        depth += (text[i] == "{") - (text[i] == "}")
        if depth == 0:
            return text[start:i]
    raise AssertionError(f"{name} has no end")


def test_wavefronts_make_no_device_work_but_copies():
    calls = set(re.findall(r"\b(cuda\w+|dalloc|vibe::\w+|k_\w+)\s*(?:<<<|\()", body("vibe_get_wavefronts")))
    assert calls == {"cudaMemcpy"}

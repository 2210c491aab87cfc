"""Tile heights and ring depths follow the device's SM count, which prop_create and
prop_forward_noalloc ask for; no rule holds one chip's number."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_10519_gb300", "csrc")


def text(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def test_the_sm_count_is_the_device_s():
    for name in ("runtime.cu", "noalloc.cu"):
        assert re.search(r"MultiProcessorCount, dev\)\);\s*P->sms = sms;", text(name)), name
    for name in ("elastic2d.cu", "stencil_tma.cu", "tti_sp_tma.cu", "tma.cuh"):
        assert not re.search(r"[<>]=? *152\b", text(name)), name

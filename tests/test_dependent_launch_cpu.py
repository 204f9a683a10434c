"""What a kernel may do before the one that it depends on has completed, read from its source.

A kernel launched with the programmatic attribute may start before its predecessor in the stream
has written its results, and only griddepcontrol.wait (pdl_wait) makes them visible.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2111_02534_gb300", "csrc")


def _functions(name):
    """Name and body of every device function of a source file, without comments."""
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    got = {}
    for m in re.finditer(r"\n(?:__global__|template|__device__)[^;{}=]*?\b(\w+)\((?:[^()]|\([^()]*\))*\)\s*\{",
                         text):
        end = text.index("\n}\n", m.end())
        got[m.group(1)] = text[m.end():end]
    return got


def test_the_fused_mode_product_reads_nothing_before_its_wait():
    # the kernel that builds the image of a mode is the predecessor of that mode's first product
    body = _functions("oz_mode.cu")["k_mode_product"]
    before = body[:body.index("pdl_wait()")]
    for what in ("image", "eK", "psi", "out"):
        assert f"g.{what}" not in before, what
        assert f"g.{what}" in body[len(before):], what

"""Rules of the kernels that no run can show, read from their sources.

What a kernel may do before the one that it depends on has completed: launched with the
programmatic attribute, it may start before its predecessor in the stream has written its results,
and only griddepcontrol.wait (pdl_wait) makes them visible.  And the alignment of shared memory.
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


_ALLOCATING = [(os.path.basename(path), name) for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")))
               for name, body in _functions(os.path.basename(path)).items() if "tmem_alloc(" in body]


def test_the_kernels_with_tensor_memory_are_found():
    assert {name for _, name in _ALLOCATING} >= {"oz_tile", "k_oz_gemm1p", "k_mode_product",
                                                 "k_fold_gemm", "k_tf32_gemm"}


@pytest.mark.parametrize("source,name", _ALLOCATING)
def test_dependents_start_after_the_tensor_memory_is_allocated(source, name):
    # a dependent's CTA on the same SM could otherwise take the tensor memory first and then wait
    # for this kernel, whose allocation would wait for that CTA: the one wait without a limit
    body = _functions(source)[name]
    if "pdl_trigger()" not in body:
        return
    alloc = body.index("tmem_alloc(")
    held = body.index("__syncthreads()", alloc)
    assert body.index("pdl_trigger()") > held
    assert "pdl_entry()" not in body


def test_shared_memory_read_as_float4_is_declared_aligned():
    # the layer products read their slabs, at the start of the dynamic array, as float4
    with open(os.path.join(CSRC, "mlp.cu")) as f:
        text = f.read()
    assert "reinterpret_cast<const float4 *>" in text
    declared = re.findall(r"extern __shared__([^;]*);", text)
    assert len(declared) >= 4
    assert all("__align__(16)" in d for d in declared), declared

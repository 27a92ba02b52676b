"""Kernels launched by programmatic dependent launch are resident while their predecessors
still write what they read.  So each begins with the wait, and none reads through the
non-coherent path (__ldg, ld.global.nc, or a __restrict__ pointer to const), which is defined
only for memory that is constant during a kernel's whole life."""
from __future__ import annotations

import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2410_00486_gb300" / "csrc"


def code(path: Path) -> str:
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", path.read_text(), flags=re.S)


def is_chain(text: str) -> bool:
    return bool(re.search(r"\blaunch\(\s*k", text))


CHAIN = sorted(p.name for p in CSRC.glob("*.cu*") if is_chain(code(p)))


def test_the_chain_is_found():
    assert {"adam.cu", "binsort.cu", "preprocess.cu", "render_bwd.cu", "render_fwd.cu"} <= set(CHAIN)


@pytest.mark.parametrize("name", CHAIN + ["raster.cuh"])
def test_no_read_through_the_non_coherent_path(name):
    text = code(CSRC / name)
    assert "<<<" not in text          # a file of the chain launches nothing the ordinary way
    assert not re.findall(r"__ldg|ld\.global[.\w]*\.nc|__ldlu|__ldcs", text)
    assert not re.findall(r"const\s+\w+(?:\s+\w+)*\s*\*\s*__restrict__", text)


@pytest.mark.parametrize("name", CHAIN)
def test_every_kernel_begins_with_the_wait(name):
    text = code(CSRC / name)
    for at in (m.end() for m in re.finditer(r"__global__", text)):
        body = text[text.index("{", at) + 1:].lstrip()
        assert body.startswith("pdl_begin("), text[at:at + 120]

"""Copies to the device are ordered with the kernels that read them.

A context's stream does not wait for the legacy stream, and a plain cudaMemcpy
from pageable memory returns when the data is staged, not when it has reached
the device: a kernel launched right behind it on the context's stream can read
what the memory held before (and follow it as an index)."""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_11082_gb300", "csrc")


@pytest.mark.parametrize("name", sorted(os.listdir(CSRC)))
def test_no_copy_on_the_legacy_stream(name):
    """Uploads and clears name a stream (the copies back follow a wait)."""
    with open(os.path.join(CSRC, name)) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    calls = re.findall(r"\b(?:cudaMemcpy|cudaMemset|cudaMemcpyToSymbol)\s*\([^;]*;", src)
    assert [c for c in calls if "cudaMemcpyDeviceToHost" not in c] == []


@pytest.mark.gpu
def test_assembly_in_recycled_memory():
    """Assemblies whose uploads land where another problem's data was, with the
    reference field computed and handed in. K_eff differs by the order of the
    element sums only (1e-13 of its largest entry), M likewise."""
    pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1906_11082_gb300 import nm
    from synth.model import layered_planet
    ctx = nm.Context(0)
    mesh, model = layered_planet(h=0.2, seed=5)
    other = layered_planet(h=0.15, seed=6)
    first = nm.Problem(ctx, mesh, model)
    ref = [first.export(w)[2] for w in range(5)]
    p2 = first.unodes()[1]
    g = np.zeros((p2.max() + 1, 3))
    g[p2] = first.gravity()
    first.free()
    for i in range(4):
        nm.Problem(ctx, *other).free()
        P = nm.Problem(ctx, mesh, model, gprime=g if i % 2 else None)
        for w in range(5):
            v = P.export(w)[2]
            assert np.abs(v - ref[w]).max() <= 1e-13 * np.abs(ref[w]).max()
        P.free()

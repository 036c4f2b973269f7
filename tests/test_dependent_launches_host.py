"""Kernels that can be launched dependently (launch_pdl) are resident while the launch before them still
writes its results, so nothing that launch writes may be read early or through the read-only path.

Read from the sources: such a kernel waits (pdl_wait, or pdl_begin, which loads the twiddle table
first) before its first statement that touches memory, and every array that it declares const and
__restrict__, or loads with __ldg, was complete before the launch before it began."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_1703_00879_gb300" / "csrc"

# const __restrict__ parameters and __ldg operands, and the launch that wrote them
COMPLETE = {
    "twg": "twiddle table, uploaded when the context is made",
    "tab": "growth table, uploaded with the model",
    "phi1": "seeds, initial conditions", "phi2": "seeds, initial conditions",
    "sx": "drift, before the force passes", "sy": "drift, before the force passes", "sz": "drift, before the force passes",
    "ax": "kick, before the LPT passes", "ay": "kick, before the LPT passes", "az": "kick, before the LPT passes",
    "Ax": "LPT pass, before the force passes or one boundary earlier", "Ay": "as Ax", "Az": "as Ax",
    "hdr": "step counter, advanced before the force passes (k_kick_drift_deposit)",
    "rho": "deposit, before the transforms that lead to k_plane_screen",
}
# read by cp.async only (coherent at L2, issued after the wait)
ASYNC = {"k_plane_r2c": {"in"}, "k_plane_screen": {"w_in"}}


def _kernels():
    """{name: (parameters, body)} of the __global__ functions that wait for the launch before them."""
    found = {}
    for f in sorted(CSRC.glob("*.cu")):
        text = re.sub(r"//[^\n]*", "", f.read_text())
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\(", text):
            i, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            start = j = text.index("{", i) + 1
            depth = 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[j], 0)
                j += 1
            if re.search(r"\bpdl_(wait|begin)\b", text[start:j]):
                found[m[1]] = (text[m.end():i - 1], text[start:j - 1])
    return found


KERNELS = _kernels()


def test_every_dependent_launch_has_a_kernel_that_waits():
    launched = set()
    for f in CSRC.glob("*.cu"):
        text = re.sub(r"//[^\n]*", "", f.read_text())
        for m in re.finditer(r"launch_(?:pdl|with)\(", text):
            head = text[max(0, text.rfind("\ncudaError_t", 0, m.start()), text.rfind("\nstatic cudaError_t", 0, m.start())):text.index(";", m.end())]
            launched |= set(re.findall(r"\bk_\w+", head)) - {"k_drift_deposit_box", "k_gather_kick_box"}
    assert launched and launched == set(KERNELS)


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_inputs_of_dependent_kernels(name):
    params, body = KERNELS[name]
    declared = set(re.findall(r"const \w+\* __restrict__ (\w+)", params))
    assert declared <= set(COMPLETE) | ASYNC.get(name, set())
    assert set(re.findall(r"__ldg\((\w+)", body)) <= set(COMPLETE)
    # nothing but the twiddle table is touched before the wait
    before = re.split(r"\bpdl_(?:wait|begin)\b", body)[0]
    assert not re.search(r"\bresolve\(|->|\bissue\(|\bstage_|\bmoved\(|cp_async", before)

"""The order that programmatic dependent launches rest on, read off the CUDA sources: a kernel lets the next one
start (pdl_trigger) only after its own wait for the kernel before it (pdl_wait), and whatever is launched with
launch_pdl has such a wait.  What a kernel reads before its wait is then at least two kernels old."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_18073_gb300", "csrc")


def kernels():
    """name -> body of every __global__ function"""
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\b", text):
            brace = text.find("{", m.end())
            name = re.findall(r"(\w+)\s*\(", re.sub(r"__\w+__\s*\([^)]*(?:\([^)]*\))*[^)]*\)", "", text[m.end():brace]))
            depth, i = 0, brace
            while True:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
                if depth == 0:
                    break
            if name:
                out[name[0]] = text[brace:i]
    return out


def test_trigger_follows_wait():
    K = kernels()
    triggers = {k: b for k, b in K.items() if "pdl_trigger(" in b}
    assert len(triggers) >= 5
    for name, body in triggers.items():
        assert 0 <= body.find("pdl_wait(") < body.find("pdl_trigger("), name


def test_dependent_launches_wait():
    K = kernels()
    text = "".join(open(p).read() for p in glob.glob(os.path.join(CSRC, "*.cu")))
    launched = {n for n in re.findall(r"launch_pdl\((k\w+)", text) if n != "k"}
    assert launched and launched <= set(K)
    for name in launched:
        assert "pdl_wait(" in K[name], name

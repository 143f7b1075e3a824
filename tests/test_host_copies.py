"""Asynchronous copies from host memory (csrc/solver.cu).  CUDA does not promise
that a copy from pageable memory has read its source when the call returns (a
GPU that reads pageable memory through the host's page tables need not stage
it), so the source has to be pinned memory that the object keeps, or the stream
has to be waited for before the block that declares the source ends.  Checked
on the source text: the failure itself would be a kernel reading wild pointers."""
import os
import re

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "..", "paper_2212_01110_gb300", "csrc", "solver.cu")
PINNED = {("copy_many", "h")}   # Batch::tab_host, waited for before it is written again


def _blocks(text):
    """(begin, end) of every brace block, innermost last for a given place."""
    out, stack = [], []
    for i, c in enumerate(text):
        if c == "{":
            stack.append(i)
        elif c == "}" and stack:
            out.append((stack.pop(), i))
    return sorted(out)


def unwaited_copies(text):
    text = re.sub(r"//[^\n]*", lambda m: " " * len(m.group()), text)
    text = re.sub(r'"(\\.|[^"\\\n])*"', lambda m: " " * len(m.group()), text)
    blocks = _blocks(text)
    bad = []
    for m in re.finditer(r"cudaMemcpyAsync\(([^;]*?)cudaMemcpyHostToDevice", text):
        source = m.group(1).split(",")[1].strip()
        name = re.match(r"&?\s*(\w+)", source).group(1)
        around = [b for b in blocks if b[0] < m.start() < b[1]]
        func = next((b for b in around if re.search(r"\)\s*$", text[:b[0]])), around[0])
        declared = func
        for b in around[around.index(func):]:   # the innermost block that declares the source
            if re.search(r"[\w>*&]\s+[*&]?%s\s*(=|;|\(|\{|\[|,)" % name, text[b[0]:m.start()]):
                declared = b
        head = text[:func[0]].rstrip()
        caller = re.findall(r"(\w+)\s*\(", head[-600:])
        if any((c, name) in PINNED for c in caller):
            continue
        if "cudaStreamSynchronize" not in text[m.end():declared[1]]:
            bad.append((text.count("\n", 0, m.start()) + 1, source))
    return bad


def test_sources_outlive_their_copies():
    with open(SRC) as f:
        text = f.read()
    assert text.count("cudaMemcpyAsync") > 10
    assert unwaited_copies(text) == []


@pytest.mark.parametrize("wait,found", [("", 1), ("CUDA_TRY(cudaStreamSynchronize(st));", 0)])
def test_the_check_sees_a_local_source(wait, found):
    text = """
static int solve(int cta) {
  if (cta) {
    const View hb = make();
    CUDA_TRY(cudaMemcpyAsync(dev, &hb, sizeof(hb), cudaMemcpyHostToDevice, st));
    %s
    launch(dev);
  }
  CUDA_TRY(cudaStreamSynchronize(st));
}
""" % wait
    assert len(unwaited_copies(text)) == found

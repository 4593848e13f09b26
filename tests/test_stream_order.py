"""Device buffers are cleared and filled in stream order. A cudaMemset, and a
cudaMemcpy from pageable memory, may still be under way on the null stream when the
call returns, and streams that do not block with it (PyTorch's, the context's own) do
not wait for it."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1607_02904_gb300", "csrc")


def test_no_clears_or_uploads_on_the_null_stream():
    found = []
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, name)) as f:
                text = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
            found += [(name, m.group(0)) for m in re.finditer(r"\bcudaMem(set|cpy)(2D)?\s*\(", text)]
    assert not found

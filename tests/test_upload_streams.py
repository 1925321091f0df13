"""Buffers of an operator are uploaded and cleared on the stream that its kernels run on.  A copy or a memset on the
default stream is not ordered with a non-blocking stream (a serving worker's, a caller's): a kernel there
could read its job list before it has landed, or write a Krylov vector before the memset has.  Only
the mesh, which waits for the default stream itself, may leave the stream out."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_06184_gb300", "csrc")


def test_every_upload_names_its_stream():
    bare = []
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cpp")):
            continue
        src = open(os.path.join(CSRC, name)).read()
        if name == "api.cu":  # sldm_mesh_create, up to its own wait
            i = src.index("int sldm_mesh_create(")
            j = src.index("SLDM_CUDA(cudaStreamSynchronize(0));", i)
            src = src[:i] + src[j:]
        for m in re.finditer(r"\.(upload|zero)\(((?:[^()]|\([^()]*\))*)\)", src):
            args = [a for a in m.group(2).split(",") if a.strip()]
            if len(args) < (2 if m.group(1) == "upload" else 1):
                bare.append((name, m.group(0)))
    assert not bare, bare

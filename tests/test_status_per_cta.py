"""The status word is read once per CTA.

In the checked build an index check may set the status while CTAs of the same
launch are still starting.  Threads of a CTA that read it one by one could
then part: those that return never reach the CTA's barriers (the half-tile
forward counts 64 threads at its own, whether or not one has exited) and
never take the item the others go on with.  So no kernel reads the word but
through step_failed(), which gives a whole CTA one answer."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_03092_gb300", "csrc")


def _code(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def test_kernels_read_the_status_through_step_failed():
    direct, through = [], 0
    for name in sorted(os.listdir(CSRC)):
        code = _code(os.path.join(CSRC, name))
        code, n = re.subn(r"\bstep_failed\((?:A\.hdr->status|__ldcg\(&A\.hdr->status\))\)", "", code)
        through += n
        direct += [(name, m.group(0).strip()) for m in re.finditer(r"[^\n]*hdr->status[^\n]*", code)]
    writes = (r"hdr->status = SPLAT2D_ERR_CAPACITY;", r"atomicCAS\(.*&hdr->status")
    assert [u for u in direct if not any(re.search(w, u[1]) for w in writes)] == []
    # scatter, the two bucket sorts, the chain rule and the six kernels of render.cu
    assert through == 10
    body = _code(os.path.join(CSRC, "splat2d_internal.cuh")).split("bool step_failed(", 1)[1].split("\n}", 1)[0]
    assert re.search(r"#ifdef S2D_CHECKS\s+return __syncthreads_or\(status != 0\);", body)

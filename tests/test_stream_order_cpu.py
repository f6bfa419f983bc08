"""Every copy and fill of the library is ordered on the stream that uses it.

The library's streams are non-blocking ones: they do not wait for the legacy
default stream, and a blocking copy there (cudaMemcpy, cudaMemset) may return
before its bytes have reached the device.  So the sources use the stream-ordered
forms only.  Checked on the source text: such a race shows on a GPU by chance."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_07577_gb300", "csrc")


def _sources():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(f) as fh:
            text = fh.read()
        yield os.path.basename(f), re.sub(r"//[^\n]*", "", text)


def test_no_copy_or_fill_without_a_stream():
    bad = [(name, m.group(0)) for name, text in _sources()
           for m in re.finditer(r"\bcudaMem(cpy|set)(2D|3D|ToSymbol|FromSymbol)?\s*\(", text)]
    assert not bad, bad


def test_overlapped_steps_promise_nothing_about_each_others_buffers():
    """spring_step_kernel starts while the launch before it still writes its
    position and velocity buffers: a read-only __restrict__ pointer to them would
    allow loads that do not see those writes."""
    text = dict(_sources())["springs.cu"]
    sig = re.search(r"\bspring_step_kernel\s*\((.*?)\)\s*\{", text, re.S).group(1)
    buffers = [p for p in sig.split(",") if "Quad<" in p]
    assert len(buffers) == 3 and not any("__restrict__" in p for p in buffers), buffers

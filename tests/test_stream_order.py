"""Every host-to-device copy and every memset of the library is ordered on the stream that its kernels
run on (source check, CPU).  cudaMemcpy from pageable memory may return before the data has reached
the device, cudaMemset before it has run, and a context on a non-blocking stream (a serving
worker's, torch.cuda.Stream) waits for neither: a kernel launched next could read what was there
before, pointers of a chain program among it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_05285_gb300", "csrc")


def test_uploads_and_memsets_are_stream_ordered():
    files = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))
    assert files
    for path in files:
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for call in re.findall(r"\bcudaMemcpy(?:2D|3D|ToSymbol)?\s*\([^;]*;", text):
            assert "cudaMemcpyDeviceToHost" in call, (os.path.basename(path), call)
        assert not re.search(r"\bcudaMemset(?:2D|3D)?\s*\(", text), os.path.basename(path)

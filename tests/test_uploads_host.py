"""Every copy of host arrays to the device that a kernel on a caller's stream reads goes through upload
or upload_symbol, which wait: a copy from pageable memory may return before its last part has arrived, and
non-blocking streams do not wait for the legacy stream. (Copies ordered on the caller's own stream are
cudaMemcpyAsync.) The missing wait is a race, so it is looked for in the sources."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_uploads_wait():
    bare = []
    for path in glob.glob(os.path.join(ROOT, "paper_1211_0540_gb300", "csrc", "*")):
        with open(path) as fp:
            text = fp.read()
        for name in ("upload", "upload_symbol"):  # the helpers' own copies, with their waits
            text = re.sub(r"cudaError_t %s\((?:.|\n)*?\n}" % name,
                          lambda m: "" if "cudaStreamSynchronize(cudaStreamLegacy)" in m.group(0) else m.group(0), text)
        text = re.sub(r"\s+", " ", text)
        for m in re.finditer(r"cudaMemcpy\((?:[^()]|\([^()]*\))*\)|cudaMemcpyToSymbol\(", text):
            if "DeviceToHost" not in m.group(0) and "DeviceToDevice" not in m.group(0):
                bare.append((os.path.basename(path), m.group(0)))
    assert not bare, bare

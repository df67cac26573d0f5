"""Rules that the kernel sources keep, read from their text (no GPU)."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2607_00790_gb300", "csrc")


def sources():
    files = sorted(f for e in ("*.cu", "*.cuh", "*.h") for f in glob.glob(os.path.join(CSRC, e)))
    assert files
    return {os.path.basename(f): open(f).read() for f in files}


def test_no_multicast():
    """A CTA loads and releases its own tiles only: one process per GPU runs this library, and an arrival
    at another CTA's barrier could come after that CTA has left."""
    assert [f for f, s in sources().items() if "multicast" in s] == []


def test_register_split(tmp_path):
    """What the warps of the residue product ask for by setmaxnreg is there at launch (an increase waits until it
    is), as compiled."""
    from paper_2607_00790_gb300 import build
    src = sources()["crt_gemm.cu"]
    val = {k: int(v) for k, v in re.findall(r"#define (CR_\w+) (\d+)\b", src)}
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-Xptxas", "-v", "-c", os.path.join(CSRC, "crt_gemm.cu"),
                        "-o", str(tmp_path / "x.o")], capture_output=True, text=True, check=True)
    regs = int(re.search(r"k_zgemm_crt.*?Used (\d+) registers", r.stderr, re.S).group(1))
    issue = val["CR_THREADS"] - val["CR_EPI"]
    assert issue * val["CR_REGS_ISSUE"] + val["CR_EPI"] * val["CR_REGS_EPI"] <= val["CR_THREADS"] * regs

"""Register spills of the batched step kernel, from the compiler's report
(-Xptxas -v) on the one instance that the 512-instance sweep launches."""
import os
import re
import subprocess

from paper_2412_16843_gb300 import build


def test_batched_step_spills_little(tmp_path):
    """1024 threads leave 64 registers a thread; what the step's cell loops
    spill goes through L1 in every cell.  Bound: 300 bytes of stores and 700
    of loads (248 and 576 when it was set; 438 and 840 made the sweep of 512
    instances 8 % slower)."""
    with open(os.path.join(build.CSRC, "k_persist.cu")) as f:
        src = f.read()
    # the kernels without their host code, which instantiates every size
    src = src[:src.index("size_t persist_tail_layout(")]
    src = src[:src.rindex("}  // namespace\n")]
    src += "template __global__ void k_batch_persist<float, 2, 1024>(BatchArgs<float>);\n}\n}\n"
    cu = tmp_path / "one.cu"
    cu.write_text(src.replace("../../include/cdi.h", "cdi.h"))
    r = subprocess.run([build.nvcc()] + build.NVCC_FLAGS + ["-I", build.CSRC, "-Xptxas", "-v", "-c", str(cu), "-o",
                                                            str(tmp_path / "one.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    m = re.search(r"k_batch_persist.*?(\d+) bytes spill stores, (\d+) bytes spill loads.*?Used (\d+) registers",
                  r.stderr, re.S)
    assert m, r.stderr
    stores, loads, registers = (int(x) for x in m.groups())
    assert registers <= 64 and stores <= 300 and loads <= 700, m[0]

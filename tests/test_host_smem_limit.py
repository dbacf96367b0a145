"""The opt-in to more than 48 KB of dynamic shared memory belongs to a kernel in
the whole process: a limit set to one launch's size can be lowered by another
host thread between that setting and the launch.  So the limit is set in one
place (allow_smem), to a value that depends on the kernel alone, and only ever
raised."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_one_limit_per_kernel():
    calls = []
    for fn in sorted(glob.glob(os.path.join(ROOT, "paper_2103_01874_gb300", "csrc", "*"))):
        text = re.sub(r"//[^\n]*", "", open(fn).read())
        calls += [(os.path.basename(fn), m.group(1).strip(), text[:m.start()])
                  for m in re.finditer(r"cudaFuncSetAttribute\s*\(([^;]*)\)\s*;", text)
                  if "MaxDynamicSharedMemorySize" in m.group(1)]
    assert [(f, a.split(",")[-1].strip()) for f, a, _ in calls] == [("ppe_internal.h", "most")], calls
    body = calls[0][2].rsplit("cudaError_t allow_smem(K kernel, size_t bytes)", 1)[1]
    most = re.search(r"most = ([^;]*);", body).group(1)
    assert "bytes" not in most and "kSmemPerCta - a.sharedSizeBytes" in most, most
    assert re.search(r"if \(a\.maxDynamicSharedSizeBytes >= most\) return cudaSuccess;", body), "lowered"

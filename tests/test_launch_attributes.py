"""Kernel attributes belong to the current device: a launcher sets the ones it needs before
every launch.  One that remembers in a static flag that it has set them fails on a second
device of the process, and host threads race on the flag.  With one device neither shows at
run time, so the sources are searched."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_launcher_remembers_an_attribute():
    found, setters = [], 0
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2007_03847_gb300", "csrc", "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        setters += text.count("cudaFuncSetAttribute(")
        found += [f"{os.path.basename(path)}: {m.group(0)}"
                  for m in re.finditer(r"\bstatic\s+(?:std::atomic<)?(?:bool|int|std::once_flag)\b[^;(]*[;=]", text)
                  if "constexpr" not in m.group(0)]
    assert setters >= 5
    assert not found, found

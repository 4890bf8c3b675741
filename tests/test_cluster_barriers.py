"""The kernels' cluster barriers, read from the sources (no GPU): the .aligned forms are undefined in a warp whose lanes have parted."""
import os
import re


def test_every_cluster_barrier_brings_its_warp_together_first(repo_root):
    csrc = os.path.join(repo_root, "paper_2511_18793_b200", "csrc")
    seen = 0
    for name in sorted(os.listdir(csrc)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(csrc, name)).read())
        for m in re.finditer(r'asm volatile\("barrier\.cluster\.(?:arrive|wait)[.a-z]*\.aligned;', text):
            seen += 1
            assert re.search(r"__syncwarp\(\);\s*$", text[: m.start()]), (name, text[m.start(): m.end()])
    assert seen >= 3

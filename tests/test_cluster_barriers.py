"""The kernels' cluster barriers and collective loads, read from the sources (no GPU): the .aligned forms are undefined in a warp whose lanes
have parted."""
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


def test_reads_of_a_peer_are_used_before_the_arrival_that_lets_it_go(repo_root):
    """A CTA's shared memory may be gone once all have arrived.  Behind the last read of a peer's comes an arrival that releases, or one
    that does not and in front of it an instruction of the whole warp that takes what was read -- also where nothing is stored."""
    csrc = os.path.join(repo_root, "paper_2511_18793_b200", "csrc")
    seen = 0
    for name in sorted(os.listdir(csrc)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(csrc, name)).read())
        reads = [m.end() for m in re.finditer(r"[=*] ?ld_peer\w*\(", text)]
        if reads:
            seen += 1
            arrival = re.search(r"cluster_(?:arrive|sync)\w*", text[reads[-1]:])
            between = text[reads[-1]: reads[-1] + arrival.start()]
            assert arrival.group() in ("cluster_arrive", "cluster_sync_all") or re.search(r"__shfl_sync\(0xffffffffu, x\.x, lane\)", between), name
    assert seen == 2


def test_a_loop_of_collective_loads_brings_its_warp_together(repo_root):
    """Between a collective load and the next round's, a branch for the rows that exist: the warp meets behind it."""
    csrc = os.path.join(repo_root, "paper_2511_18793_b200", "csrc")
    seen = 0
    for name in sorted(os.listdir(csrc)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(csrc, name)).read())
        for m in re.finditer(r"tmem_ld\w*\([^;]*;\s*if \(live[^{]*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            seen += 1
            assert re.match(r"\s*__syncwarp\(\);", text[i:]), (name, text[m.start(): m.end()])
    assert seen == 1

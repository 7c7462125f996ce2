"""Warp-aligned barriers of the CUDA sources (no GPU needed): the `.aligned`
forms (bar.sync is one) need every lane of a warp to execute them together, so
each stands directly behind a __syncwarp(), whatever loop or branch its caller
came from."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_21291_gb300", "csrc")
BARRIER = re.compile(r'asm volatile\("(bar\.sync|barrier\.cluster\.(arrive|wait)[.\w]*\.aligned)')


def test_aligned_barriers_follow_a_warp_barrier():
    seen, bare = 0, []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        prev = ""
        for no, line in enumerate(open(path), 1):
            code = line.split("//")[0].strip()
            if not code:
                continue
            if BARRIER.search(code):
                seen += 1
                if prev != "__syncwarp();" and not BARRIER.search(prev):
                    bare.append(f"{os.path.basename(path)}:{no}")
            prev = code
    assert seen >= 3 and not bare, bare

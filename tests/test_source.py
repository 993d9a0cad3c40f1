"""Rules that the device code keeps by its form (runs without a GPU)."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_aligned_cluster_barriers_follow_a_syncwarp():
    """barrier.cluster.*.aligned needs all lanes of the warp at it together; a loop or a branch in front of it may have split them."""
    found = 0
    for f in glob.glob(os.path.join(ROOT, "paper_2606_12370_b200", "csrc", "*.cu*")):
        text = re.sub(r"//[^\n]*", "", open(f).read())
        for m in re.finditer(r'asm volatile\("barrier\.cluster\.(arrive|wait)[a-z.]*\.aligned', text):
            found += 1
            assert text[:m.start()].rstrip().endswith("__syncwarp();"), (os.path.basename(f), m.group(0))
    assert found >= 2

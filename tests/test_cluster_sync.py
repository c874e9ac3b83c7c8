"""The cluster barriers of the one-launch k-means++ seeding, by reading the source (a missing wait
is not provoked on a GPU): every barrier is reached by converged warps, and another CTA's shared
memory is only written between two barriers, the first of which shows that the CTA runs and the
last that it has not ended."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_04477_gb300", "csrc")


def _sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            text = open(os.path.join(CSRC, f)).read()
            yield f, re.sub(r"//[^\n]*", "", text)


def test_aligned_cluster_barriers_follow_a_warp_barrier():
    found = 0
    for f, text in _sources():
        for m in re.finditer(r'asm volatile\(\s*"barrier\.cluster\.[a-z.]*\.aligned', text):
            found += 1
            assert text[:m.start()].rstrip().endswith("__syncwarp();"), (f, text[:m.start()].count("\n") + 1)
    assert found


def test_remote_shared_memory_is_written_between_cluster_barriers():
    kernels = 0
    for f, text in _sources():
        for body in re.split(r"__global__", text)[1:]:
            if "st.shared::cluster" not in body:
                continue
            kernels += 1
            first, loop = body.index("st.shared::cluster"), body.index("for (int64_t t = 1;")
            assert "cluster_sync();" in body[:loop], f
            assert loop < first and body.rindex("cluster_sync();") > body.rindex("st.shared::cluster"), f
    assert kernels

"""A CTA may store to another's shared memory only once that one has started: in every kernel that does, a
cluster barrier comes before the first address of a peer is used (read from the sources; on the device
the order shows only when a CTA of a cluster starts late)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_18694_gb300", "csrc")


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//.*", "", open(path).read())
        for m in re.finditer(r"__global__", text):
            start = text.index("{", text.index("(const", m.end()) if "(const" in text[m.end():] else m.end())
            end = text.index("\n}\n", start)
            body = text[start:end]
            if "cluster" in body:
                yield pytest.param(body, id=os.path.basename(path) + ":" + re.findall(r"(k_\w+)\(", text[:start])[-1])


@pytest.mark.parametrize("body", list(kernels()))
def test_cluster_barrier_before_the_first_remote_store(body):
    # (remote(): addresses only; the first pass, which stores there, comes after the set-up's barrier)
    use = re.search(r"map_shared_rank\(|passes<", body)
    sync = re.search(r"(cl|this_cluster\(\))\.sync\(\)", body)
    assert use and sync and sync.start() < use.start()

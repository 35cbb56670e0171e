"""What one thread block of a cluster hands to another is ordered by the PTX memory model as written: an
arrival on another block's barrier, and a wait for one, name the cluster as their scope.  (The default is
the block, which orders nothing between two of them, whatever a run shows.)"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_18085_b200", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//.*", "", f.read())


def test_arrivals_on_another_blocks_barrier_name_the_cluster():
    found = re.findall(r"mbarrier\.arrive[\w.:]*shared::cluster[\w.:]*", source("sm100_ptx.cuh"))
    assert len(found) >= 2
    for op in found:
        assert re.match(r"mbarrier\.arrive\.(release|relaxed)\.cluster\.", op), op


def test_waits_of_the_pair_kernel_name_the_cluster():
    """Its barriers count both blocks' arrivals and copies.  (The quiet ones wait for copies and products to
    be over, and read nothing.)"""
    calls = re.findall(r"\bmbar_(?:try_)?wait\w*", source("attention_pair.cu"))
    assert calls and set(calls) <= {"mbar_wait_pair", "mbar_wait_quiet"}
    body = source("sm100_ptx.cuh").split("bool mbar_wait_pair(")[1].split("\n}\n")[0]
    assert "try_wait.parity.relaxed.cluster" in body and "fence.acquire.sync_restrict::shared::cluster.cluster" in body


def test_a_hand_over_of_shared_memory_releases_it():
    body = source("sm100_ptx.cuh").split("void mbar_arrive_remote_own(")[1].split("\n}\n")[0]
    assert body.index("fence.release.sync_restrict::shared::cta.cluster") < body.index("mbar_arrive_remote_relaxed")

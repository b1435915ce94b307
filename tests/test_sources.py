"""Properties of the CUDA sources that hold whatever machine runs them."""
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_load_is_multicast_to_a_cluster():
    """The benchmark starts one replica per GPU, and multicast loads are for programs of one GPU alone."""
    src = os.path.join(ROOT, "paper_2306_08792_gb300", "csrc")
    for f in sorted(os.listdir(src)):
        with open(os.path.join(src, f)) as fh:
            assert ".multicast" not in fh.read(), f


def test_a_warp_leaves_the_accumulator_wait_together():
    """The epilogue's warps vote on the wait for a tile: what follows it needs every lane."""
    with open(os.path.join(ROOT, "paper_2306_08792_gb300", "csrc", "umma.cu")) as fh:
        waits = [ln for ln in fh if "mbar_wait(&bars.tfull" in ln]
    assert waits and all("__all_sync(GCR_FULL, mbar_wait(" in ln for ln in waits)

"""CPU checks of the order of waits and memory accesses in the many-iteration kernel's source (k_iter_local):
what must hold there shows in no result on the hardware at hand, so it is read off the code."""
import os

import bench

SRC = os.path.join(bench.ROOT, "paper_2604_00250_gb300", "csrc", "prism_local.cuh")


def kernel():
    src = bench.strip_c_comments(open(SRC).read())
    return src[src.index("k_iter_local(const IterArgs a)"):]


def test_partials_are_read_after_a_warp_barrier():
    """One lane acquires the volume's count; the others read the tiles' partials after a warp barrier (a
    vote would order no memory accesses)."""
    k = kernel()
    wait = k.index("ld_acquire(")
    read = k.index("local_dsig_sum(", wait)
    assert "__syncwarp();" in k[wait:read]


def test_timed_out_copy_is_waited_for_and_none_follows():
    """After a copy's wait has run out the CTA lets the copy land, issues no further one and stores no state."""
    k = " ".join(kernel().split())
    assert "if (tid == 0 && !failed) { const uint32_t bytes" in k                    # no further copy
    out = k[k.index("if (!failed && !mbar_wait(&s_bar, phase)) {"):]
    assert "mbar_wait(&s_bar, phase);" in out[out.index("{"):out.index("}")]          # lets it land
    assert "e < Q * TV && !failed; e += kFusedThreads" in k                           # no state stored

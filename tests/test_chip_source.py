"""What the on-chip time loop's source has to say about waits between CTAs: such a
mistake need not show in results, and is not provoked on a GPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2304_05592_gb300", "csrc")


@pytest.fixture(scope="module")
def chip():
    text = open(os.path.join(CSRC, "step2d_chip.cu")).read()
    return re.sub(r"//[^\n]*", "", text)  # (no string holds a //)


def test_halo_waits_acquire_at_cluster_scope(chip):
    # the halo rows come from other CTAs' st.async, released at cluster scope
    assert "st.async" in chip
    waits = re.findall(r"\b(mbar_\w*(?:wait|try)\w*)\s*\(\s*&halo", chip)
    assert len(waits) >= 2 and set(waits) == {"mbar_wait_cluster"}, waits
    forms = re.findall(r"mbarrier\.(?:try_wait|test_wait)[\w.:]*", chip)
    assert forms and all(".acquire.cluster" in f for f in forms), forms


def test_a_wait_that_gave_up_waits_again_before_the_cta_leaves(chip):
    # a row that lands in the shared memory of a CTA that has left is a fault: after the barrier behind
    # which every CTA has sent its rows, a CTA with a wait given up stays for those under way, and it does
    # not arrive a second time on a barrier whose phase is open
    tail = chip[chip.index("for (int i = 0; i < a.nsteps; ++i)"):]
    tail = tail[: tail.index("k_chip_tap_gradient")]
    left = tail[tail.rindex("cluster_wait();"):]
    assert re.search(r"!alive\)(?:(?!alive).)*mbar_wait_cluster\s*\(\s*&halo", left, re.S)
    assert re.search(r"tid == 0 && alive\)\s*mbar_expect_tx", tail)

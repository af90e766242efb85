"""What the prefill GEMM waits for before a CTA of a pair may leave, read from
the kernel's source: its shared memory is written from outside (copies, and
arrivals from the peer), and such a write after the CTA has left would go to
whatever runs there next."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2607_14618_gb300", "csrc", "polyq_gemm.cu")


def _roles():
    """Source of each role's branch of gemm_main, by the heading above it."""
    text = open(SRC).read()
    body = text[text.index("gemm_main(const __grid_constant__"):text.index("all roles of both CTAs done")]
    parts = re.split(r"// -{8,} (.*?) -{8,}\n", body)
    return dict(zip((h.split(":")[0] for h in parts[1::2]), parts[2::2]))


def test_both_ctas_wait_for_the_last_commit():
    """The MMA issuer's commits arrive in both CTAs; the one on bar_done is the
    last, and both CTAs wait for it."""
    roles = _roles()
    issuer, relay = roles["MMA issuer (leader CTA)"], roles["X relay (second CTA)"]
    assert re.findall(r"tc_commit2\(smem_u32\(&(\w+)", issuer)[-1] == "bar_done"
    for branch in (issuer, relay):
        assert re.findall(r"mbar_wait\w*\(smem_u32\(&(\w+)", branch)[-1:] == ["bar_done"]


def test_copies_in_flight_are_waited_for():
    """The roles that start copies wait for those in flight, and a role that
    gives up keeps both CTAs while those of others may still be under way."""
    roles = _roles()
    for role, bar in (("X producer", "bar_xfull"), ("code producers", "bar_cfull")):
        end = roles[role].split("in flight")[1]
        assert re.search(r"mbar_wait\(smem_u32\(&%s" % bar, end)
    fail = re.search(r"auto fail = .*?\n  };", open(SRC).read(), re.S).group(0)
    assert fail.index("s_abort = 1") < fail.index("clock64() - t0 < kAbortStayCycles")

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


def test_copies_are_waited_for_by_the_role_that_asked():
    """Each role that starts copies waits for those in flight also after a role
    has given up, in both CTAs."""
    roles = _roles()
    x = roles["X producer"].split("while (!s_abort")[1]
    assert re.search(r"if \(rank != 0 \|\| s_abort\)\s+for .*\s+mbar_wait_sleep\(smem_u32\(&bar_xfull", x)
    codes = roles["code producers"]
    assert "bar_cfull" in codes[codes.index("wait (bounded) for the copies still in flight"):]
    fp16 = roles["dequantisation"]
    fp16 = fp16[fp16.index("tma_load_2d"):]
    assert re.search(r"kWaitAborted && r == 0\) mbar_wait\(smem_u32\(&bar_w16", fp16)

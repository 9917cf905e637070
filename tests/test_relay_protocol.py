"""The hand-overs between the CTAs of a cluster, checked as a protocol on the CPU from the kernels' sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_13935_b200", "csrc")


def source(name="lr_relay_kernel.cu"):
    return open(os.path.join(CSRC, name)).read()


def constant(name):
    return int(re.search(r"constexpr int (?:.*, )?%s = (\d+)" % name, source()).group(1))


def gram_races(warps, buffers, blocks=9):
    """(reader, writer, block) where a warp may write its part of a block over parts another one still adds up.

    Per block kb a warp writes part [kb % buffers], arrives at the barrier of kb's parity and, if its half adds up blocks of that
    parity, waits there and then reads the parts of all warps."""
    half = warps // 2
    sums = [[w for w in range(warps) if (w < half) == (kb % 2 == 0)] for kb in range(blocks)]
    steps = [[(kind, kb) for kb in range(blocks) for kind in ("write", "arrive") + (("read",) if w in sums[kb] else ())]
             for w in range(warps)]
    before = {}    # (warp, step): the steps it must follow
    for w in range(warps):
        for a, b in zip(steps[w], steps[w][1:]):
            before.setdefault((w, b), []).append((w, a))
    for kb in range(blocks):
        for w in sums[kb]:
            before.setdefault((w, ("read", kb)), []).extend((v, ("arrive", kb)) for v in range(warps))

    def follows(node, seen):
        for p in before.get(node, ()):
            if p not in seen:
                seen.add(p)
                follows(p, seen)
        return seen

    races = []
    for w in range(warps):
        for kb in range(buffers, blocks):
            past = follows((w, ("write", kb)), set())
            races += [(r, w, kb) for r in sums[kb - buffers] if (r, ("read", kb - buffers)) not in past and r != w]
        for kb in range(2, blocks):   # a barrier is not entered again before the last use of it is complete
            past = follows((w, ("arrive", kb)), set())
            assert all((v, ("arrive", kb - 2)) in past for v in range(warps) if v != w)
    return races


def test_gram_parts_are_read_before_they_are_written_over():
    warps = constant("kNg")
    assert gram_races(warps, 2)                              # two buffers: nothing holds a warp of the half that adds up
    assert not gram_races(warps, constant("kGramParts"))
    assert "part[kGramParts][kNg][kCoup]" in source()


def test_what_peers_sent_is_waited_for_at_cluster_scope():
    # st.async and remote arrivals come from other CTAs of the cluster: whoever waits for them acquires, and whoever frees a
    # peer's slot releases, at that scope (a CTA-scope wait orders nothing against another CTA's accesses)
    text = source()
    sent = set(re.findall(r"peer_addr\(smem_addr\(&sm\.(\w+)\[", text)) | set(re.findall(r"bar = smem_addr\(&sm\.(\w+)\[", text))
    barriers = set(re.findall(r"mbar_init\(&sm\.(\w+)\[", text)) & sent
    assert barriers == {"bz", "bg", "gfree", "delta"}
    waits = [(how, bar) for how, bar in re.findall(r"\b(\w+)\(&sm\.(\w+)\[[^;]*?\) & 1\)", text) if how.startswith("wait")]
    assert {bar for how, bar in waits} >= barriers | {"full", "done"}
    assert all((how == "wait_peer") == (bar in barriers) for how, bar in waits), waits
    assert "mbarrier.arrive.relaxed" not in text


@pytest.mark.parametrize("name", ["lr_relay_kernel.cu", "lr_chain_kernel.cu", "mlp_mma_kernel.cu", "mlp_wide_kernel.cu", "cnn_mma_kernel.cu"])
def test_who_has_given_up_arms_and_sends_nothing(name):
    # A barrier that counts bytes must not be armed again while it is short of some, nor be sent bytes without end that nobody
    # armed it for: inside a round's loops both happen only while no wait of the thread has given up.
    lines = source(name).split("\n")
    start = next(i for i, l in enumerate(lines) if "bool ok = true;" in l)
    first = {"lr_relay_kernel.cu": 2, "lr_chain_kernel.cu": 2}.get(name, 0)    # (armed for the first time, before the loop)
    guard = re.compile(r"if \(!?ok\b|&& ok\b")
    seen = []
    for i in range(start + 1, len(lines)):
        if not re.search(r"\b(mbar_expect_tx|send1|send_peer|send_pair|send_quad)\(", lines[i]):
            continue
        depth, at, held = len(lines[i]) - len(lines[i].lstrip()), i, bool(guard.search(lines[i]))
        while not held and depth > 4 and at > start:     # the lines that enclose it, innermost first, and a skip beside it
            at -= 1
            here = len(lines[at]) - len(lines[at].lstrip())
            if lines[at].strip() and not lines[at].startswith("#") and here <= depth:
                held = bool(guard.search(lines[at])) and (here < depth or "continue" in lines[at])
                depth = here
        seen.append((i + 1, held))
    assert len(seen) >= 4
    assert [held for _, held in seen].count(False) <= first, seen

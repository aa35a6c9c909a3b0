"""How a product's CTAs end (tc_kernel.cuh), read from the source: a late signal cannot be provoked safely on a GPU."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def kernel():
    with open(os.path.join(ROOT, "paper_2404_19163_gb300", "csrc", "tc_kernel.cuh")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    start = text.index("{", text.index(") k_tc_gemm("))
    depth = 0
    for i in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[start + 1:i]


def depth_at(body, i):
    return body[:i].count("{") - body[:i].count("}")


def test_every_commit_is_waited_for_in_both_ctas():
    body = kernel()
    end = body.rindex("cluster_sync()")
    commit = body.index("tc_commit<CG>(smem_u32(done_bar))")
    waits = [m.start() for m in re.finditer(r"mbar_wait(_warp)?\(done_bar", body)]
    # the last commit reaches both CTAs: the wait for it is outside the leader's branch, before the pair's barrier
    assert len(waits) == 1 and commit < waits[0] < end and depth_at(body, waits[0]) == 0
    assert "rank" not in body[body.rindex("__syncthreads()"):waits[0]]
    # so do the releases of the stages: the streaming warp of each CTA waits for all of them after its last load
    drain = body.index("for (int s = 0; s < C::STAGES && ok; ++s)")
    assert body.rindex("tma_load_2d_pair") < drain < body.index("else if (warp == 1)")
    assert depth_at(body, drain) == 1 and "empty0 + 8 * st" in body[drain:body.index("else if (warp == 1)")]

"""A CTA of the tensor-core convolution may give up (a bounded wait runs out).  It then has copies and matrix instructions under
way, which must have ended before its shared memory and TMEM are given back.  Running out is not provoked on a GPU here: the
order of the source is checked.  The role that issues each kind of work ends with the wait for it."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_03644_gb300", "csrc")


def test_every_issuing_role_ends_with_the_wait_for_its_work():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "hlbm_surrogate.cu")).read())
    kernel = src[src.index("conv_tc_kernel(const"):]
    copy = kernel[kernel.index("if (warp == TC_COPY_WARP)"):kernel.index("if (warp == TC_MMA_WARP)")]
    mma = kernel[kernel.index("if (warp == TC_MMA_WARP)"):kernel.index("if (warp == TC_READY_WARP)")]
    epilogue = kernel[kernel.index("if (warp == TC_READY_WARP)"):kernel.index("tcgen05.dealloc")]
    for role, issue, wait in ((copy, r"tell\(q\);", r"mbar_wait\(bar\(G::BAR_FULL"), (mma, r"umma_commit\(", r"mbar_wait\(bar\(G::BAR_ACC"),
                              (epilogue, r"cp\.async\.bulk\.commit_group;", r"cp\.async\.bulk\.wait_group 0;")):
        last = [m.end() for m in re.finditer(issue, role)][-1]
        assert re.search(wait, role[last:]), issue

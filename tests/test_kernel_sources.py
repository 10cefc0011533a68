"""Rules that the kernels' sources keep and that no run on a GPU shows: what breaks one goes wrong by timing only, or by a
hang after a wait has run out."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_26692_b200", "csrc")


def source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(SRC, name)).read())


def test_overlapping_kernels_read_coherently():
    """A kernel that starts while its predecessor still writes (grid_dep_wait) may not declare its inputs read-only for its
    whole duration: no const __restrict__ parameters, and .nc loads only in the backward stages whose inputs come from
    kernels that were complete before they began."""
    seen = 0
    for name in sorted(os.listdir(SRC)):
        text = source(name)
        assert "ld.global.nc" not in text or name in ("kda_bwd.cuh", "kda_bwd_intra.cu", "kda_bwd_out.cu"), name
        for kernel in re.split(r"(?=__global__)", text)[1:]:
            if "grid_dep_wait" not in kernel:
                continue
            head = kernel[:kernel.index("{")]
            seen += 1
            assert not re.search(r"const[^,]*__restrict__", head), (name, head)
    assert seen >= 15


def test_backward_chain_waits_do_not_part_a_warp():
    """The lanes of a warp may find out apart that a wait has run out, so no warp-wide role branches on a lane's own answer: the
    ones that do would leave the others in the next warp-wide instruction.  They leave on a vote; only the loader, one lane,
    leaves on its own."""
    text = source("kda_bwd_chain.cu")
    loader = text[text.index("if (lane == 0) {\n                auto get"):text.index("} else if (w == kCompute / 32) {")]
    rest = re.sub(r"!__all_sync\(0xffffffffu, wait\(\w+, i\)\)\) break;", "", text.replace(loader, ""))
    assert "if (!wait(" in loader and "break" not in rest and not re.search(r"if \([^{;]*!\s*wait", rest)
    assert not re.search(r"for \([^;{]*;[^;{]*\b(ok|abort_word)\b", rest)


def test_prefill_chain_roles_leave_together():
    """The abort flag may change between two looks at it.  The roles of kda_fused_tc.cu's chain that are whole warps leave on
    a vote, those that share a barrier on the barrier's own answer; only single lanes go by the flag as they see it."""
    text = source("kda_fused_tc.cu")
    chain = text[text.index("__device__ void chain_run("):text.index("__device__ void chain_init(")]
    compute, loader, giver, mma, out = re.split(r"reg_inc<kChainRegs>|if \(warp == 9\)|if \(kRing && warp == 10\)|if \(warp == 8\)|if \(warp >= 12 && op\)",
                                                chain)[1:]
    for single in (loader, giver):
        assert re.search(r"for \([^{;]*;[^;{]*!\*abort_flag", single) and single.lstrip(" {\n").startswith("if (lane == 0)")
    for together in (compute, mma, out):
        assert not re.search(r"for \([^{;]*;[^;{]*\*abort_flag", together)
        assert not re.search(r"if \(\*abort_flag\)\s*\{?\s*(break|return)", together)
    assert out.count("stop = ptx::named_bar_or(6, 128, seen != 0);") == 2 and len(re.findall(r"for \([^{;]*;[^;{]*!stop", out)) == 2


def test_matrix_products_end_before_their_memory_does():
    """After a wait has run out products may be under way that nobody waited for.  The warp that issued them commits once more
    and waits for that, with the limit of every wait, before its CTA gives its TMEM and shared memory back."""
    for name in ("kda_bwd_intra.cu", "kda_bwd_chain.cu", "kda_bwd_out.cu", "kda_fused_tc.cu"):
        text = source(name)
        at = [m.end() for m in re.finditer(r"umma_commit\(done\);", text)]
        assert len(at) == 1 and re.match(r"\s*(if \(!)?ptx::mbar_wait\(done, 0, a\.wait_limit_ns\)", text[at[0]:]), name
        assert re.search(r"tmem_dealloc", text[at[0]:]), name


def test_misaligned_shared_memory_is_not_called_a_timeout():
    """A kernel that finds its dynamic shared memory not aligned says so by a code of its own."""
    seen = 0
    for name in sorted(os.listdir(SRC)):
        text = source(name)
        for m in re.finditer(r"& 1023u\) != 0\) \{([^}]*)\}", text):
            seen += 1
            assert "KDA_ERR_CUDA" in m.group(1) and "TIMEOUT" not in m.group(1) and "timeout" not in m.group(1), name
    assert seen == 4

"""Rules of the device code that a run on a GPU does not show, checked on the sources: breaking one is a hang that
takes a rare order of events."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2604_15750_b200 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_15750_b200", "csrc")


def _closing(src, at, pair):
    """index of the bracket that closes the one at `at`"""
    depth = 0
    for i in range(at, len(src)):
        depth += (src[i] == pair[0]) - (src[i] == pair[1])
        if depth == 0:
            return i


def _kernel(name, kernel):
    """the body of a __global__ function, without comments"""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    at = re.search(r"__global__[^;{]*?\b" + kernel + r"\(", src).end() - 1
    head = src.index("{", _closing(src, at, "()"))
    return src[head:_closing(src, head, "{}") + 1]


@pytest.mark.parametrize("name,kernel", [("tc_gemm.cuh", "k_gemm_tc"), ("tc_lmhead.cuh", "k_lmhead_tc"),
                                         ("tc_attn.cuh", "k_attn_tc"), ("tc_attn_few.cuh", "k_attn_few")])
def test_the_next_kernel_is_let_in_behind_the_tmem_allocation(name, kernel):
    """A block of the next kernel that gets an SM before the one it waits for has its TMEM columns could take them
    and hold them while it waits.  Only blocks that leave without an allocation may trigger before it."""
    body = _kernel(name, kernel)
    alloc = body.index("tmem_alloc(")
    triggers = [m.start() for m in re.finditer(r"pdl_trigger\(\)", body)]
    assert any(t > alloc for t in triggers)
    for t in triggers:
        if t < alloc:
            end = body.index("return;", t)
            assert end < alloc and body[t:end].count("{") <= body[t:end].count("}") + 1
        else:
            assert "__syncthreads()" in body[alloc:t]


@pytest.mark.parametrize("name,first,last", [
    ("tc_chain.cuh", "const bool el = ptx::elect_one();", "umma_commit_pair(c.acc_full)"),
    ("tc_attn_few.cuh", "const bool pv = warp == 2;", "umma_commit(pv ? &c.p_empty"),
    ("tc_gemm.cuh", "// ---------------- TMA producer", "// ---------------- MMA issuer"),
    ("tc_gemm.cuh", "// ---------------- MMA issuer", "// ---------------- epilogue"),
    ("tc_attn.cuh", "// ---------------- issuer of S = Q K^T", "// ---------------- issuer of O (+)= P V"),
    ("tc_attn.cuh", "// ---------------- issuer of O (+)= P V", "// ---------------- softmax warps"),
])
def test_a_warp_that_issues_together_gives_up_together(name, first, last):
    """A bounded wait is decided lane by lane.  Where the whole warp runs the issuing loop, whose votes take all
    lanes, every wait is voted on: lanes that gave up alone would leave the others in the next vote for good."""
    src = open(os.path.join(CSRC, name)).read()
    part = src[src.index(first):src.index(last)]
    waits = list(re.finditer(r"ptx::mbar_wait", part))
    assert waits
    for m in waits:
        statement = part[max(part.rfind(c, 0, m.start()) for c in ";{}"):part.index(";", m.start())]
        later = part[m.start():]
        assert "__all_sync(" in statement or re.search(r"ok = __all_sync\(0xffffffffu, ok\);\s*if \(!ok\) break;", later)


@pytest.mark.parametrize("name,first,last,meet", [
    ("tc_chain.cuh", "epilogue: all warps", "tc_fence_after", True), ("tc_gemm.cuh", "epilogue: warps 2..5", "tc_fence_after", False),
])
def test_warps_that_meet_in_an_epilogue_give_up_together(name, first, last, meet):
    """The epilogues read TMEM warp-wide: the wait in front of them is voted on in the warp.  Where the rotation meets on
    named barriers of four warps (the chain's; the other one's is an exchange inside a warp) these four agree too."""
    src = open(os.path.join(CSRC, name)).read()
    part = src[src.index(first):]
    part = part[:part.index(last)]
    waits = re.findall(r"[^;]*ptx::mbar_wait\([^;]*;", part)
    assert waits and all("__all_sync(" in w for w in waits)
    assert bool(re.search(r"EPI_QKV\) ok = ptx::all_agree\([^;]*, 128, ok\);", part)) == meet
    assert ("bar.sync" in src or "all_agree" in src) == meet


@pytest.mark.parametrize("name,kernel", [("tc_gemm.cuh", "k_gemm_tc"), ("tc_attn_few.cuh", "k_attn_few"), ("tc_chain.cuh", "k_dense_chain"),
                                         ("tc_attn.cuh", "k_attn_tc"), ("tc_lmhead.cuh", "k_lmhead_tc")])
def test_what_is_on_its_way_is_waited_for_when_every_role_has_decided(name, kernel):
    """A CTA that has given up waits for its TMA writes before it leaves, with a limit of its own.  A producer may be
    through with its loop when another role gives up: the flag is looked at behind a barrier that all roles come to after
    their last wait, and before the CTA (or its partner) may leave."""
    body = _kernel(name, kernel)
    drain = body.index("late_flag)")
    flag = body.rindex("abort_flag != 0)", 0, drain)
    role_waits = body.rindex("abort_flag)", 0, flag)
    assert "__syncthreads();" in body[role_waits:flag]
    leave = body.find("cluster_sync()", drain)
    assert leave == -1 or "__syncthreads();" not in body[drain:leave]


@pytest.mark.parametrize("name,kernel", [("tc_gemm.cuh", "k_gemm_tc"), ("tc_chain.cuh", "k_dense_chain"), ("tc_lmhead.cuh", "k_lmhead_tc"),
                                         ("tc_attn.cuh", "k_attn_tc"), ("tc_attn_few.cuh", "k_attn_few")])
def test_the_tcgen05_instructions_of_a_kernel_have_one_cta_group(name, kernel):
    """Pair MMAs and commits go with an allocation, a relinquished permit and a release of cta_group::2, and those
    of a CTA alone with cta_group::1; the pair's release comes behind a cluster barrier."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    body = _kernel(name, kernel)
    pair = bool(re.search(r"umma_\w*pair", src))
    both = pair and bool(re.search(r"umma_(bf16_lo|bf16|commit|commit_a)\(", src))    # a template with both
    want = "PAIR" if both else "true" if pair else ""
    calls = re.findall(r"ptx::tmem_(?:alloc|relinquish|dealloc)\([^;]*?(PAIR|true|)\);", body)
    assert calls == [want] * 3
    if pair:
        assert "cluster_sync()" in body[:body.index("tmem_dealloc")].rsplit("__syncthreads();", 1)[1]


@pytest.mark.parametrize("name,rule", [("tc_gemm.cuh", r"if \(left >= stages\) \{\s*if \(PAIR\) "),
                                       ("tc_chain.cuh", r"if \(EPI != CEPI_QKV \|\| kb < refills\) ")])
def test_no_ring_slot_is_handed_back_for_nothing(name, rule):
    """The commit behind a k-block arrives on the slot's barrier in both CTAs of a pair.  Nothing waits for an arrival on a
    slot that is not filled again (the accumulator's is another one): it could come when the partner has left.  A launch of
    the chain that ends with a projection waits for these arrivals at its end."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    commits = re.findall(r"umma_commit_pair_a\(", src)
    assert len(commits) == len(re.findall(rule + r"ptx::umma_commit_pair_a\(", src)) == 1
    if name == "tc_chain.cuh":
        body = _kernel(name, "k_dense_chain")
        wait = body.index("mbar_wait(&bar_empty[c.lane]")
        assert body.rindex("if (!has_qkv && c.warp == 0)", 0, wait) < wait < body.index("late_flag)") < body.rindex("cluster_sync()")


@pytest.mark.skipif(shutil.which(build._nvcc()) is None, reason="no nvcc")
def test_the_fused_cuda_core_step_keeps_its_sums_in_registers(tmp_path):
    """512 threads of 128 registers and 32 sums a thread: nothing is left over, and a spill is 1.5% of a step."""
    r = subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-Xptxas", "-v", "-c", os.path.join(CSRC, "simt_step.cu"), "-o",
                        str(tmp_path / "x.o")], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    assert r.returncode == 0, r.stdout
    of_step = re.findall(r"Function properties for \S*k_simt_step\S*\n.*?(\d+) bytes spill stores, (\d+) bytes spill loads", r.stdout)
    assert of_step == [("0", "0")] * 2, r.stdout

"""The rules that overlapped launches rest on, checked in the kernels' source (a violation is a race or a mutual wait, which
no test may provoke on a GPU): every kernel waits for its predecessor, reads its inputs through ordinary loads only, and
lets its successor in only when its own tensor memory is allocated."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_00023_b200", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def text(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def kernels(src):
    """(name, parameters, body) of every kernel."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(([^{;]*)\)\s*\{", src):
        depth, end = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(src[end], 0)
            end += 1
        yield m.group(1), m.group(2), src[m.end():end]


def global_reads(params, code):
    """Names through which a piece of a kernel reaches global memory: pointer parameters indexed or dereferenced, members of
    parameter structs likewise, tensor maps that are fetched through."""
    pointers = re.findall(r"\*\s*(?:__restrict__\s+)?(\w+)", params)
    out = {n for n in pointers if re.search(r"(?<![\w.])%s\s*(\[|->|\+)|\*\s*%s\b" % (n, n), code)}
    out |= set(re.findall(r"\bp\.(\w+)\s*(?:\[|->)", code))
    return out | set(re.findall(r"\b(?:tma_load\w*|f3_fetch|dsw_load|atomic\w+)\b", code))


@pytest.mark.parametrize("name", SOURCES)
def test_overlapped_launches(name):
    src = text(name)
    assert "__ldg" not in src and "ld.global.nc" not in src
    assert not re.search(r"const\s+\w+\s*\*\s*(const\s+)?__restrict__", src)      # functions called by kernels too
    for kernel, params, body in kernels(src):
        assert not re.search(r"const\s+\w+\s*\*\s*(const\s+)?__restrict__", params), kernel
        if re.search(kernel + r"\s*<<<", src):
            continue                                         # launched without overlap
        if "tcgen05.alloc" not in body:
            first = body.index("grid_sync();")
            assert not re.search(r"\bp\.\w+\[|stats->|\w+\[", re.sub(r"__shared__[^;]*;", "", body[:first])), kernel
            continue
        early = global_reads(params, body[:body.index("grid_wait();")])
        assert not early, kernel
        order = [body.index(s) for s in ("tcgen05.alloc", "grid_wait();", "__syncthreads();", "grid_release();")]
        assert order == sorted(order) and "grid_sync" not in body, kernel
        if "tcgen05.dealloc.cta_group::2" in body:           # the pair leaves together
            assert "cluster_sync_all();" in body[body.index("tcgen05.dealloc.cta_group::2"):], kernel


def test_the_kernels_are_found():
    names = [k for f in SOURCES for k, _, _ in kernels(text(f))]
    assert len(names) >= 30 and "tc_grouped_gemm_swap_kernel" in names and "combine_kernel" in names


TILED = [f for f in SOURCES if re.search(r"extern __shared__ [^;]*uint8_t", text(f))]


@pytest.mark.parametrize("name", TILED)
def test_tiles_start_at_a_multiple_of_1024(name):
    """The dynamic shared memory of a kernel with swizzled tiles is declared so aligned and its address taken as it is, or the
    address is rounded up and the launch asks for the 1024 bytes that this may skip."""
    src = text(name)
    rounds = []
    for kernel, _, body in kernels(src):
        block = re.search(r"extern __shared__ ([^;]*)uint8_t", body)
        if block:
            rounds.append("1023u" in body)
            assert rounds[-1] != ("__align__(1024)" in block.group(1)), kernel
    sizes = re.findall(r"constexpr size_t (?:smem|\w+_SMEM) = ([^;]*);", src)
    assert len(sizes) == len(rounds) and sum("+ 1024" in s for s in sizes) == sum(rounds)


def test_the_tiled_kernels_are_found():
    assert TILED == ["gemm_tcgen05.cu", "gemm_tf32x3.cu", "score_tcgen05.cu"]


def test_pooling_reads_stay_inside_the_row():
    """The pooling kernel loads without predicates: a piece beyond the row is replaced by one of the row's own.  Every lane and
    batch of rows of 1 to 600 pieces of 16 bytes (a row of 64 bf16 values has 8, fewer than the lanes of a warp)."""
    body = next(b for k, _, b in kernels(text("affinity.cu")) if k == "grap_pool_kernel")
    batch = int(re.search(r"constexpr int BATCH = (\d+);", body).group(1))
    cond, there, else_ = re.search(r"q\[g\]\.load\(x \+ \(size_t\)\((.+?) \? (.+?) : (.+?)\) \* PE\);", body).groups()
    named = dict(re.findall(r"(\w+) = (min\(lane, npieces - 1\))", body))
    pick = compile(f"({there}) if ({cond}) else ({named.get(else_, else_)})", "piece", "eval")
    for npieces in range(1, 601):
        for p0 in range(0, npieces, 32 * batch):
            for g in range(batch):
                for lane in range(32):
                    at = eval(pick, {"min": min}, {"p": p0 + 32 * g + lane, "lane": lane, "npieces": npieces})
                    assert 0 <= at < npieces, (npieces, p0, g, lane)


@pytest.mark.parametrize("stages", [3, 4])
def test_the_split_of_fp32_operands_waits_for_the_block_it_takes(stages):
    """Two groups of converter warps take alternate K blocks of a ring of 3 or 4 stages, and a wait tells the uses of a stage
    apart by their parity: it passes when the number of completed uses is of the other one.  Over every state that a group
    may find when it comes to use `u` of a stage (`split`: uses split so far, `landed`: uses whose copy has landed, both only
    grow), its waits, as the source has them, may pass in turn only when use u has landed."""
    src = text("gemm_tf32x3.cu")
    branch = src[src.index("if (turn == group) {"):src.index("f3_split_box<A_MN>(st")]
    waits = re.findall(r"(if \(F3_STAGES % 2 != 0\)\s+ok = |ok = (?:ok && )?)__all_sync\(0xffffffffu, "
                       r"mbar_wait\((\w+)_bar \+ 8 \* stage, phase( \^ 1u)?", branch)
    assert len(waits) == branch.count("mbar_wait(")
    waits = [(bar, 1 if flip else 0) for cond, bar, flip in waits if stages % 2 or not cond.startswith("if")]
    for u in range(2, 8):
        # the group's own last use of the stage, u - 2 or u - 1, is split, this one is not; a stage holds one block
        states = [(split, landed) for split in range(u - 1 if stages % 2 else u, u + 1) for landed in (split, split + 1)]
        at = set(states)
        for bar, flip in waits:
            done = {"conv": 0, "full": 1}[bar]
            later = {b for a in at for b in states if b[0] >= a[0] and b[1] >= a[1]}
            at = {x for x in later if x[done] & 1 != (u ^ flip) & 1}
        assert at and all(landed > u for _, landed in at), (u, at)

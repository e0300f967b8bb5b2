"""Contracts of the device code that no run can show without faulting the GPU, checked in
the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_12196_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _body(text, start):
    """The braces' contents that follow position ``start``."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def test_split_gemm_outlasts_its_copies_and_mmas_after_an_abort():
    """An aborted wait returns at once. The waits that keep shared and tensor memory alive
    (the copies in either ring, the MMAs' last commit, in both CTAs of the pair) go on,
    bounded, without a look at the abort flag."""
    src = _source("gemm_split.cu")
    drain = _body(src, src.index("void mbar_drain("))
    assert "abort" not in drain and "kDrainPolls" in drain
    kernel = _body(src, src.index("void __cluster_dims__(2, 1, 1)"))
    waits = re.findall(r"(!?)mbar_wait\(bar\((full \+ sl\.i|kDone)\)[^;]*;", kernel)
    assert [w for _, w in waits] == ["full + sl.i", "kDone", "kDone"]
    for m in re.finditer(r"mbar_wait\(bar\((full \+ sl\.i|kDone)\)", kernel):
        assert re.search(r"if \([^;]*$", kernel[:m.start()]), "the wait's result decides"
        assert f"mbar_drain(bar({m.group(1)})" in kernel[m.start():m.start() + 200]
    # every slot that was loaded is waited for, also when only one ring's copy was issued
    assert re.search(r"finish\(lead, nlead, RG::kLeadStages", kernel)
    assert re.search(r"finish\(rest, nrest, RG::kRestStages", kernel)
    # the last commit arrives in both CTAs, which both wait for it
    assert "umma_commit(bar(kDone))" in kernel


# what ytn_plan uploads and no kernel writes
TABLES = {"CopyJob", "CopyItem", "SectorDev", "GemmTile", "TraceChunk", "TraceOut", "TraceContrib", "CScatterJob",
          "CScatterChunk", "SplitOperand", "SplitItem", "SliceItem", "SliceSeg", "SplitSector", "SplitTile",
          "SplitCheckChunk", "VdotChunk", "VdotPiece"}


def test_only_the_plans_tables_are_read_as_constant():
    """Kernels of a call start before their predecessor has finished and wait for it first:
    what it wrote is not read-only for their lifetime."""
    kernels = 0
    for name in sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))):
        src = _source(name)
        for m in re.finditer(r"const (\w+) \*__restrict__", src):
            assert m.group(1) in TABLES, f"{name}: {m.group(0)}"
        for m in re.finditer(r"__ldg\((\w+(?:\.\w+)?)", src):
            assert m.group(1) in ("base", "out.base"), f"{name}: {src[m.start():m.start() + 60]}"
        if "launch_chained(" not in src:
            continue
        for m in re.finditer(r"__global__", src):
            body = _body(src, src.index(")", src.index("_kernel(", m.start())))
            first = body.index("after_previous_kernel();")
            assert not re.search(r"\w\[[^\]]*\](?!;)|->|=[^=]", re.sub(r"__shared__[^;]*;|constexpr[^;]*;|using[^;]*;|extern[^;]*;", "", body[:first])), name
            kernels += 1
    assert kernels >= 17

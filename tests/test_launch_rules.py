"""Rules that every kernel launched with programmatic stream serialization has to follow, checked in the sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_08301_b200", "csrc")
WAIT = "griddepcontrol.wait"


def _strip_comments(text):
    return re.sub(r"//[^\n]*", "", text)


def _kernels():
    """(name, body) of every __global__ function."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = _strip_comments(open(path).read())
        for m in re.finditer(r"__global__", text):
            start = text.index("{", text.index(")", text.index("(", re.compile(r"\w+_kernel\s*\(").search(text, m.end()).start())))
            name = re.compile(r"(\w+_kernel)\s*\(").search(text, m.end()).group(1)
            depth, end = 0, start
            for end in range(start, len(text)):
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                if depth == 0:
                    break
            out.append((name, text[start:end + 1]))
    return out


CHAINED = [(n, b) for n, b in _kernels() if WAIT in b]


def _header_check():
    text = open(os.path.join(CSRC, "mwu_gemm_dev.cuh")).read()
    return text[text.index("#define MWU_CHECK_HEADER"):].split("while (0)")[0]


def test_the_kernels_were_found():
    assert len(CHAINED) >= 15


@pytest.mark.parametrize("name,body", CHAINED, ids=[n for n, _ in CHAINED])
def test_no_chained_kernel_ends_before_it_has_waited(name, body):
    before = body[:body.index(WAIT)]
    assert not re.search(r"\breturn\s*;", before)
    if "MWU_CHECK_HEADER" in before:
        check = _header_check()
        assert WAIT in check and check.index(WAIT) < check.index("return;")


@pytest.mark.parametrize("name,body", [k for k in CHAINED if "tmem_alloc" in k[1] and "launch_dependents" in k[1]],
                         ids=lambda x: x if x.endswith("_kernel") else "")
def test_dependents_start_only_once_tensor_memory_is_held(name, body):
    # A dependent may take all 512 columns of an SM before its own wait, which lasts until this kernel has ended.  One
    # thread's trigger counts for its CTA, so it is the warp that holds the allocation which triggers.
    assert re.search(r"\{\s*tmem_alloc\([^;]*;\s*asm volatile\(\"griddepcontrol.launch_dependents;\"[^;]*\);\s*\}", body)
    assert body.count("griddepcontrol.launch_dependents") == 1


def test_the_question_for_clusters_names_their_shared_memory():
    # without it several CTAs seem to fit an SM, and a part of a device that cannot place the cluster would answer yes
    text = _strip_comments(open(os.path.join(CSRC, "mwu_common.cuh")).read())
    body = text[text.index("inline bool cluster_runs"):]
    body = body[:body.index("\n}\n")]
    ask = body.index("cudaOccupancyMaxActiveClusters")
    assert "dynamicSmemBytes" in body[:ask] and "cudaFuncAttributeMaxDynamicSharedMemorySize" in body[:ask]


def test_boxes_alternate_over_all_stores_of_a_warp():
    # bulk_wait_read_1 lets the latest store go on reading its box, so the next box must be the other one, whichever tile the
    # store belongs to: its place is kept across tiles and flipped at every store, not derived from the store's number in a tile
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = _strip_comments(open(path).read())
        for m in re.finditer(r"bulk_wait_read_1\(\)", text):
            start = text.rindex("unsigned char *box", 0, m.start())
            assert re.match(r"unsigned char \*box = stg \+ box_at;\s*box_at \^= box_flip;", text[start:]), path
            assert len(re.findall(r"box_at\s*[\^+*|&-]?=(?!=)", text)) == 2, path      # set once, flipped in one place


def test_the_short_reduction_kernel_brings_only_stages_that_are_multiplied_to_l2():
    text = _strip_comments(open(os.path.join(CSRC, "mwu_gemm5.cu")).read())
    lines = [l for l in text.splitlines() if "tma_prefetch_2d(" in l]
    assert lines and all("(wanted >> ks) & 1u" in l for l in lines)

"""Rules that hold for every kernel of the library, read from its source: a violation may show as wrong results
only now and then on a GPU, so they are checked where they stand."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_21244_gb300", "csrc")


def _source(path):
    """Text without comments."""
    with open(path) as f:
        text = f.read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


SOURCES = {os.path.basename(p): _source(p) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}


def _dependent_kernels():
    """(file, kernel) of every kernel that a launch_dep call names, directly or through a variable."""
    found = set()
    for name, text in SOURCES.items():
        for call in re.finditer(r"\blaunch_dep\(\s*(\w+)", text):
            arg = call.group(1)
            kernels = {arg} if arg.startswith("k_") else set()
            if not kernels:   # a variable: the kernels in its last assignment before the call
                values = re.findall(r"\b%s\s*=([^;]*);" % arg, text[:call.start()])
                kernels = set(re.findall(r"\bk_\w+", values[-1])) if values else set()
            assert kernels, f"{name}: launch_dep({arg}): kernel not found"
            found |= {(name, k) for k in kernels}
    return sorted(found)


@pytest.mark.parametrize("where,kernel", _dependent_kernels())
def test_kernel_placed_early_waits_for_the_one_before(where, kernel):
    """A kernel launched by launch_dep may be placed while the kernel before it runs: it has to wait for that
    one's end, and so for all before it, ahead of everything else."""
    m = re.search(r"__global__[^;{}]*\b%s\s*\([^{;]*\)\s*\{\s*([^;]*;)" % kernel, SOURCES[where])
    assert m, "definition not found"
    assert re.fullmatch(r"dep_wait(_alone)?\(\);", m.group(1)), m.group(1)


def _body(text, start):
    """The braced block that opens first after `start`, and what follows it up to the next __syncwarp()."""
    at = text.index("{", start)
    depth, end = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
        if depth == 0:
            break
    return text[at:end], text[end:text.index("__syncwarp();", end)]


def test_chi_mlp_copy_lane_leaves_no_copy_in_flight():
    """However its loop ends (all chunks issued, or another role's failure), the lane that issues the weight
    copies waits for the last one into each buffer before the CTA can release its shared memory."""
    text = SOURCES["chi_mlp.cu"]
    body, rest = _body(text, text.index("for (; m < total; ++m)"))
    assert "bulk_g2s" in body
    assert re.match(r"\s*for \(int q = m > kNbuf \? m - kNbuf : 0; q < m; \+\+q\)\s*tc::mbar_wait\(full \+ q % kNbuf", rest), rest


def test_chi_mlp_issuing_lane_leaves_no_mma_in_flight():
    """The lane that issues the MMAs waits for all of them before the CTA can release its tensor memory, also
    when it has issued its last one and the epilogue of that pass fails."""
    text = SOURCES["chi_mlp.cu"]
    body, rest = _body(text, text.index("for (int it = 0; it < my_its && ok; ++it)"))
    assert "mma_bf16_ta" in body
    assert re.match(r"\s*tc::commit\(drain\);\s*tc::mbar_wait\(drain, 0,", rest), rest


def test_training_leaves_no_mma_in_flight():
    """When a wait of the training kernel runs out, the MMAs that are committed but not waited for by every thread
    end before the tensor memory is released: the issuing thread waits for them after the loop over tiles."""
    text = SOURCES["train.cu"]
    start = text.index("for (int64_t tile = blockIdx.x; tile < ntiles && alive;")
    _, rest = _body(text + "__syncwarp();", text.index("{", start) - 1)
    rest = rest[:rest.index("tmem_dealloc")]
    assert re.search(r"if \(!alive && t == kIssuer\) \{\s*tc::commit\(drain\);\s*tc::mbar_wait\(drain, 0,[^;]*;\s*\}"
                     r".*__syncthreads\(\);", rest, flags=re.S), rest


def test_autotuner_times_the_gather_of_the_step():
    """The step's sort and the autotuner's trials share the gather, which for up to kGatherAll particles forms the
    cell starts; the form that reads them is the static sort's alone."""
    text = SOURCES["cells.cu"]
    calls = [m.start() for m in re.finditer(r"k_gather<false>", text)]
    assert len(calls) == 1 and calls[0] > text.index("int dsmc_sort_cells_static(")

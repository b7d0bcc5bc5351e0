"""Rules of the device code that a GPU run cannot show without a hang or a race, checked on the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_08816_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


# waits of one elected lane (the copies' warps): every lane of the other roles takes part
ONE_LANE = {"kernels_digit.cu": {"31"}, "kernels_tc.cu": {"11", "13b"}}


@pytest.mark.parametrize("name", sorted(ONE_LANE))
def test_bounded_waits_of_whole_warps_are_decided_by_the_warp(name):
    """A wait with the user's limit may run out for some lanes only; lanes that leave alone would miss the votes,
    shuffles and aligned tensor-memory loads that the others go on to."""
    src = _source(name)
    seen = 0
    for m in re.finditer(r"mbar_wait\(", src):
        stmt = src[max(src.rfind(c, 0, m.start()) for c in ";{}") + 1:]
        stmt = stmt[:re.search(r"[;{]", stmt).start()]
        code = re.search(r"t\.err, (\d+), t\.spins", stmt)
        if not code:
            continue
        seen += 1
        tag = code.group(1) + ("b" if "bfree" in stmt else "")
        after = src[m.start():]
        after = after[after.index(";") + 1:]
        voted = "__all_sync(0xffffffffu" in stmt or re.match(r"\s*if \(!__all_sync\(0xffffffffu, ok\)\)", after)
        assert voted or tag in ONE_LANE[name], f"{name}: wait {tag} is decided lane by lane"
    assert seen >= 7


@pytest.mark.parametrize("name", sorted(ONE_LANE))
def test_matrix_products_drain_before_tensor_memory_is_freed(name):
    """The MMA warp waits for its products whether or not it gave up itself: another role's wait can run out after the
    last product has been issued, and the block would free the accumulators and exit under it."""
    src = _source(name)
    drain = src.index("mma_commit(smem_u32(&bar_drain))")
    assert "tcgen05.dealloc" in src[drain:]
    before = src[:drain].rstrip()
    assert before.endswith("if (elect_one())")
    before = before[:-len("if (elect_one())")].rstrip()
    assert before.endswith("}") and not re.search(r"if \(!ok\) \{$", before)


def test_kernel_attributes_are_set_for_every_grid():
    """A kernel's shared-memory limit belongs to a device: a flag of the process would leave a second one without it."""
    create = _source("fv_api.cpp")
    create = create[create.index("int fv_grid_create("):create.index("int fv_grid_destroy(")]
    setups = set()
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cpp")):
            continue
        src = _source(name)
        assert not re.search(r"static bool attr", src), name
        for m in re.finditer(r"cudaFuncSetAttribute\(", src):
            function = re.findall(r"^(?:static )?int (\w+)\(", src[:m.start()], re.M)[-1]
            assert "_setup" in function, f"{name}: {function}"
            setups.add(re.sub(r"_setup_\w+", "_setup", function))
    assert len(setups) >= 7
    for f in setups - {"digit_setup"}:
        assert re.search(rf"\b{f}\b", create), f
    assert "upload_digits" in create and "digit_setup()" in _source("fv_api.cpp")


def test_overlapping_kernels_read_their_predecessors_results_by_ordinary_loads():
    """A kernel that overlaps its predecessor is resident while that one still writes; the read-only load path (__ldg, or a
    kernel's const __restrict__ pointer) is defined for data that nobody writes meanwhile.  Grid data, written once at
    creation, may take it: metrics (g.*), matrices (M, t.M) and eigenvalues (lx, ly, lz); so may a kernel that is only
    launched without the overlap."""
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        src = _source(name)
        if "pdl_wait()" not in src:
            continue
        seen += 1
        for m in re.finditer(r"__ldg\(\s*([\w.]+)", src):
            assert re.match(r"(g\.|t\.M)", m.group(1)), f"{name}: __ldg({m.group(1)}"
        for m in re.finditer(r"const \w+\* __restrict__ (\w+)", src):
            kernel = re.findall(r"\b(k_\w+)\(", src[:m.start()])[-1]
            alone = f"launch_spread({kernel}<" in src and not re.search(rf"launch(_cluster)?\([^;]*\b{kernel}\b", src)
            assert alone or m.group(1) in {"M", "lx", "ly", "lz"}, f"{name}: const __restrict__ {m.group(1)}"
    assert seen >= 8


def test_grid_creation_waits_for_its_own_fills():
    """The field maxima, the error word, metrics and operands are filled on the default stream; a handle's non-blocking stream
    does not wait for that one, and a solve would add its largest magnitude to what the memory held."""
    create = _source("fv_api.cpp")
    create = create[create.index("int fv_grid_create("):create.index("int fv_grid_destroy(")]
    sync = create.index("cudaStreamSynchronize(nullptr)")
    assert all(m.start() < sync for m in re.finditer(r"cudaMemset\(|upload_\w+[<(]|tc_setup\(", create))
    assert sync < create.index("*out = g")

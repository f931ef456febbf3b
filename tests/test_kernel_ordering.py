"""Memory order inside the kernels that no result can show reliably: each check reads the source for the
barrier, fence or load that orders what one thread or kernel writes and another one reads."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_21207_gb300", "csrc")


def _code(name):
    """A source file without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def _function(code, start):
    """From `start` to the closing brace of the function whose head it begins."""
    at = code.index(start)
    depth = 0
    for i in range(code.index("{", at), len(code)):
        depth += {"{": 1, "}": -1}.get(code[i], 0)
        if depth == 0:
            return code[at:i + 1]
    raise AssertionError("unbalanced braces after " + start)


def test_the_walk_follows_a_barrier_after_the_direction_stores():
    """Every lane of a fill warp stores directions; lanes 0 and 1 read other lanes' and write over them."""
    fill = _function(_code("sc_search.cuh"), "void fill_super_tile(")
    stores = [m.end() for m in re.finditer(r"\b(?:down_row|up_row)\(e|\bup_row\(g|\bdown_row\(e", fill)]
    walk = fill.index("fb[rel]")
    assert stores and max(stores) < walk
    assert "__syncwarp();" in fill[max(stores):walk]


def test_tensor_maps_in_global_memory_are_acquired():
    """The batched kernels copy through maps the host wrote into global memory: the thread that issues the
    copies (the producer warp's first) acquires each image's map before its first search."""
    for name, item, search in (("sc_batch.cuh", "void batch_carve_item(", "batch_seam_pass<"),
                               ("sc_batch_cl.cuh", "void clb_carve_item(", "clb_seam_pass<")):
        body = _function(_code(name), item)
        fence = re.search(r"if \((?:T\w+ && )?threadIdx\.x == NW \* 32\) fence_tensormap_acquire\(tmap\);", body)
        assert fence and fence.start() < body.index(search), name
    fence = _function(_code("sc_ptx.cuh"), "void fence_tensormap_acquire(")
    assert "fence.proxy.tensormap::generic.acquire.sys" in fence


def test_loads_ahead_of_the_wait_go_past_l1():
    """The refresh kernels read energies and lists of the kernel before last ahead of their
    griddepcontrol.wait, which alone would make an SM's L1 current: every such load is an L2 one."""
    kernels, rows = _code("sc_kernels.cu"), _code("sc_rowops.cuh")
    for name in ("k_refresh(", "k_refresh_wide(", "k_refresh_fwd("):
        body = _function(kernels, name)
        ahead = body[body.index("{"):body.index("pdl_wait_prerequisites();")]
        assert not re.search(r"\b(?:seam|img|lists_in|lists_out|E|er)\s*\[", ahead), name
        assert "lazy_row(" not in ahead and "refresh_pixel(" not in ahead, name
        for cast in re.findall(r"[\w:(]*\(?\s*reinterpret_cast<const \w+ \*>\([^;]*;", ahead):
            assert cast.startswith("__ldcg("), (name, cast)
    lane = _function(rows, "RefreshLane refresh_lane(")
    assert "lazy_row_l2(" in lane and "lazy_row(" not in lane
    assert _function(rows, "LazyRow lazy_row_l2(").count("__ldcg(") == 2


def test_check_clears_the_search_words_in_stream_order():
    """sc_check clears words that a running search counts in; the caller's stream may not be ordered with
    the default stream, so the clearing goes on the caller's."""
    body = _function(_code("sc_api.cu"), "int sc_check(")
    clears = re.findall(r"cudaMemset(?:Async)?\(ws\.flags[^;]*;", body)
    assert len(clears) == 1 and clears[0].startswith("cudaMemsetAsync(") and ", st)" in clears[0]
    enqueued = [m.start() for m in re.finditer(r"Async\(", body)]
    waits = [m.start() for m in re.finditer(r"cudaStreamSynchronize\(st\)", body)]
    # the first wait refuses a stream that is being captured, the last one completes the copy and the clearing
    assert waits[0] < min(enqueued) and body.index(clears[0]) < waits[-1]


def test_a_search_checks_the_cost_of_the_one_before():
    """A two-ended search leaves 0 in its cost word when its super-tiles' costs add up to its own; the next
    one looks at what it finds there and takes it away, so that two differences cannot cancel."""
    kernel = _function(_code("sc_dp.cu"), "k_dp_two(DpArgs p")
    assert kernel.index("__ldcg(p.sync + 1)") < kernel.index("two_join<") < kernel.index("atomicAdd(")
    found = kernel[kernel.index("if (left != 0u)"):]
    assert "atomicSub(reinterpret_cast<uint32_t *>(p.sync + 1), left);" in found
    assert "atomicOr(p.err, ERR_COST_MISMATCH);" in found
    assert re.search(r"if \(h\[3\] != 0\) e \|= ERR_COST_MISMATCH", _function(_code("sc_api.cu"), "int sc_check("))

"""Rules of the kernels' sources that no run can show to be broken."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2311_17089_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def kernel(text, name):
    """The parameters and body of a __global__ function."""
    at = re.search(r"\b%s\s*\(" % name, text).start()
    depth, i = 0, text.index("{", at)
    for j in range(i, len(text)):
        depth += (text[j] == "{") - (text[j] == "}")
        if depth == 0:
            return text[at:i], text[i:j]
    raise AssertionError(name)


# per dependent launch (common.cuh, pdl_wait): what the kernel before it may
# still be writing when it starts, as the reading code names it
WRITTEN_BEFORE = {
    "bin.cu": ["a.filter", "a.keys_in", "a.vals_in", "a.hist", "stats", "order_stats"],
    "bin_tiles.cu": ["a.order", "a.b.", "item", "idx", "a.item", "a.idx", "a.meta", "a.matrix",
                     "a.offsets", "a.part", "a.tile_sums", "row"],
    "raster.cu": ["a.seg_off", "a.seg_len", "a.use_list", "a.ranges", "ranges"],
    "raster_list.cu": ["a.seg_off", "a.seg_len", "a.use_list", "a.rowmask", "ml"],
    "backward.cu": ["g2", "p.g2"],
}


def test_dependent_launches_read_no_fresh_data_as_constant():
    for name, fields in WRITTEN_BEFORE.items():
        text = source(name)
        for load in re.findall(r"__ldg\(\s*&?\s*([^;]*)", text):
            for f in fields:
                assert not re.match(r"%s(?![A-Za-z0-9_])" % re.escape(f), load) and not (
                    f.endswith(".") and load.startswith(f)), (name, load)
    # the first kernels of ms_bin and ms_raster: no parameter the compiler
    # may take for constant
    for name, k in (("bin.cu", "bin_start_kernel"), ("raster.cu", "segment_offsets_kernel")):
        params, body = kernel(source(name), k)
        assert not re.search(r"const[^,]*__restrict__", params), k
        assert "__ldg" not in body
    # and ml, row_mask_kernel's masks
    assert not re.search(r"const uint32_t \*__restrict__ ml", source("raster_list.cu"))


def test_dependent_kernels_wait_first():
    """Every kernel launched with launch_after waits before anything else."""
    texts = {f: source(f) for f in os.listdir(CSRC) if f.endswith(".cu")}
    seen = 0
    for text in texts.values():
        names = set(re.findall(r"launch_after\(\s*(?:vec \? )?(\w+)", text))
        for k in names - {"rank"} | ({"tile_rank_kernel"} if "rank" in names else set()):
            _, body = kernel(text, k)
            first = body.lstrip("{ \n").split(";")
            decl = [s.strip() for s in first[:12]]
            at = next(i for i, s in enumerate(decl) if s.startswith("pdl_wait"))
            for s in decl[:at]:
                assert re.match(r"(using |extern __shared__|__shared__|constexpr |BwdSmem &)", s), (k, s)
            seen += 1
    assert seen >= 12


def test_assembly_that_touches_memory_says_so():
    """Loads, stores, copies and barriers in inline PTX are volatile and name
    "memory", so that the compiler moves no access across them."""
    seen = 0
    for f in os.listdir(CSRC):
        for m in re.finditer(r"\basm\b(\s+volatile)?\s*\((.*?)\)\s*;", source(f), re.S):
            text = m.group(2)
            if re.search(r"\b(ld|st|cp|red|atom|mbarrier|fence|bar|griddepcontrol)\.", text):
                seen += 1
                assert m.group(1) and '"memory"' in text, (f, text)
    assert seen > 20

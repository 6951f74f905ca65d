"""Chained kernels (programmatic stream serialization) live while the kernel
before them still writes.  What that kernel writes must not be read through the
read-only path: not with __ldg, nor through a kernel parameter that is const
and __restrict__.  Checked on the sources, since no run can show the absence of
a reordering."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_04449_gb300", "csrc")

# const __restrict__ parameters of chained kernels, each with the kernels that
# may stand directly before it in a chain: none of those writes the buffer
READ_ONLY = {
    "k_voxelize_small": {"q", "tris"},               # k_vox_clear: seeds, big_count
    "k_voxelize_big": {"q", "tris"},                 # k_voxelize_small: seeds, big_list, big_count
    "k_sah_prims": {"verts", "tris"},                # k_sah_root: tasks, chunks, bins, blist, counters
    "k_sah_partition": {"chunks", "pbox"},           # k_sah_split: left_off, bins, hist, tasks, next chunks, links
    "k_leaves_up": {"verts", "tris", "leaf_parent"},  # a memset, k_top_detach (not chained)
    "k_depth": {"leaf_parent"},                      # k_collapse_kids: nodes, from, lev
    "k_batch_boxes": {"nbox", "lbox"},               # k_collapse_level: wide, from, lev
    "k_obj_init": {"motion"},                        # a memset
    "k_obj_boxes": {"verts", "vobj", "motion"},      # k_obj_init: boxes, list, count
    "k_translate": {"vobj", "trans"},                # k_obj_boxes: boxes
    "k_transform": {"vobj", "xf"},                   # k_obj_boxes: boxes
}
# device functions that read with __ldg / ldg256: only BVH nodes and leaf
# triangles (written before the mask kernel, the tracer's direct predecessor),
# or under a template switch that chained kernels turn off
LDG_FUNCTIONS = {"jfa_voxel", "jfa_zblock_column", "sample", "build_front", "node_step", "leaf_step"}


def _sources():
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            text = open(os.path.join(CSRC, f)).read()
            out[f] = re.sub(r"//[^\n]*", "", text)
    return out


def _close(text, i, pair):
    """Position after the bracket that closes the one before text[i]."""
    depth = 1
    while depth:
        depth += {pair[0]: 1, pair[1]: -1}.get(text[i], 0)
        i += 1
    return i


def _functions(text):
    """(name, parameter text, body, is a kernel) of every device function."""
    while True:
        m = re.search(r"__launch_bounds__\(", text)
        if not m:
            break
        text = text[:m.start()] + text[_close(text, m.end(), "()"):]
    for m in re.finditer(r"__(?:global|device)__[^;{}()=]*?(\w+)\s*\(", text):
        j = _close(text, m.end(), "()")
        brace = re.match(r"\s*(?:const\s*)?\{", text[j:])
        if brace:
            k = j + brace.end()
            yield m.group(1), text[m.end():j - 1], text[k:_close(text, k, "{}")], "__global__" in m.group(0)


def _chained():
    out = {}
    for text in _sources().values():
        for name, params, body, kernel in _functions(text):
            if kernel and re.search(r"\bchain_(begin|wait)\(\)", body):
                out[name] = (params, body)
    return out


def test_every_launched_chain_kernel_waits():
    chained = _chained()
    named = set()
    for text in _sources().values():
        named |= set(re.findall(r"launch_chain\(c, (k_\w+)", text))
        # kernels chosen into a variable first
        for var in re.findall(r"launch_chain\(c, ((?!k_)\w+)", text):
            for rhs in re.findall(rf"\b{var} = ([^;]*);", text):
                named |= set(re.findall(r"\b(k_\w+)", rhs))
    assert len(named) >= 20
    assert named <= set(chained), named - set(chained)


def test_chained_kernels_read_their_predecessors_output_with_plain_loads():
    chained = _chained()
    found = {}
    for name, (params, body) in chained.items():
        ro = {re.search(r"(\w+)\s*$", p).group(1) for p in params.split(",")
              if re.search(r"\bconst\b", p) and "__restrict__" in p}
        if ro:
            found[name] = ro
        assert "__ldg" not in body and "ldg256" not in body, name
    assert found == READ_ONLY


def test_read_only_path_is_off_in_chained_kernels():
    for f, text in _sources().items():
        for name, _, body, _ in _functions(text):
            if name != "ldg256" and re.search(r"\b(__ldg|ldg256)\(", body):
                assert name in LDG_FUNCTIONS, (f, name)
    chained = _chained()
    columns = re.findall(r"jfa_zblock_column<([^>]*)>", chained["k_jfa_zblock"][1])
    assert columns and all(c.split(",")[3].strip() == "false" for c in columns)
    assert "jfa_voxel" not in "".join(b for _, b in chained.values())
    samples = re.findall(r"\bsample<([^>]*)>", chained["k_shadow"][1])
    assert samples and all(s.split(",")[1].strip() == "false" for s in samples)

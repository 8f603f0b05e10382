"""Rules that the kernels' sources keep (no GPU needed)."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_24593_b200", "csrc")


def _kernels(text):
    """(name, parameter list, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        params = text[m.end():i - 1]
        j = text.index("{", i)
        depth, k = 1, j + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        yield m.group(1), params, text[j:k]


def test_kernels_that_start_before_their_predecessor_ends_take_no_read_only_pointers():
    """A kernel that waits for its predecessor inside (grid_dependency_wait) must not promise the compiler
    that what it reads is constant: such loads may be moved in front of the wait."""
    seen = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for name, params, body in _kernels(text):
            if "grid_dependency_wait" not in body:
                continue
            seen.append(name)
            bad = [p.strip() for p in params.split(",") if "__restrict__" in p and re.match(r"\s*const\b", p)]
            assert not bad, f"{os.path.basename(path)}: {name}: {bad}"
    assert {"scan_select_tc_kernel", "refine_tc_kernel", "decode_scan_kernel", "decode_select_kernel",
            "decode_window_kernel", "entries_topk_kernel", "merge_parts_kernel"} <= set(seen)


def test_candidates_of_the_kernel_before_are_not_read_as_constants():
    """Candidate sets are written by the scan, the select or the merge and read by the re-score that starts early."""
    for name in ("refine_tc.cu", "segselect.cuh", "decode_tc.cu"):
        text = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"__ldg\([^)]*cand|__ldg\(cp\b", text), name

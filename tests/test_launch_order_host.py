"""Kernels that start while the one before them still runs (launch_next).

Until such a kernel has passed after_previous(), earlier kernels write the buffers
it works on.  A ``__restrict__`` pointer promises the compiler that nobody else does:
it may then read through the non-coherent path, or move an access over the wait.  Only
tables that are complete before any launch (the plan's and the mask's) may carry it, and
what uploads them waits for its copies: cudaMemcpy from pageable memory and cudaMemset
may return before the device has them, and non-blocking streams do not wait for the
legacy stream."""
import glob
import os
import re

import pytest

from paper_2603_29785_gb300 import build

# parameters that name tables uploaded before the first launch that reads them
TABLES = {"rows", "row_list", "tw", "tws", "t", "twM", "twN", "tw4", "ftw", "wtab", "invP", "tabA", "tabAi", "tabG", "kc"}


def _closing(text, i, pair):
    """Index just past the bracket that closes the one at text[i]."""
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] == pair[0]) - (text[j] == pair[1])
        if depth == 0:
            return j + 1
    raise ValueError("unbalanced")


def _functions():
    """(file, name, parameters, body, is a kernel) of every device function defined in csrc."""
    out = []
    for path in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__(global|device)__", text):
            stop = re.compile(r"[;{]").search(text, m.end())
            name = None
            for c in re.finditer(r"(\w+)\s*\(", text[m.end():]):
                if c.group(1) not in ("__launch_bounds__", "__align__"):
                    name = c
                    break
            if name is None:
                continue
            p0 = m.end() + name.end() - 1
            if stop and stop.start() < p0:
                continue                                # a variable or a member without parameters
            p1 = _closing(text, p0, "()")
            b0 = re.compile(r"[;{]").search(text, p1)
            if b0 is None or b0.group() == ";":
                continue                                # a declaration
            body = text[b0.start():_closing(text, b0.start(), "{}")]
            out.append((os.path.basename(path), name.group(1), text[p0 + 1:p1 - 1], body, m.group(1) == "global"))
    return out


FUNCTIONS = _functions()
EARLY = [f for f in FUNCTIONS if f[4] and "after_previous()" in f[3]]


def test_the_early_kernels_are_found():
    names = {f[1] for f in EARLY}
    assert {"k_untangle_forward", "k_untangle_inverse", "k_col_forward", "k_long_columns", "k_long_rows", "k_rows_forward_any",
            "k_rows_inverse_any", "k_rows_forward", "k_rows_inverse_tc", "k_plane_metrics", "k_zero", "k_scale_rows",
            "k_best_planes", "k_stream_gather_x", "k_stream_phases"} <= names
    # what launch_next is given waits before it works
    launched = set()
    for path in glob.glob(os.path.join(build.CSRC, "*.cu*")):
        for m in re.finditer(r"launch_next\(\s*(k_\w+)", open(path).read()):
            launched.add(m.group(1))
    assert launched and launched <= names


@pytest.mark.parametrize("kernel", sorted({f[1] for f in EARLY}))
def test_only_tables_are_restrict(kernel):
    by_name = {}
    for f in FUNCTIONS:
        by_name.setdefault(f[1], []).append(f)
    seen, todo = set(), [kernel]
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        for file, _, params, body, _ in by_name[name]:
            promised = set(re.findall(r"__restrict__\s+(\w+)", params))
            assert promised <= TABLES, (kernel, file, name, sorted(promised - TABLES))
            # and what it calls, by name
            todo += [w for w in set(re.findall(r"\b(\w+)\s*(?:<[^;(){}]*>)?\(", body)) if w in by_name and w not in seen]


@pytest.mark.parametrize("file,function,wait", [("qtam_api.cu", "upload_tables", "return finish_uploads();"),
                                                ("qtam_api.cu", "build_mask", "s = finish_uploads();"),
                                                ("qtam_stream.cu", "qtam_stream_create",
                                                 "e = cudaStreamSynchronize(cudaStreamLegacy);")])
def test_uploads_are_complete_before_the_handle_is_out(file, function, wait):
    text = open(os.path.join(build.CSRC, file)).read()
    m = re.search(r"\bqtam_status\s+" + function + r"\(", text)
    body = text[m.start():_closing(text, text.index("{", m.start()), "{}")]
    copies = [c.start() for c in re.finditer(r"\bupload\w*(?:<\w+>)?\(|cudaMem(?:cpy|set)\(", body)]
    waits = [w.start() for w in re.finditer(re.escape(wait), body)]
    assert waits and max(copies[1:] or copies) < max(waits)
    if "finish" in wait:
        f = re.search(r"qtam_status finish_uploads\(\) \{(.*?)\n\}", text, re.S)
        assert "cudaStreamSynchronize(cudaStreamLegacy)" in f.group(1)

"""What the benchmark reports beside its times names what was timed."""
import os
import re
import shutil

from paper_2603_29785_gb300 import qtam

BENCH = open(os.path.join(qtam._build.ROOT, "bench.py")).read()


def test_reported_variants_are_those_that_ran():
    """The plan's info holds the first registered variant, taken when the plan was made."""
    assert not re.search(r"info\[.row_variant.\]", BENCH)
    names = re.findall(r'"row_variant": ([^,}\n]+)', BENCH)
    assert len(names) >= 3
    for n in names:
        assert re.fullmatch(r"(chosen|tuned)\[.name.\]", n.strip()), n


def test_traffic_is_tied_to_what_the_row_kernels_are_built_from(tmp_path):
    """Counters are reported only for the sources and the variant they were taken of."""
    import bench
    files = bench.row_kernel_sources()
    assert {"kernels_any.cu", "rows_any.cuh", "pass_fft.cuh", "row_shapes.inc", "kernels_rows.cu", "rows_common.cuh",
            "fft_core.cuh", "qtam_internal.h"} <= set(files)
    digests = {bench.row_kernel_digest()}
    for i, f in enumerate(files):
        d = tmp_path / str(i)
        shutil.copytree(bench.CSRC, d)
        with open(d / f, "a") as out:
            out.write("\n// changed\n")
        digests.add(bench.row_kernel_digest(str(d)))
    assert len(digests) == 1 + len(files)
    assert bench.measured_traffic("k_rows_forward", -2) is None

"""What the benchmark reports beside its times names what was timed."""
import os
import re

from paper_2603_29785_gb300 import qtam

BENCH = open(os.path.join(qtam._build.ROOT, "bench.py")).read()


def test_reported_variants_are_those_that_ran():
    """The plan's info holds the first registered variant, taken when the plan was made."""
    assert not re.search(r"info\[.row_variant.\]", BENCH)
    names = re.findall(r'"row_variant": ([^,}\n]+)', BENCH)
    assert len(names) >= 3
    for n in names:
        assert re.fullmatch(r"(chosen|tuned)\[.name.\]", n.strip()), n

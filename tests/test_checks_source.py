"""The bounds-checked build's checks, by the kernels' source: a check that fails
has to keep the access it guards from being made."""
import os
import re

from paper_2204_03756_gb300 import build


def _source():
    with open(os.path.join(build.SRC_DIR, "kernels.cuh")) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_no_check_is_ignored():
    src = _source()
    calls = re.findall(r"([^\n;{}]*)\bcheck\((?!bool)", src)
    assert len(calls) > 10
    for before in calls:
        assert re.search(r"\bif \(!?$|return $|[&|]\s*$", before), before


def test_kept_words_and_lists_are_checked():
    """Every index taken out of a mask word or a list goes through KeptIndex: the
    only other bits-to-index conversions are the searches' own."""
    src = _source()
    body = src[src.index("struct KeptIndex"):]
    body = body[body.index("};") + 2:]
    assert not re.findall(r"__ffs\(", body)
    assert len(re.findall(r"of_(?:word|list)\(", body)) >= 5

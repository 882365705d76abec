"""What the header says of pixels_per_thread = 0 and of the parts that wide tiles are
composited in, against the rules in the sources."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _read(*path):
    return open(os.path.join(ROOT, *path)).read()


def test_header_states_the_default_pixels_per_thread_and_the_parts():
    header = re.sub(r"\s+", " ", _read("include", "gftorf.h"))
    rule = _read("paper_2505_05356_gb300", "csrc", "api.cu")
    rule = rule[rule.index("int default_ppt("):rule.index("size_t chunk_rows(")]
    # the rule: wide tiles 4, double 2, else 1, 2 or 4 by the number of warps
    assert re.findall(r"return (\d)", rule)[:3] == ["4", "2", "1"] and "? 4 : 2" in rule
    assert "0: 4 for tiles 32 or more wide (which take only 4), else 2 in double and 1, 2 or 4 " \
           "by the batch's size in single precision" in header
    parts = _read("paper_2505_05356_gb300", "csrc", "render_impl.cuh")
    assert "narrow_parts(L) ? 16 : 32" in parts
    assert "parts of 32x32 pixels, one CTA each, or of 32x16 in large single-precision" in header

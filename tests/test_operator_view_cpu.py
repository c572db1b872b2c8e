"""No host function of the single handle keeps an operator view across an
allocation: an allocation that fails gives the encoded diagonal's memory back
(dmalloc), so every launch takes its view anew."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1308_1856_gb300", "csrc",
                   "tdse_api.cu")


def test_every_launch_takes_its_own_view():
    src = open(SRC).read()
    assert len(re.findall(r"\bview\(h(?:, plain)?\)", src)) >= 20
    for m in re.finditer(r"\bOperatorView (\w+) = view\(", src):
        # the one use outside a launch's argument list returns the view at once
        assert re.search(r"return " + m.group(1) + r";", src[m.end():m.end() + 200]), src[m.start():m.end()]

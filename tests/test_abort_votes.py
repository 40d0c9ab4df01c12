"""A warp of the staged kernels gives up as one (CPU: the source is read).  The lanes of a warp read
a CTA's abort flag at different times; a lane that left on its own reading would be missing from
the full-mask shuffles and votes of the others, so every reading is voted over the warp."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1412_6367_gb300", "csrc")


def test_every_reading_of_the_abort_flag_is_voted():
    text = open(os.path.join(CSRC, "integrate.cu")).read()
    readings = re.findall(r"[^\n]*\*abort_flag\s*(?:!=|==)[^\n]*", text)
    assert len(readings) >= 6  # producers and consumers of three kernels
    for line in readings:
        assert "__any_sync(0xffffffffu," in line, line.strip()
    # ... and what is not compared is written
    others = [x for x in re.findall(r"[^\n]*\*abort_flag[^\n]*", text)
              if not re.search(r"\*abort_flag\s*(?:!=|==)", x)]
    for line in others:
        assert re.search(r"\*abort_flag = (?:0|1);|volatile int \*abort_flag", line), line.strip()

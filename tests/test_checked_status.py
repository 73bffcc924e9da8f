"""Bounds checks of the checked build report somewhere: no check is given a null status word, and no
function that checks leaves it out."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_check_has_a_status_word():
    checks = 0
    for path in glob.glob(os.path.join(ROOT, "paper_2303_08163_gb300", "csrc", "*.cu*")):
        text = open(path).read()
        assert not re.search(r"\*status\s*=\s*nullptr\s*[,)]", text), path
        for m in re.finditer(r"LBM_CHECK\(", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            args = text[m.end():i - 1]
            if args.startswith("ok, status"):  # the macro itself
                continue
            checks += 1
            assert "status" in args.rsplit(",", 1)[1], (path, args)
    assert checks >= 8

"""The inner GMRES keeps the precision of its scalars: rotations by hypot and division."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_16863_gb300", "csrc")


def _function(name, header="arnoldi.cuh"):
    text = re.sub(r"//.*", "", open(os.path.join(CSRC, header)).read())
    body = text[re.search(r"\b%s\s*\([^;{]*\)\s*\{" % name, text).start():]
    return body[:re.search(r"^\}", body, flags=re.M).start()]


def test_rotations_are_formed_by_hypot_and_division():
    body = _function("ar_givens")
    assert "hypot(x, hk1)" in body and not re.search(r"\br?sqrtf?\s*\(", body)
    assert re.search(r"cc = x / den", body) and re.search(r"ss = hk1 / den", body)

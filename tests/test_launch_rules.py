"""Host rules of the launches (rix_rules.h)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_10343_gb300", "csrc")


def test_one_name_for_the_number_of_SMs():
    for f in sorted(os.listdir(CSRC)):
        for line in open(os.path.join(CSRC, f)):
            code = line.split("//")[0]
            assert f == "rix_rules.h" or not re.search(r"\b152\b", code), (f, line)

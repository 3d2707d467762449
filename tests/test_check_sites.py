"""The range checks of the checked build: a report names its place only if every site number stands in one place."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_27042_b200", "csrc")
CALL = re.compile(r"\b(CIP?|copy16)\(")


def sites():
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())
        for m in CALL.finditer(text):
            args, depth, k = [""], 1, m.end()
            while depth:
                c = text[k]
                depth += (c == "(") - (c == ")")
                if c == "," and depth == 1:
                    args.append("")
                elif depth:
                    args[-1] += c
                k += 1
            number = args[4 if m.group(1) == "copy16" else -1].strip()
            if number.isdigit():                             # a definition or a call that hands its caller's number on has none
                yield int(number), name, text.count("\n", 0, m.start()) + 1


def test_site_numbers_are_unique():
    seen = {}
    for number, *place in sites():
        assert number not in seen, (number, seen[number], place)
        seen[number] = place
    assert len(seen) > 80

"""Inline assembly of several instructions: an output written while inputs are still to
be read may not share a register with them, which only an early clobber ("=&") rules out."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_13111_gb300", "csrc")


def _statements(text):
    """(template, output constraints) of each asm statement; macros with one argument expanded."""
    for name, arg, body in re.findall(r"#define (FP_\w+)\((\w+)\) ((?:.*\\\n)*.*)", text):
        text = text.replace("#define " + name, "")
        body = body.replace("\\\n", " ")
        text = re.sub(re.escape(name) + r"\((\w+)\)", lambda m: re.sub(r"\b%s\b" % arg, m[1], body), text)
    for m in re.finditer(r"\basm\s*(?:volatile)?\s*\(", text):
        depth, i, quoted = 1, m.end(), False
        while depth:
            c = text[i]
            quoted ^= c == '"' and text[i - 1] != "\\"
            depth += 0 if quoted else (c == "(") - (c == ")")
            i += 1
        body = text[m.end():i - 1]
        head = re.match(r'\s*(?:"(?:[^"\\]|\\.)*"\s*)+', body)
        template = "".join(re.findall(r'"((?:[^"\\]|\\.)*)"', head[0]))
        rest = body[head.end():]
        outputs = "" if rest.startswith("::") else re.split(r":(?![^\"]*\"\s*\()", rest[1:], maxsplit=1)[0]
        yield template, re.findall(r'"([=+][^"]*)"', outputs)


def test_outputs_written_before_the_last_input_is_read_are_early_clobber():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for template, out in _statements(open(path).read()):
            written = set()
            for ins in re.split(r";|\\n", template):
                ops = {int(n) for n in re.findall(r"%(\d+)", ins)}
                if ops and max(ops) >= len(out):  # reads an input
                    bad = [n for n in written if out[n].startswith("=") and "&" not in out[n]]
                    assert not bad, (os.path.basename(path), template, bad)
                    seen += len(written) > 0
                written |= {n for n in ops if n < len(out)}
    assert seen > 0  # the loads of two places in one statement

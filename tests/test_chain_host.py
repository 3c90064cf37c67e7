"""Source check of the kernels that a programmatically serialised launch may
start while their predecessor still writes (csrc/lgf_internal.cuh,
chain_launch): what a pass hands to the next one is read by ordinary loads
after chain_wait, so no such array carries __restrict__ and none goes through
the read-only path.  (A load under either promise may move ahead of the wait,
which no run shows reliably.)"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1604_01814_gb300", "csrc")


def _strip(text):
    return re.sub(r"//[^\n]*", "", text)


def _functions(text):
    """name -> (parameter list, body) of the functions that have a body."""
    out = {}
    for m in re.finditer(r"\b(\w+)\(", text):
        i, depth = m.end(), 1
        while depth and i < len(text):
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        rest = text[i:].lstrip()
        if not rest.startswith("{"):
            continue
        j = text.index("{", i)
        k, depth = j + 1, 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        out.setdefault(m.group(1), (text[m.end():i - 1], text[j:k]))
    return out


def _read(name):
    return _strip(open(os.path.join(CSRC, name)).read())


def _chained(text):
    """The kernels that the chain_launch calls of this source start."""
    used = set()
    for name, (_, body) in _functions(text).items():
        for arg in re.findall(r"chain_launch\([^,]+,\s*(\w+)", body) if name != "chain_launch" else ():
            if arg.startswith("k_"):
                used.add(arg)
            else:   # a local alias: every kernel assigned to it
                for value in re.findall(rf"\b{arg} = ([^;]*);", body):
                    used |= set(re.findall(r"\bk_\w+(?=<)", value))
    return used


def test_chained_passes_take_plain_pointers():
    text = _read("lgf_poisson_kernels.cuh")
    f = _functions(text)
    assert _chained(text) == {"k_row_inverse", "k_col_forward", "k_col_inverse", "k_col_convolve"}
    for kern in sorted(_chained(text)):
        for name in (kern, kern[2:] + "_body"):
            params, body = f[name]
            handed = [p for p in params.split(",") if re.search(r"\*[^,]*\b(in|out|A|B|u)\s*$", p)]
            assert handed, name
            assert not [p for p in handed if "__restrict__" in p], name
            assert "__ldg" not in body, name
            for alias in re.findall(r"__restrict__\s*(\w+)\s*=\s*([^;]*)", body):
                assert not re.search(r"\b(in|out|A|B|u|ib|ob|bb|uu)\b", alias[1]), (name, alias)


def test_chained_integrating_factor_takes_plain_loads():
    text = _read("lgf_intfactor_win.cuh")
    f = _functions(text)
    assert _chained(text) == {"k_sep_z", "k_sep_win"}
    for kern in sorted(_chained(text)):
        body = f[kern][1]
        assert "__ldg" not in body, kern
        for alias in re.findall(r"__restrict__\s*(\w+)\s*=\s*([^;]*)", body):
            assert not re.search(r"\bJ\.(in|out)\b", alias[1]), (kern, alias)
    # the fields of a job are plain pointers
    job = re.search(r"struct SepJob \{(.*?)\}", text, re.S).group(1)
    assert re.search(r"const T \*in;", job) and re.search(r"T \*out;", job)


def test_nothing_of_a_pass_is_read_before_the_wait():
    text = _read("lgf_poisson_kernels.cuh")
    f = _functions(text)
    for name in ("row_inverse_body", "col_forward_body", "col_inverse_body", "col_convolve_body"):
        body = f[name][1]
        head = body[:body.index("load_twiddles(")]
        assert "[" not in re.sub(r"smem_raw\[\]", "", head), name
    assert "chain_wait();" in f["load_twiddles"][1]

"""Kernels launched early behind their predecessor (programmatic serialization),
read as source: they live while the predecessor still writes, so

  * what it writes is read by ordinary loads (ld_prev) behind the wait, never by
    a non-coherent load (__ldg and its wrappers) nor through a __restrict__
    pointer, which lets the compiler choose one;
  * a kernel lets its successor start only after its own wait, so that no kernel
    starts beside the last but one, whose input the one between may rewrite."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_1402_6081_gb300" / "csrc"

# kernel or helper -> its parameter that points to what the predecessor writes
READS = {
    "group_impl.cuh": {"k_gz_fwd": "xy", "rows": "spec", "k_gmac": "spec", "load_row": "base", "sources2": "base",
                       "k_gprod": "img", "k_gz_image": "xy", "k_gxy_inv": "xy"},
    "kernels_impl.cuh": {"persist_load": "fh", "k_mac_persist": "fh"},
}
WAIT = re.compile(r"wait_previous\(\)|griddepcontrol\.wait")
TRIGGER = re.compile(r"let_next_start\(\)|griddepcontrol\.launch_dependents")
NONCOHERENT = re.compile(r"\b(?:__ldg|ld|ldg_cx)\(")


def closing(text, i):
    """Index behind the bracket that closes the one at text[i]."""
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] in "({") - (text[j] in ")}")
        if depth == 0:
            return j + 1
    raise AssertionError("unbalanced")


def functions(name):
    """name -> (parameters, body) of every function of a source file."""
    text = re.sub(r"//[^\n]*", "", (CSRC / name).read_text())
    out = {}
    for m in re.finditer(r"__(?:global|device)__[^;{}()]*(?:__launch_bounds__)?", text):
        i = m.end()
        if m.group().endswith("__launch_bounds__"):
            i = closing(text, text.index("(", i))
        k = text.index("(", i - 1 if text[i - 1] == "(" else i)
        fn = re.findall(r"\w+", text[:k])[-1]
        e = closing(text, k)
        b = text.find("{", e)
        if b < 0 or text[e:b].strip() not in ("", "const"):
            continue
        out[fn] = (text[k + 1:e - 1], text[b:closing(text, b)])
    return out


def derived(body, root):
    """Names of the function that hold an address made from root."""
    names = {root}
    while True:
        pat = r"(\w+)\s*=\s*[^;]*\b(?:%s)\b\s*[+;]" % "|".join(names)
        new = {m.group(1) for m in re.finditer(pat, body)} - names
        if not new:
            return names
        names |= new


@pytest.mark.parametrize("name", sorted(READS))
def test_predecessor_data_is_read_coherently(name):
    fns = functions(name)
    waiting = {f for f, (_, body) in fns.items() if WAIT.search(body)} - {"wait_previous"}
    assert waiting <= set(READS[name]), "a kernel that waits must be listed with what it reads"
    for fn, param in READS[name].items():
        params, body = fns[fn]
        (decl,) = [p for p in params.split(",") if re.search(r"\b%s$" % param, p.strip())]
        assert "__restrict__" not in decl, (fn, decl)
        names = derived(body, param)
        for m in NONCOHERENT.finditer(body):
            arg = body[m.start():closing(body, body.index("(", m.start()))]
            assert not names & set(re.findall(r"\w+", arg)), (fn, arg)


@pytest.mark.parametrize("name", sorted(READS))
def test_successor_starts_after_the_wait(name):
    for fn, (_, body) in functions(name).items():
        wait, trigger = WAIT.search(body), TRIGGER.search(body)
        if fn != "wait_previous" and wait and trigger:
            assert wait.start() < trigger.start(), fn

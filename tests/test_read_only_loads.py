"""Read-only loads (__ldg, const __restrict__ parameters) are for what no running kernel writes.
A kernel launched before the one ahead has completed, and a phase of the persistent batched
kernel, read what the one ahead or an earlier phase wrote by ordinary loads: in the sources, the
kernels launched by launch_pdl and the functions that the persistent kernel runs take only the
plan's constants (tables, symbols, twiddles, descriptors) through such pointers."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1810_03275_gb300", "csrc")
CONSTANTS = {"jobs", "tw", "sym", "geom", "march", "sd", "prefix", "pre", "src"}     # (src: stage_tw's twiddles)


def _sources():
    out = {}
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        out[f] = re.sub(r"//[^\n]*", "", text)
    return out


def _overlapped(sources):
    names = set()
    for text in sources.values():
        for m in re.finditer(r"launch_pdl\(", text):
            names |= set(re.findall(r"\b(k_\w+)", text[m.start():text.index(";", m.end())]))
        names |= set(re.findall(r"\b(k_\w+)\s*<", " ".join(re.findall(r"auto kern = [^;]*;", text))))
    return names


def _signature(text, name):
    """The parameter lists of the definitions of `name`."""
    out = []
    for m in re.finditer(r"\b%s\s*\(" % name, text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        if text[i:].lstrip().startswith("{"):
            out.append(text[m.end():i - 1])
    return out


def test_overlapped_kernels_and_phases_take_constants_only():
    sources = _sources()
    names = _overlapped(sources)
    assert {"k_forward_orbit", "k_bp_fold", "k_gfft_cols", "k_orbit_sino", "k_dot2"} <= names
    bodies = {n for n in re.findall(r"\b(\w+_body|march\w*|fwd_march|tv_dual_at|orbit_fold4?|bp_epilogue_value)\b",
                                    " ".join(sources.values()))} - {"bp_reduce_body"}     # (of k_bp_reduce alone)
    seen = 0
    for name in sorted(names | bodies | {"k_batch_iteration", "persist_stage_block"}):
        for text in sources.values():
            for params in _signature(text, name):
                seen += 1
                for p in re.findall(r"const\s+[\w:<>]+(?:\s+[\w:<>]+)?\s*\*\s*__restrict__\s+(\w+)", params):
                    assert p in CONSTANTS, (name, p)
    assert seen > 30


def test_ldg_reads_constants_only():
    for f, text in _sources().items():
        for arg in re.findall(r"__ldg\(([^;]*)\)", text):
            assert re.match(r"\(?\s*(%s)\b" % "|".join(CONSTANTS), arg), (f, arg)

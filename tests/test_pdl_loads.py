"""Kernels of a programmatic dependent launch are resident while the kernel before them still writes, so memory that it
writes must be read by plain loads behind griddepcontrol.wait: the read-only path (__ldg, or a `const __restrict__`
parameter, which the compiler may turn into it or move up) promises that the memory does not change while the kernel
runs.  That holds for the links, the group table and what else is written before the first kernel of a chain; this
reads the sources and lets no other pointer have it."""
import glob
import os
import re

from paper_0901_3512_gb300.build import CSRC

# written once, long before: links (FP32, FP64, fixed point), the batch's group table
CONSTANT_PARAMS = {"u", "G"}
CONSTANT_LDG = re.compile(r"^\s*(u \+|F\.u \+|lp \+)")
# outputs that their kernel never reads
OUTPUTS = {"k_lz_D": {"v", "Vrow", "t"}, "k_lz_Ddag": {"f"}, "k_lz_eo": {"out", "Vrow"}, "k_lz_fix": {"out", "Vrow"},
           "k_po_sub_seg": {"part"}, "k_po_sub_fix": {"part"}, "k_po_normalise": {"Vrow"}, "k_to_internal_f32": {"out"},
           "k_proj_partial": {"part"}, "k_proj_reduce": {"C"}, "k_proj_fix": {"part"}, "k_proj_fix_reduce": {"C"}}
# the learned guess is launched in plain stream order
PLAIN = {"guess.cu"}


def _sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        yield os.path.basename(path), text


def _closing(text, at, a, b):
    depth = 0
    for k in range(at, len(text)):
        depth += (text[k] == a) - (text[k] == b)
        if depth == 0:
            return k
    raise AssertionError("unbalanced")


def _functions(text, start):
    """(name, parameters, body) of the definitions that `start` opens."""
    for m in re.finditer(start, text):
        k = m.end()
        while True:   # past __launch_bounds__(...)
            p = text.index("(", k)
            name = re.search(r"(\w+)\s*$", text[k:p])
            e = _closing(text, p, "(", ")")
            if name.group(1) != "__launch_bounds__":
                break
            k = e + 1
        rest = text[e + 1:].lstrip()
        if rest.startswith("{"):
            b = text.index("{", e)
            yield name.group(1), text[p + 1:e], text[b:_closing(text, b, "{", "}") + 1]


def _read_only(params):
    return set(re.findall(r"\bconst\s+[^,]*?__restrict__\s+(\w+)", params))


def test_early_kernels_promise_nothing_about_what_their_predecessor_writes():
    seen = 0
    for name, text in _sources():
        for kernel, params, body in _functions(text, r"__global__\s+void"):
            if "pdl_enter()" in body:
                seen += 1
                assert _read_only(params) <= CONSTANT_PARAMS, (name, kernel, _read_only(params))
                promised = set(re.findall(r"__restrict__\s+(\w+)", params))
                assert promised <= CONSTANT_PARAMS | OUTPUTS.get(kernel, set()), (name, kernel, promised)
                assert "__restrict__" not in body, (name, kernel)
    assert seen >= 20


def test_every_kernel_launched_early_waits():
    waits = {k for _, text in _sources() for k, _, body in _functions(text, r"__global__\s+void") if "pdl_enter()" in body}
    for name, text in _sources():
        for m in re.finditer(r"launch_pdl\(", text):
            call = text[m.start():_closing(text, m.end() - 1, "(", ")")]
            for k in re.findall(r"\bk_\w+", call):
                assert k in waits, (name, k)


def test_device_functions_load_fields_plainly():
    for name, text in _sources():
        if name in PLAIN:
            continue
        for m in re.finditer(r"__ldg\(", text):
            arg = text[m.end():_closing(text, m.end() - 1, "(", ")")]
            assert CONSTANT_LDG.match(arg), (name, arg)
        for fn, params, _ in _functions(text, r"__device__ (?:__forceinline__|__noinline__)(?: static)? [\w<>&]+(?= )"):
            assert _read_only(params) <= CONSTANT_PARAMS, (name, fn, _read_only(params))

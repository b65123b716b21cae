"""Source check of the kernels launched with programmatic dependence.  Their CTAs are resident before
`griddepcontrol.wait` while the launches before still write, so buffers those write must not go through the read-only
path (`__ldg`, `const T* __restrict__` kernel parameters), whose contract is data constant for the whole kernel and
which leaves the compiler free to load before the wait.  No run can show such a load: it depends on the compiler.
Host only."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2008_00446_gb300" / "csrc"

# const __restrict__ parameters that were complete before the chain began (the chain's first launch is a plain one)
FIXED = {
    ("k_noalloc_cost", "pts"), ("k_noalloc_cost", "obs_cam"), ("k_noalloc_cost", "obs_pt"),
    ("k_noalloc_cost", "obs_uv"),          # the caller's arrays
    ("k_vp_finalize", "counts"),           # written by the re-ordering
    ("k_step_tc", "S"),                    # S' is complete before k_diag_scale, which begins this chain
}


def _block(text, i, opening, closing):
    """text[i] is `opening`: the index after its match."""
    depth = 0
    for k in range(i, len(text)):
        depth += (text[k] == opening) - (text[k] == closing)
        if depth == 0:
            return k + 1
    raise AssertionError("unbalanced")


def _source(f):
    """without comments and launch bounds"""
    text = re.sub(r"//[^\n]*", "", f.read_text())
    while (i := text.find("__launch_bounds__(")) >= 0:
        text = text[:i] + text[_block(text, text.index("(", i), "(", ")"):]
    return text


def _functions():
    """name -> list of (parameters, body) of every device function and kernel."""
    out = {}
    for f in sorted(CSRC.glob("*.cu*")):
        text = _source(f)
        for h in re.finditer(r"__(?:global|device)__[^;{}()]*?\b(\w+)\s*\(", text):
            e = _block(text, h.end() - 1, "(", ")")
            b = re.match(r"\s*(?:const)?\s*\{", text[e:])
            if b:
                s = e + b.end() - 1
                out.setdefault(h.group(1), []).append((text[h.end():e - 1], text[s:_block(text, s, "{", "}")]))
    return out


def _chained():
    names = set()
    for f in sorted(CSRC.glob("*.cu")):
        text = _source(f)
        for m in re.finditer(r"\blaunch_after\(", text):
            names |= set(re.findall(r"\bk_\w+", text[m.end():_block(text, m.end() - 1, "(", ")")].split("stream")[0]))
        if "cudaLaunchAttributeProgrammaticStreamSerialization" in text:   # launches with the attribute set by hand
            for m in re.finditer(r"\bcudaLaunchAttributeProgrammaticStreamSerialization\b", text):
                names |= set(re.findall(r"\bk_(?:tri_push|step_tc)\b", text[m.end():m.end() + 1500]))
    return names


def test_chained_kernels_use_ordinary_loads():
    fn, chained = _functions(), _chained()
    assert {"k_vp_reduce", "k_pt_acc", "k_vp_finalize", "k_point_rhs", "k_point_update", "k_finalize", "k_apply",
            "k_scatter_step", "k_residual", "k_tri_push", "k_step_tc", "k_noalloc_cost", "k_noalloc_final"} <= chained
    bad = []
    for k in sorted(chained):
        assert k in fn, k
        seen, todo = set(), [k]
        while todo:   # the kernel and the device functions it reaches
            name = todo.pop()
            if name in seen:
                continue
            seen.add(name)
            for params, body in fn[name]:
                if "__ldg" in body:
                    bad.append((k, name, "__ldg"))
                if name == k:
                    bad += [(k, name, p) for p in re.findall(r"const\s+[\w ]+\*\s*__restrict__\s+(\w+)", params)
                            if (k, p) not in FIXED]
                todo += [c for c in re.findall(r"\b(\w+)\s*(?:<[^;(){}]*>)?\(", body) if c in fn]
    assert not bad, bad

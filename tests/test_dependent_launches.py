"""CPU check of the kernels that may become resident while the kernel before them
still stores (programmatic dependent launch): each waits for that kernel, and
neither it nor a device function that it calls reads global memory by the
read-only path, whose loads need not stay behind the wait."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_1205_2927_gb300" / "csrc"


def _balanced(text, i, pair):
    depth = 0
    while True:
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        i += 1
        if depth == 0:
            return i


def _functions(text):
    """{name: its text, from the declaration to the closing brace} of a file's device code."""
    found = {}
    for m in re.finditer(r"__(?:global|device)__", text):
        head = re.compile(r"(\w+)\s*\(").finditer(text, m.end())
        for h in head:   # the first call-like word that is no attribute is the name
            if h.group(1) not in ("__launch_bounds__", "__maxnreg__", "__cluster_dims__", "__align__"):
                break
        i = _balanced(text, h.end() - 1, "()")
        rest = text[i:].lstrip()
        if rest.startswith("{"):
            j = text.index("{", i)
            found.setdefault(h.group(1), "")
            found[h.group(1)] += text[m.start(): _balanced(text, j, "{}")]
    return found


def _dependent_kernels(text):
    names = set(re.findall(r"launch_dep\(\s*(\w+)", text))
    if "cudaLaunchAttributeProgrammaticStreamSerialization" in text:
        names |= set(re.findall(r"cudaLaunchKernelEx\(&cfg,\s*(\w+)", text))
    if "kern" in names:   # a variable: every kernel that it may hold
        names.discard("kern")
        names |= set(re.findall(r"auto kern = (\w+)", text))
    return names


def test_dependent_kernels_wait_and_read_by_plain_loads():
    seen, common = set(), _functions((CSRC / "ptx.cuh").read_text())
    for path in sorted(CSRC.glob("*.cu")):
        text = re.sub(r"//[^\n]*", "", path.read_text())
        functions = {**common, **_functions(text)}
        for kernel in _dependent_kernels(text):
            assert kernel in functions, (path.name, kernel)
            seen.add(kernel)
            reached, todo = set(), [kernel]
            while todo:
                name = todo.pop()
                reached.add(name)
                todo += [f for f in functions if f not in reached and re.search(r"\b%s\b" % f, functions[name])]
            assert re.search(r"\bdep_(wait|start)\(\)", functions[kernel]), (path.name, kernel)
            for name in reached:
                assert "__ldg(" not in functions[name], (path.name, kernel, name)
                assert not re.search(r"const \w+\* __restrict__", functions[name]), (path.name, kernel, name)
    assert {"leaf_gemm_kernel", "leaf_gemm_pair_kernel", "small_gemm_kernel", "mlp_adam_kernel", "rowdot64_kernel",
            "post_add3_kernel", "split16_kernel"} <= seen

"""Loads of the kernels that start while their predecessor still runs.

A kernel that calls launched() is resident on the SMs while the kernel before
it writes. Read-only (non-coherent) loads, __ldg and what the compiler makes of
const __restrict__ pointers, are defined only for data that nothing writes
during the kernel's lifetime, so neither may occur in such a kernel or in what
it calls. Checked on the source text, over the functions that each kernel's
body reaches by name.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2505_07392_gb300", "csrc")


def functions(text):
    """{name: [signature and body, ...]} of the functions defined at the start of a line."""
    text = re.sub(r"//[^\n]*", "", text)
    text = re.sub(r"^#[^\n]*(\\\n[^\n]*)*", "", text, flags=re.M)
    found = {}
    for m in re.finditer(r"\{", text):
        # a body opens at depth 0 of namespaces, after a parameter list
        head = text[:m.start()].rstrip()
        if not head.endswith(")"):
            continue
        begin = max(head.rfind(c, 0, len(head)) for c in ";}")
        sig = head[begin + 1:]
        if "__device__" not in sig and "__global__" not in sig:
            continue
        flat = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)|__maxnreg__\([^()]*\)", "", sig)
        name = re.search(r"(\w+)\s*\(", flat).group(1)
        depth, end = 0, m.start()
        while True:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
            if depth == 0:
                break
        found.setdefault(name, []).append(sig + text[m.start():end])
    return found


def reached(found, name):
    seen, todo = set(), [name]
    while todo:
        n = todo.pop()
        if n in seen:
            continue
        seen.add(n)
        for body in found[n]:
            todo += [w for w in set(re.findall(r"\b\w+\b", body)) if w in found and w not in seen]
    return seen


def test_no_read_only_loads_in_overlapped_kernels():
    found = {}
    for f in ("igr_kernels.cu", "igr_api.cu"):
        for name, bodies in functions(open(os.path.join(CSRC, f)).read()).items():
            found.setdefault(name, []).extend(bodies)
    kernels = [n for n, bodies in found.items() if any("__global__" in b and "launched();" in b for b in bodies)]
    assert len(kernels) >= 15 and {"k_flux", "k_speed", "k_sweep", "k_jacobi_full", "k_source"} <= set(kernels)
    bad = set()
    for k in kernels:
        for n in reached(found, k):
            for body in found[n]:
                if "__ldg" in body or "__restrict__" in body:
                    bad.add((k, n))
    assert not bad, sorted(bad)


def test_every_overlapped_kernel_waits_first():
    """launched() is the first statement: no access is made before the wait."""
    for f in ("igr_kernels.cu", "igr_api.cu"):
        for name, bodies in functions(open(os.path.join(CSRC, f)).read()).items():
            for b in bodies:
                if "__global__" in b and "launched();" in b:
                    assert re.search(r"\)\s*\{\s*launched\(\);", b), name

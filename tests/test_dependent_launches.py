"""Kernels may be set up while the kernel before them on the stream still writes (programmatic launches).  What
that asks of the sources, checked by reading them:

  - a kernel that is launched so waits for the end of the one before it (grid_dep_wait);
  - it reads nothing through the non-coherent path, which promises that the memory does not change during the
    kernel's life: no __ldg, no .nc loads, no pointer parameters that are const and __restrict__ at once.  (A kernel
    with an ordinary launch, or a cooperative one, may.)"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_23111_b200", "csrc")


def sources():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            text = open(os.path.join(CSRC, name)).read()
            yield name, re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def functions(text, head):
    """(name, parameters, body) of each function whose declaration starts with `head`."""
    for m in re.finditer(head + r"[^;{]*?(\w+)\s*\(", text):
        name, i, depth = m.group(1), m.end(), 1
        if name == "__launch_bounds__":
            i = text.index(")", i) + 1
            m2 = re.compile(r"\s*(\w+)\s*\(").match(text, i)
            name, i = m2.group(1), m2.end()
        p0 = i
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        j = text.index("{", i)
        k, depth = j + 1, 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        yield name, text[p0:i], text[j:k]


def read():
    kernels, device, ordinary = {}, {}, set()
    for _, text in sources():
        ordinary |= set(re.findall(r"cudaLaunchCooperativeKernel\(reinterpret_cast<void\*>\((\w+)", text))
        ordinary |= set(re.findall(r"(\w+)(?:<\w+>)?<<<", text))
        kernels.update((n, (p, b)) for n, p, b in functions(text, "__global__"))
        device.update((n, (p, b)) for n, p, b in functions(text, "__device__"))
    # (the eigen-solver picks its kernel through a pointer: kern is jacobi_kernel<..>, on_grid a kernel that waits)
    return kernels, device, (ordinary - {"kern", "on_grid"}) | {"jacobi_kernel"}


def test_kernels_wait_for_the_one_before_them():
    kernels, device, ordinary = read()
    assert len(kernels) >= 30 and {"chol_inv_kernel", "ln_colsum_partial_kernel"} <= ordinary <= set(kernels)
    assert "grid_dep_wait();" in device["gemm_tc_body"][1]
    for name, (_, body) in kernels.items():
        assert ("grid_dep_wait();" in body or "gemm_tc_body<" in body) != (name in ordinary), name
    for _, text in sources():                     # an ordinary launch is the only one that such a kernel gets
        for name in ordinary:
            assert not re.search(r"PRAC_LAUNCH\(" + name + r"\b", text), name


def test_no_load_promises_that_memory_does_not_change():
    kernels, device, ordinary = read()
    for name, (params, body) in list(kernels.items()) + list(device.items()):
        if name in ordinary:
            continue
        if name == "gemm_tc_body":                # (its loaders of plain loads: in kernels with an ordinary launch)
            loaders = re.search(r"\} else if \(A_LDG && warp >= .*?\n  \} else \{", body, flags=re.S).group(0)
            body = body.replace(loaders, "")
            assert "ldg_pair(" not in body
            assert any("cfg.numAttrs = LDG ? 1 : 2;" in text for _, text in sources())
        if name == "ldg_pair":
            continue
        assert "__ldg(" not in body and not re.search(r"ld\.global\.[\w.:]*\bnc\b", body), name
        assert not re.search(r"const\s+[\w:]+\s*\*\s*__restrict__", params), name

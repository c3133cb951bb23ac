"""Kernels that may start before their predecessor has ended (they call grid_dep_wait())
read its results: no such load may go through a pointer that promises read-only data for
the kernel's whole life (const with __restrict__, or __ldg), which would let the compiler
move it in front of the wait.  Checked in the sources, in the kernels and in every
device function that they call."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_09001_gb300", "csrc")
SHARED_MEMORY = {"stab"}   # parameters that point to shared memory


def _functions():
    """name -> list of (parameters, body) of the functions marked __global__ or __device__."""
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__(?:global|device)__\s[^;{}=]*?\b(\w+)\s*\(", src):
            name, i = m.group(1), m.end()
            if name == "__launch_bounds__":   # the name follows the bounds
                m2 = re.compile(r"[^;{}]*?\)\s*\n?\s*(\w+)\s*\(").match(src, i)
                name, i = m2.group(1), m2.end()
            depth, j = 1, i
            while depth:
                depth += {"(": 1, ")": -1}.get(src[j], 0)
                j += 1
            params, k = src[i:j - 1], j
            rest = re.compile(r"\s*(?:const\s*)?\{").match(src, k)
            if not rest:
                continue
            depth, k = 1, rest.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[k], 0)
                k += 1
            out.setdefault(name, []).append((params, src[rest.end():k]))
    return out


def test_no_read_only_loads_behind_a_dependent_launch():
    funcs = _functions()
    waiting = {n for n, fs in funcs.items() if n != "grid_dep_wait" and any("grid_dep_wait()" in b for _, b in fs)}
    # every kernel given to launch_pdl waits itself or in a body that it calls
    assert {"wl_table_kernel", "adj_finalize_kernel", "adj_gx_tma_kernel", "adj_gh_tma_body", "adj_gh_tma_batched_kernel",
            "sq_error_kernel", "sq_error_grad_kernel", "adam_kernel", "basis_kernel", "gram_lag_reduce_kernel",
            "gram_lag_reduce_few_kernel", "gram_lag_assemble_kernel", "chol_pair_kernel", "chol64_kernel",
            "chol_solve_kernel"} <= waiting, waiting
    reach, todo = set(), list(waiting)
    while todo:
        n = todo.pop()
        if n in reach:
            continue
        reach.add(n)
        for _, body in funcs[n]:
            todo += [c for c in set(re.findall(r"\b(\w+)\s*[<(]", body)) if c in funcs]
    for n, fs in funcs.items():   # a member of a structure of one of them
        if n in ("window", "init", "issue"):
            reach.add(n)
            for _, body in fs:
                reach |= {c for c in re.findall(r"\b(\w+)\s*[<(]", body) if c in funcs}
    bad = []
    for n in sorted(reach):
        for params, body in funcs[n]:
            for p in re.findall(r"\bconst\s+\w+\s*\*\s*__restrict__\s*(\w+)", params):
                if p not in SHARED_MEMORY:
                    bad.append(f"{n}: const __restrict__ {p}")
            if "__ldg" in body:
                bad.append(f"{n}: __ldg")
    assert not bad, "\n".join(bad)

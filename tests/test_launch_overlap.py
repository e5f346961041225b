"""Kernels whose blocks are set up before the kernel ahead of them is done: what the
sources have to keep for that to be safe.  ld4 and __ldg read by the non-coherent
path, which is for data that nobody writes while the reading kernel is resident; so a
kernel that writes real arrays does not let the next kernel in before its last block
is done, and the column lists (written by kernels that do) are read by __ldg only in
kernels launched plainly."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2405_13165_gb300", "csrc")


def _kernels():
    """(file, name, parameters, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?"
                             r"(k_\w+)\s*\(", src):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            params, depth = src[m.end():i - 1], 0
            j = k = src.index("{", i)
            while True:
                depth += {"{": 1, "}": -1}.get(src[k], 0)
                k += 1
                if not depth:
                    break
            yield os.path.basename(path), m.group(1), params, src[j:k]


def _writes_real(params):
    """A parameter through which real arrays are written: a pointer to non-const 4-vectors
    or reals, or a particle state other than the input."""
    for p in params.split(","):
        p = " ".join(p.split())
        if re.match(r"(vec4_t<\w+>|float4|TS?|float) \*", p) or re.match(r"StateT<T> (?!in\b)", p):
            return True
    return False


def test_every_kernel_waits_first():
    kernels = list(_kernels())
    assert len(kernels) >= 35
    for path, name, _, body in kernels:
        assert re.match(r"\{\s*pdl_(sync|wait)\(\);", body), (path, name)


# writers that do, with the kernel that always follows and what that one may read by ld4
FOLLOWED = {"k_classify": ("k_smooth", None), "k_survivors": ("k_to2d", r"in\."),
            "k_to2d": ("k_append", r"in\."), "k_cells": ("k_cell_table", None)}


def test_followers_read_nothing_of_theirs_non_coherently():
    bodies = {name: body for _, name, _, body in _kernels()}
    for follower, allowed in FOLLOWED.values():
        assert "__ldg" not in bodies[follower]
        for arg in re.findall(r"\bld4\(\s*([^,]*?)\)", bodies[follower]):
            assert allowed and re.match(allowed, arg), (follower, arg)
    # the launches are in that order: nothing is launched between the two
    for first, (follower, _) in FOLLOWED.items():
        if first == "k_cells":    # the last kernel of the sort; the search goes on with the other
            continue
        src = "".join(open(p).read() for p in sorted(glob.glob(os.path.join(CSRC, "*.cu"))))
        tail = src[[m.end() for m in re.finditer(r"\blaunch\(\s*" + first + r"\b", src)][-1]:]
        assert re.search(r"\blaunch\(\s*(k_\w+)", tail).group(1) == follower, first


def test_writers_of_real_arrays_do_not_trigger_early():
    seen = set()
    for path, name, params, body in _kernels():
        if _writes_real(params):
            seen.add(name)
            if name in FOLLOWED:
                continue
            assert "pdl_sync()" not in body and "launch_dependents" not in body, (path, name)
    # the parameters are recognised: the operators, the states and the step's frames
    assert {"k_stencil", "k_stencil_redo", "k_stencil_grad", "k_apply", "k_apply_T_scatter",
            "k_classify", "k_cells", "k_append", "k_ghost_seed", "k_film_momentum"} <= seen


def test_lists_are_read_non_coherently_by_plain_launches_only():
    launched = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        launched |= set(re.findall(r"\blaunch\(\s*(k_\w+)", open(path).read()))
    assert "k_hash" in launched
    for path, name, _, body in _kernels():
        assert "__ldg" not in body or name not in launched, (path, name)

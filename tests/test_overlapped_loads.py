"""Kernels that may start before their predecessor ends read its results with ordinary loads.

A kernel launched with programmatic serialisation exists while the kernel before it still writes.
__ldg, and loads through a kernel's `const * __restrict__` parameters, are defined only for data that
nobody writes during the kernel's life.  This reads the sources: every kernel whose launch may overlap
(launch_k with anything but `false`) and every device function that it calls."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2401_10287_gb300", "csrc")
UPLOADED = {"nuc", "atom", "descs", "hf"}        # written by the host when the handle is set up


def _functions(text):
    """name -> [(kind, signature, body)] of the __global__ and __device__ functions of a source."""
    out = {}
    for m in re.finditer(r"\b(__global__|__device__)\b[^;{}()=]*?(\w+)\(", text):
        i, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        sig = text[m.start():i]
        j = i
        while text[j] in " \n" or text.startswith("const", j):
            j += 5 if text.startswith("const", j) else 1
        if text[j] != "{":
            continue
        k, depth = j + 1, 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        out.setdefault(m.group(2), []).append((m.group(1), sig, text[j:k]))
    return out


def _sources(csrc):
    texts = {}
    for path in sorted(glob.glob(os.path.join(csrc, "*.cu")) + glob.glob(os.path.join(csrc, "*.cuh"))):
        with open(path) as f:
            texts[os.path.basename(path)] = re.sub(r"//[^\n]*|__launch_bounds__\([^)]*\)", "", f.read())
    return texts


def faults(csrc):
    texts = _sources(csrc)
    funcs, overlapped = {}, set()
    for text in texts.values():
        for name, defs in _functions(text).items():
            funcs.setdefault(name, []).extend(defs)
        for m in re.finditer(r"\blaunch_k\(", text):
            i, depth = m.end(), 0                     # the first argument: whether the launch may overlap
            while depth or text[i] != ",":
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            first = text[m.end():i].strip()
            if first in ("false", "bool overlap"):    # (the latter: launch_k's own declaration)
                continue
            name = re.match(r",\s*(?:tc::)?(\w+)", text[i:]).group(1)
            kernels = re.findall(r"auto " + name + r" = (k_\w+)", text) or [name]
            overlapped.update(kernels)
    out = []
    for kernel in sorted(overlapped):
        assert any(kind == "__global__" for kind, _, _ in funcs.get(kernel, [])), kernel
        seen, todo = set(), [kernel]
        while todo:
            name = todo.pop()
            if name in seen:
                continue
            seen.add(name)
            for _, sig, body in funcs.get(name, []):
                if "__ldg(" in body:
                    out.append(f"{kernel}: __ldg in {name}")
                todo.extend(c for c in re.findall(r"\b(\w+)(?:<[^;()]*?>)?\(", body) if c in funcs)
        for kind, sig, _ in funcs[kernel]:
            if kind == "__global__":
                out.extend(f"{kernel}: const __restrict__ {p}" for p in
                           re.findall(r"const [\w:]+\s*\*\s*__restrict__ (\w+)", sig) if p not in UPLOADED)
    return overlapped, out


def test_overlapped_kernels_use_ordinary_loads():
    overlapped, out = faults(CSRC)
    assert {"k_prep", "k_features", "k_propose", "k_accept", "k_spin_means_bf16", "k_adam", "k_unprep", "k_tc",
            "k_layer_res", "k_orbital_fixup", "k_det_energy_grp", "k_bwd_dh"} <= overlapped
    assert not out, out

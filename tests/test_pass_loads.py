"""The passes that launch_pass starts while the kernel before them is still running
read what that kernel writes by TMA or by ordinary loads: a read-only load (__ldg,
or a restrict pointer, which the compiler may turn into one) is not ordered by the
wait at their start.  Shown on the sources: such a fault is a matter of timing and
of the compiler's schedule on a GPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_10519_gb300", "csrc")
FILES = ["stencil_tma.cu", "tti_sp_tma.cu", "elastic2d.cu", "tma.cuh", "common.cuh", "tile.cuh"]
# what no pass writes: layer tables, the model in the source factors, a batch's tables
READ_ONLY = re.compile(r"__ldg\((g\.tab|tab[xyz]|tzt|s[xyz])\b|__ldg\(inj(->|\.)m\b")


def text(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def block(src, start):
    """From `start` to the end of the function that begins there."""
    i = src.index("{", start)
    depth = 0
    for j in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if depth == 0:
            return src[start:j + 1]


def functions():
    """Name -> (signature, body) of every function of the files, with the callees still to be followed."""
    found = {}
    for name in FILES:
        src = text(name)
        for m in re.finditer(r"(?:WP_DEV|__global__)\s+[\w:<> ]+?(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\(", src):
            whole = block(src, m.start())
            i = whole.index("{")
            found[m.group(1)] = (whole[:i], whole[i:])
    return found


def launched():
    names = set()
    for name in FILES:
        names |= set(re.findall(r"launch_pass\((\w+)[<,]", text(name)))
    return sorted(names)


def reached(kernel, fns):
    todo, seen = [kernel], []
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.append(f)
        todo += [c for c in re.findall(r"\b(\w+)(?:<[^;{}()]*>)?\(", fns[f][1]) if c in fns]
    return seen


def test_the_passes_are_found():
    assert launched() == ["acu_tma", "el2_tpass_tma", "el2_vpass_tma", "el_tpass_tma", "el_vpass_tma", "tti_rot_tma",
                          "tti_sp_rot_tma", "tti_sp_upd_tma", "tti_upd_tma"]
    fns = functions()
    assert {"el_vpass_body", "v_preload", "ldf2"} <= set(reached("el_vpass_tma", fns))
    assert {"record_point", "sample_receivers"} <= set(reached("acu_tma", fns))


@pytest.mark.parametrize("kernel", launched())
def test_no_read_only_load_of_a_field(kernel):
    fns = functions()
    for f in reached(kernel, fns):
        head, body = fns[f]
        for m in re.finditer(r"__ldg\([^;]*", body):
            assert READ_ONLY.match(m.group()), (f, m.group()[:60])
        # fields are float arrays; restrict is for what is written only, the sparse-point tables and the wavelets
        for m in re.finditer(r"const float \*\s*__restrict__ (\w+)", head):
            assert (f, m.group(1)) in {("record_point", "w"), ("inject_sum", "w"), ("inject_sum", "traces")}, (f, m.group())

"""The step's kernels are launched so that one may begin before the writes of
the one before it are visible (programmatic stream serialization), and wait
for them in the kernel.  Loads through the non-coherent path are not ordered
by that wait and may be moved ahead of it, so the step has none; the readers
of the state, launched plainly, take it through one function's argument."""

import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2004_11286_gb300" / "csrc"


def test_step_kernels_use_coherent_loads():
    used = {}
    for f in sorted(CSRC.glob("lbm_*.cuh")):
        code = re.sub(r"//[^\n]*", "", f.read_text())
        used[f.name] = len(re.findall(r"__ldg\s*\(|ld\.global\.nc", code))
        if f.name in ("lbm_collide.cuh", "lbm_split.cuh", "lbm_batch.cuh", "lbm_frame.cuh"):
            assert not re.search(r"\bld<|(RowLoad|RowSide|RecLoad)<[^>]*true|eq_incoming|incoming_terms|load_rec", code), f.name
            for call in re.findall(r"\b(?:incoming_corr|deferred_terms)<([^>]*)>", code):
                assert len(call.split(",")) <= 3 and (call.count(",") < 2 or "WALL" in call), (f.name, call)
    assert {k: v for k, v in used.items() if v} == {"lbm_helpers.cuh": 1}      # ld<true>


def test_every_kernel_launched_so_waits_before_touching_memory():
    src = {f.name: re.sub(r"//[^\n]*", "", f.read_text()) for f in CSRC.glob("lbm_*.cuh")}
    names = set(re.findall(r"launch_next\(\s*(?:[^?(;]*\? )?(\w+)<", src["lbm_kernels.cuh"]))
    assert len(names) >= 9
    for name in names:
        body = next(s for s in src.values() if re.search(r"\b%s\(const __grid_constant__" % name, s))
        body = body[re.search(r"\b%s\(const __grid_constant__" % name, body).end():]
        body = body[body.index("{"):]
        wait = body.index("wait_previous()")
        before = body[:wait]
        for state in ("pops", "side", "gtid"):
            assert not re.search(r"\b%s\s*\[" % state, before) and "= gtid" not in before, (name, state)

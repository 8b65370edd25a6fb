"""The step's kernels are launched so that one may begin before the writes of
the one before it are visible (programmatic stream serialization), and wait
for them in the kernel.  Loads through the non-coherent path are not ordered
by that wait and may be moved ahead of it, so the device code that the step
shares must not contain any."""

import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2004_11286_gb300" / "csrc"


def test_step_kernels_use_coherent_loads():
    for f in sorted(CSRC.glob("lbm_*.cuh")):
        code = re.sub(r"//[^\n]*", "", f.read_text())
        assert not re.search(r"__ldg\s*\(|ld\.global\.nc", code), f.name


def test_every_kernel_launched_so_waits_before_touching_memory():
    src = {f.name: re.sub(r"//[^\n]*", "", f.read_text()) for f in CSRC.glob("lbm_*.cuh")}
    names = set(re.findall(r"launch_next\(\s*(?:parity == 0 \? )?(\w+)<", src["lbm_kernels.cuh"]))
    assert len(names) >= 9
    for name in names:
        body = next(s for s in src.values() if re.search(r"\b%s\(const __grid_constant__" % name, s))
        body = body[re.search(r"\b%s\(const __grid_constant__" % name, body).end():]
        body = body[body.index("{"):]
        wait = body.index("wait_previous()")
        before = body[:wait]
        for state in ("pops", "side", "gtid"):
            assert not re.search(r"\b%s\s*\[" % state, before) and "= gtid" not in before, (name, state)

"""The one-launch iterations share one arrival counter among their blocks.  The
first block through the last barrier may not touch it: another block's next
poll would read a counter below its target and wait out its two seconds.  The
source is checked here: only the kernel that prepares a launch stores to the
counter, no kernel but the one that resets a solve stores the whole state, and
what the scalar steps of BiCGSTAB change is what the end of a launch stores."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_03563_gb300", "csrc")


def _code():
    out = {}
    for f in sorted(os.listdir(CSRC)):
        s = open(os.path.join(CSRC, f)).read()
        out[f] = re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", s, flags=re.S))
    return out


def _body(code, name):
    """Text of the function `name` (from its parameter list to the matching brace)."""
    at = re.search(r"\b%s\s*\(" % name, code).start()
    i = code.index("{", at)
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(code[j], 0)
        j += 1
        if depth == 0:
            return code[i:j]


def test_only_the_preparation_stores_to_the_counter():
    stores = re.compile(r"\bgbar\s*=(?!=)")
    for f, code in _code().items():
        want = 1 if f == "cart_kernels.cu" else 0
        assert len(stores.findall(code)) == want, f
    assert stores.search(_body(_code()["cart_kernels.cu"], "k_set_budget"))


def test_whole_state_is_stored_by_the_reset_alone():
    whole = re.compile(r"[;{}]\s*\*\s*st\s*=(?!=)")
    for f, code in _code().items():
        assert len(whole.findall(code)) == (1 if f == "cart_kernels.cu" else 0), f
    assert whole.search(_body(_code()["cart_kernels.cu"], "k_init_state"))


def test_the_end_of_a_launch_stores_what_the_scalar_steps_change():
    code = _code()["spherical.cu"]
    changed = set()
    for f in ("bicg_scalar_logic", "bicg_replace_logic", "bicg_direction"):
        changed |= set(re.findall(r"st->(\w+)\s*[-+*]?=(?!=)", _body(code, f)))
    stored = set(re.findall(r"st->(\w+)\s*=(?!=)", _body(code, "bicg_store")))
    assert changed and stored == changed, stored ^ changed


def test_a_wait_that_ran_out_is_reported():
    """Any block whose wait runs out sets the solve's fault flag, and the host
    honours the flag whatever the kernel's first block reports."""
    code = _code()
    assert re.search(r"atomicExch\(\s*fault\s*,\s*1\s*\)", _body(code["stencil.cuh"], "grid_barrier"))
    assert re.search(r"->fault\s*\)\s*\w[\w>.-]*done\s*=\s*DONE_FAULT", _body(code["solver.cu"], "poll_active"))

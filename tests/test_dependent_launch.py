"""Kernels that may start before the kernel in front of them has finished (programmatic dependent
launch) read that kernel's results after their wait.  ``__restrict__`` on such a pointer would
promise that nobody else writes the memory while the kernel runs, and let the compiler move its loads
above the wait or take them through the non-coherent path; so in these kernels it may only stand on
the call's own inputs."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2608_28113_gb300" / "csrc"

# kernel -> parameters that only hold the call's own inputs, complete before its first kernel starts
INPUTS = {
    "rtn_codes_kernel": {"w"},
    "amax_kernel": {"w"},
    "split_u_kernel": {"U"},
}


def dependent_kernels():
    found = {}
    for path in sorted(CSRC.glob("*.cu")):
        src = re.sub(r"//[^\n]*", "", path.read_text())
        for m in re.finditer(r"__global__\s+void\s+(?:__\w+__\s*\([^()]*(?:\([^()]*\)[^()]*)*\)\s*)*(\w+)\s*\(", src):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            params, body = src[m.end():i - 1], src[i:]
            body = body[:re.search(r"\n}\n", body).start()]
            if "pdl_wait_primary()" in body:
                found[m.group(1)] = params
    return found


def test_only_inputs_are_restrict_in_dependent_kernels():
    kernels = dependent_kernels()
    assert {"rtn_codes_kernel", "factor_panel_kernel", "factor_diag_kernel", "split_u_kernel", "update_kernel",
            "gptq_panel_kernel", "hessian_colsumsq_kernel"} <= set(kernels)
    for name, params in kernels.items():
        restricted = set(re.findall(r"__restrict__\s+(\w+)", params))
        assert restricted <= INPUTS.get(name, set()), f"{name}: {restricted - INPUTS.get(name, set())}"

"""Rules of the device code that a run cannot show to be broken (a race or a hang that a build happens not to
have), checked on the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1801_05648_gb300", "csrc")


def _source(name):
    """The file without comments and line continuations."""
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _kernels():
    """{kernel name: (file, parameter list, body)} of every __global__ function defined in the sources."""
    found = {}
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        text = _source(name)
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            params = text[m.end():i - 1]
            body = text.index("{", i)
            depth, j = 1, body + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[j], 0)
                j += 1
            found[m.group(1)] = (name, params, text[body:j])
    return found


def test_kernels_are_found():
    k = _kernels()
    assert {"k_bsr_spmv", "k_operator_rows", "k_spgemm_sym", "k_gj_panel", "k_mlp_tc", "k_jacobian"} <= set(k)


def test_spgemm_rows_leave_their_loop_together():
    """A flag in shared memory that another warp may be setting can look different to the 32 lanes of a
    warp; lanes that leave a loop on it would miss the warp-wide operations that the others wait in."""
    body = _kernels()["k_spgemm_sym"][2]
    exits = re.findall(r"if \(([^;{}]*)\) break;", body)
    assert exits
    for cond in exits:
        assert "volatile" not in cond or cond.startswith("__any_sync(0xffffffffu,"), cond


# What no queued kernel writes while another may be resident: matrices with their patterns, the inverse
# diagonals and the coarse inverse of a built preconditioner, the weights.
_CONSTANT = {"ord2", "rp1", "ci1", "v1", "rp2", "ci2", "v2", "rp", "ci", "v", "M", "dinv", "w16"}


def test_overlapping_kernels_read_vectors_with_ordinary_loads():
    """A kernel that may be resident before the kernel ahead of it has finished must not declare what
    that kernel writes read-only: an invariant load may be moved ahead of the wait."""
    overlapping = {k: v for k, v in _kernels().items() if re.search(r"\bdep_wait|\bbsr_rows<", v[2])}
    assert len(overlapping) >= 28, sorted(overlapping)
    for kernel, (name, params, _) in overlapping.items():
        declared = set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params))
        assert declared <= _CONSTANT, (name, kernel, declared - _CONSTANT)
    text = _source("spmv.cuh")
    assert set(re.findall(r"__ldg\((\w+)", text)) == {"ord2"}
    for loader in ("load_gather", "load_gather_keep"):
        assert re.search(r"void %s\(const \w+\* p," % loader, text), loader
    rows = text[text.index("void bsr_rows("):]
    assert set(re.findall(r"const\s+\w+\*\s*__restrict__\s+(\w+)", rows[:rows.index("{")])) <= _CONSTANT
    for name in os.listdir(CSRC):
        if name.endswith((".cu", ".cuh")):
            assert "ld.global.nc" not in _source(name), name
    for name in ("vec.cu", "solver.cu", "mlp_tc.cu", "amg.cu"):
        assert "__ldg" not in _source(name), name


def _function(text, name):
    """The body of the function whose definition names `name(`."""
    start = text.index("{", text.index(name + "("))
    depth, i = 1, start + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[start:i]


def test_persistent_launches_neither_load_early_nor_trigger():
    """The registers of the early loads cost a launch that fills the GPU its occupancy; a persistent one
    (more rows per CTA than threads allow in a pass) fills it although its CTAs are few."""
    text = _source("spmv_inst.cuh")
    assert "rows_per_cta * tpr <= 256" in _function(text, "bool one_pass")
    assert "one_pass(rows_per_cta, tpr)" in _function(text, "bool loads_early")
    assert re.search(r"one_pass\(rows_per_cta, tpr\) \? kDepTrigger : 0", text)
    for name, source in (("spmv_inst.cuh", text), ("spmv64.cu", _source("spmv64.cu"))):
        decided = re.findall(r"const bool early = ([^;]*);", source)
        assert decided and all("loads_early(" in d for d in decided), name


def test_fp64_preconditioner_calls_share_their_launch_shapes():
    """Every call that runs products of the FP64 preconditioner runs them as the solve does."""
    solver = _source("solver.cu")
    for text, name in ((solver, "void precond_apply"), (solver, "void apply_block"),
                       (_source("noalloc.cu"), "int fsi_mass_solve_noalloc"),
                       (_source("fsi_api.cu"), "int fsi_smoother_step")):
        assert "WideRows64 wide(" in _function(text, name), name

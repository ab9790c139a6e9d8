"""A refused kernel launch is reported by the call that made it: a successful
cudaFuncSetAttribute clears the runtime's last error, so every limit is raised through
raise_smem_limit, which keeps an error that is pending, and every check reads
the kept one (take_launch_error)."""
import ctypes
import os
import re

import pytest

from paper_2102_11576_gb300 import LIB_PATH, workloads

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2102_11576_gb300", "csrc")


@pytest.mark.parametrize("call,users", [("cudaFuncSetAttribute", 1), ("cudaGetLastError", 1)])
def test_errors_are_kept_and_read_in_one_place(call, users):
    found = []
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".inc", ".h")):
            with open(os.path.join(CSRC, name)) as f:
                code = re.sub(r"//.*", "", f.read())
            found += [name] * len(re.findall(call + r"\s*\(", code))
    assert found == ["transforms.cu"] * users


@pytest.mark.gpu
@pytest.mark.parametrize("opts", [dict(), dict(precond="bf16x3", matvec="fp32", resid="exact"),
                                  dict(precond="fp32", matvec="fp32")])
def test_an_error_before_the_last_launch_is_reported_once(opts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2102_11576_gb300 import RsfdeError, Solver
    w = workloads.random_problem(3, 96, 80)
    s = Solver(w["n1"], w["n2"], w["box"], w["in_omega"], w["alpha1"], w["alpha2"], w["kx"], w["ky"], w["dt"],
               w["eta"], use_graph=False, **opts)
    v = torch.as_tensor(w["field"]).cuda()
    refuse = ctypes.CDLL(LIB_PATH)["_ZN5rsfde16raise_smem_limitEPKvi"]  # rsfde::raise_smem_limit
    refuse.argtypes = [ctypes.c_void_p, ctypes.c_int]
    refuse.restype = None
    for call in (lambda: s.apply_precond(v), lambda: s.apply_M(v), lambda: s.solve(v)):
        refuse(None, 1024)  # no such kernel: an error of the runtime
        with pytest.raises(RsfdeError) as e:
            call()
        assert e.value.name == "ECUDA"
        call()
    s.close()

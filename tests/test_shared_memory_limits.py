"""A kernel's dynamic shared-memory limit belongs to the process. Calls that run without the fit lock
set it by the helper that only raises it (fitcore_raise_eval_smem), or to one constant; a limit set
to the model in hand could be lowered by another thread's call between here and the launch."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_models_limits_are_only_raised():
    set_in = {}
    for path in glob.glob(os.path.join(ROOT, "paper_2502_15253_gb300", "csrc", "*.cu")):
        src = re.sub(r'"[^"\n]*"', '""', open(path).read())
        n = len(re.findall(r"cudaFuncSetAttribute\s*\(", src))
        if n:
            set_in[os.path.basename(path)] = n
    # capi.cu: the helper, and the fits (under the lock that their launches hold too); gemm_tc.cu: raises
    # under a lock of its own; events.cu: one constant
    assert set(set_in) == {"capi.cu", "gemm_tc.cu", "events.cu"}
    events = open(os.path.join(ROOT, "paper_2502_15253_gb300", "csrc", "events.cu")).read()
    assert "const int dyn = 2 * (int)sizeof(fitcore::Stage);" in events
    gemm = open(os.path.join(ROOT, "paper_2502_15253_gb300", "csrc", "gemm_tc.cu")).read()
    assert re.search(r"if \(\(int\)smem > cur\) \{[^}]*cudaFuncSetAttribute", gemm)

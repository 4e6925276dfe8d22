"""GPU: a tuned choice is reused for the same launch only.

The autotuner runs one iteration before it times a handle's variants, so hbugks_create enqueues one iteration more when it
tunes than when it finds the choice (the graphs take 18: one, sixteen and the body of the loop), which the NVTX ranges show.
"""
import pytest

from test_tracing import recorder, run_traced  # noqa: F401  (recorder is a fixture)

pytestmark = pytest.mark.gpu

CODE = """
import torch
from paper_2605_03479_gb300 import hbugks as hb, inputs as I
def case(precision, pr=2 / 3):
    return I.make_case('t', 6, 8, kn=0.1, st=1.0, nh=1, pr=pr, drive='shear', precision=precision)
for precision in (0, 1):
    hb.Solver(case(precision)).destroy()                        # tunes
    hb.Solver(case(precision)).destroy()                        # the same
    hb.Solver([case(precision), case(precision)]).destroy()     # a batch: another instance of the kernel
    hb.Solver(case(precision, pr=1.0)).destroy()                # another collision model
empty = torch.empty
full = hb.workspace_bytes([case(0)])
def scarce(n, *args, **kw):
    if isinstance(n, int) and n >= full:
        raise torch.OutOfMemoryError('short')
    return empty(n, *args, **kw)
torch.empty = scarce
hb.Solver(case(0)).destroy()                                    # slopes formed again
"""


def test_a_choice_is_reused_for_the_same_launch_only(recorder, tmp_path):  # noqa: F811
    lines = run_traced(recorder, tmp_path, CODE)
    tuned, depth, count = [], 0, 0
    for ln in lines:
        if ln == "push hbugks_create":
            depth, count = 1, 0
        elif depth:
            depth += 1 if ln.startswith("push ") else -1
            count += ln == "push k5_finish"
            if depth == 0:
                assert count in (18, 19)
                tuned.append(count == 19)
    assert tuned == [True, False, True, True] * 2 + [True]

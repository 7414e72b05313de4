"""The barrier schedule of slice_gemm_kernel (csrc/slicemm.cuh) over every interleaving, in the GEMM kernels' model.

Its eight sums are handed over in three groups: the UMMA thread goes over a chunk's groups in turn, waits before a
flush's first UMMAs of a group until every read-back warp has read that group's last flush, and commits the group after
its last chunk, the stage after all three.  To the model, group h of flush f is segment 3 f + h of three accumulators,
whose UMMAs of one chunk lie between those of the others."""
import pytest

import test_gemm_protocol as base

STAGES, GROUPS = 2, 3


def _programs(flushes, readers):
    """flushes: chunks of each."""
    chunks = sum(flushes)
    tma = []
    for i in range(chunks):
        tma += [("wait", (base.EMPTY, i % STAGES), i // STAGES - 1), ("load", (base.FULL, i % STAGES), i)]
    tma += [("wait", (base.FULL, i % STAGES), i // STAGES) for i in range(max(0, chunks - STAGES), chunks)]
    mma, i = [], 0
    for f, n in enumerate(flushes):
        for c in range(n):
            mma.append(("wait", (base.FULL, i % STAGES), i // STAGES))
            for h in range(GROUPS):
                if c == 0:
                    mma += [("wait", (base.ACCE, h, r), f - 1) for r in range(readers)]
                mma.append(("umma", GROUPS * f + h, c == 0))
                if c == n - 1:
                    mma.append(("commit", (base.ACCF, h), ("seg", GROUPS * f + h)))
            mma.append(("commit", (base.EMPTY, i % STAGES), ("step", i)))
            i += 1
    mma += [("commit", (base.DRAIN,), ("drain",)), ("wait", (base.DRAIN,), 0)]
    read = []
    for r in range(readers):
        read.append([op for m in range(GROUPS * len(flushes)) for op in
                     (("wait", (base.ACCF, m % GROUPS), m // GROUPS), ("read", m, r),
                      ("arrive", (base.ACCE, m % GROUPS, r)))])
    return [tma, mma] + read


@pytest.mark.parametrize("readers", [1, 2])
@pytest.mark.parametrize("flushes", [[1], [2], [1, 1, 1], [2, 1], [2, 2, 1], [4, 4], [3, 1, 2]])
def test_three_groups_a_flush(flushes, readers):
    assert base.explore(flushes, STAGES, GROUPS, readers, _programs(flushes, readers)) > 0


@pytest.mark.parametrize("drop", [base.EMPTY, base.ACCE, base.FULL])
def test_the_model_sees_a_missing_wait(drop):
    progs = _programs([2, 2, 1], 1)
    role = 0 if drop == base.EMPTY else 1
    progs[role] = [op for op in progs[role] if not (op[0] == "wait" and op[1][0] == drop)]
    with pytest.raises(base.Violation):
        base.explore([2, 2, 1], STAGES, GROUPS, 1, progs)

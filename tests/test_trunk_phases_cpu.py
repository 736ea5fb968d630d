"""The trunk kernel's barriers as a model.  Between the epilogue and the MMA
issuer: a parity wait only tells a barrier's current phase from the one before
it, so the issuer has to wait for every phase in turn.  The model delays one
arrival as long as the waits allow and looks whether a job is issued on a tile
that is not complete.  Between the MMAs and the weight loader: the arrivals
that release a stage come from the even CTA's tensor core on both CTAs'
barriers, so each loader has to see the last of them before its CTA may exit.
Which waits are made is read from the kernel's source."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_05009_gb300", "csrc",
                   "trunk.cuh")


def waits_at_a_tile_start():
    """True if the issuer waits for the slot's previous job before job 0 too."""
    with open(SRC) as f:
        text = f.read()
    issuer = text[text.index("even CTA: MMA issuer"):]
    issuer = issuer[:issuer.index("tc_fence_after")]
    return re.search(r"jobs\[p\] == 0 \|\|\s*tr_wait\(&ctl->aready\[p\]", issuer) is not None


def loader_waits_at_its_end():
    """True if the weight loader waits for the release of every stage last."""
    with open(SRC) as f:
        text = f.read()
    end = text[text.index("copy_async_wait_all"):]
    end = end[:end.index("} else if")]
    return re.search(r"i < TR_WSTAGES.*\n\s*ok = tr_wait\(&ctl->wempty\[w\.s\], w\.ph \^ 1u", end) is not None


def parity_wait_returns(completed, parity):
    """mbarrier.try_wait.parity with `completed` phases complete: true for the
    parity of the phase before the current one."""
    return (completed - 1) & 1 == parity


@pytest.mark.parametrize("jobs_per_tile", [8, 9])
def test_no_job_reads_an_incomplete_tile(jobs_per_tile):
    at_start = waits_at_a_tile_start()
    for late in range(3 * jobs_per_tile):  # the job whose last arrival is delayed
        for job in range(3 * jobs_per_tile):
            # jobs before `job` have arrived but for `late`; phases complete in order
            completed = min(job, late)
            waits = (job - 1) & 1 if job > 0 and (job % jobs_per_tile != 0 or at_start) else None
            if waits is not None and not parity_wait_returns(completed, waits):
                break  # the issuer waits, until the arrival comes
            # issued: jobs in the middle of a tile read the previous job's output
            assert job % jobs_per_tile == 0 or completed == job, (late, job)


@pytest.mark.parametrize("fills", [1, 4, 5, 6, 33, 330])
def test_no_release_is_on_its_way_when_the_loader_ends(fills):
    stages = 5
    seen = [0] * stages  # releases of each stage that the loader has waited for
    s, ph = 0, 0
    for i in range(fills + (stages if loader_waits_at_its_end() else 0)):
        # the wait before fill i: parity ph ^ 1, true at once in the first turn
        turn = i // stages
        assert (s, ph) == (i % stages, turn & 1)
        seen[s] = turn
        s, ph = (s + 1, ph) if s + 1 < stages else (0, ph ^ 1)
    for k in range(stages):
        assert seen[k] == len(range(k, fills, stages)), k

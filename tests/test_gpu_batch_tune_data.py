"""The batch tuner times the vector passes on ordinary numbers: before the first step, when
the basis holds nothing yet, they take as long as after one (zeros would send every
sum to the binary64 fallback, 1.25 times the time of the passes that steps run)."""
import pytest
import torch

from paper_1607_06834_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_passes_are_timed_on_the_path_that_steps_take():
    from paper_1607_06834_gb300 import rok
    inst = W.batched_instances(64, 32, 384)
    b = rok.rok_batch_init([i.problem for i in inst], krylov_max=16)
    y0 = b.pack([i.y0 for i in inst])

    def passes():   # the fastest of four tunings, each candidate's mean over three launches
        t = [rok.rok_batch_tune(b, y0)['mgs_ms'] for _ in range(4)]
        return [min(x[q] for x in t) for q in range(4)]

    before = passes()
    y = y0.clone()
    rok.rok_batch_step(b, y, 1e-4, 16)
    torch.cuda.synchronize()
    after = passes()
    assert max(x / z for x, z in zip(before, after)) <= 1.12, (before, after)

    # and the tuner leaves nothing behind that a step could see
    c = rok.rok_batch_init([i.problem for i in inst], krylov_max=16)
    t = rok.rok_batch_get_tuning(b)
    rok.rok_batch_set_tuning(c, t['tile'], t['chunks_per_cta'], t['vec_chunks_per_cta'])
    z = y0.clone()
    rok.rok_batch_step(c, z, 1e-4, 16)
    y.copy_(y0)
    rok.rok_batch_step(b, y, 1e-4, 16)
    assert torch.equal(y, z)

"""Drafts of 17..64 sequences on a shape whose phases all give their tiles whole CTAs: the column groups of a tile are dealt to
its contributors, which wait for one another."""
import time

import numpy as np
import pytest

from tests.harness import LOGIT_RTOL, row_rel_err
from tests.recorded import Run

pytestmark = pytest.mark.gpu


def start(shape, B, seed):
    r = Run(shape, seed, batch=B, rows=200)
    r.counts = [1 + (7 * b) % 90 for b in range(B)]
    r.prefill(r.counts)
    r.forced = r.torch.randint(0, r.dims.vocab, (B, 3), dtype=r.torch.int32, device="cuda", generator=r.gen)
    return r


def window(r, B):
    r.dr.set_kv_len_batch([n - 1 for n in r.counts], restore_pending=True)
    _, logits = r.dr.draft(B, 3, r.resid, forced_ids=r.forced, want_logits=True)
    rows = [t for b in range(B) for t in r.dr.read_kv(b, r.counts[b] - 1, 3)]
    return logits.cpu().numpy(), r.torch.stack(rows).cpu().numpy()


@pytest.mark.parametrize("shape", ["wide128", "wide64"])
@pytest.mark.parametrize("B", [17, 32, 33, 49, 64])
def test_dealt_column_groups_against_the_per_phase_kernels(shape, B):
    """Both round the activations between the layers to bf16 and add in fp32: the logits agree to the tolerance that the oracle
    comparison of bf16 drafts has, the appended rows to one unit in the last place of bf16 (2^-8) where a sum falls next to a
    rounding, of values whose inputs differ by the same again."""
    r = start(shape, B, 21)
    got, rows = window(r, B)
    r.dr.set_tc_kernel(0)
    want, ref = window(r, B)
    r.dr.status()
    assert row_rel_err(got, want).max() <= LOGIT_RTOL
    assert np.abs(rows - ref).max() <= 2.0 ** -6 * np.abs(ref).max()


@pytest.mark.parametrize("B", [17, 32, 33, 64])
def test_waits_run_out_cleanly_and_the_context_recovers(B):
    """The grid barriers of one draft are made impossible to complete: every wait, those for a tile's other contributors among
    them, ends at its limit, the status says so, and the same draft then gives what it gave before, bit for bit."""
    from paper_2509_23928_b200 import HivisError
    r = start("wide128", B, 22)
    want, ref = window(r, B)
    r.dr.set_wait_limit_us(2000)
    r.dr.miss_next_barrier()
    t0 = time.perf_counter()
    window(r, B)
    assert time.perf_counter() - t0 < 10.0
    with pytest.raises(HivisError) as e:
        r.dr.status()
    assert e.value.code == -7
    r.dr.status()
    r.dr.set_wait_limit_us(1000000)
    got, rows = window(r, B)
    r.dr.status()
    assert np.array_equal(got, want) and np.array_equal(rows, ref)

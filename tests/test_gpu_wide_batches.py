"""Drafts of 17..64 sequences on a shape whose phases all give their tiles whole CTAs: the column groups of a tile are dealt to
its contributors, which wait for one another."""
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

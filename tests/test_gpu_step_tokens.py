"""Token copies of a decode step: steps whose tokens nobody reads (uploads that follow
one another without a wait in between), reads after steps on the device alone, and the
tokens of several sequences, against steps read one by one."""
import numpy as np
import pytest

from oracle import model as M
from tests.gpu_helpers import arch_dict, torch_mod

pytestmark = pytest.mark.gpu

TINY = M.Arch(1, 512, 8, 8, 64, 1376, 32000)


@pytest.fixture(scope="module")
def fp():
    torch_mod()
    import paper_2501_13111_gb300 as fp

    return fp


@pytest.mark.parametrize("batch", [1, 5])
def test_unread_steps_and_reads_agree(fp, batch):
    rng = np.random.default_rng(batch)
    prompt = rng.integers(0, 32000, (batch, 9)).astype(np.int32)
    forced = rng.integers(0, 32000, (12, batch)).astype(np.int32)
    results = []
    for read in (True, False):
        h = fp.fp_create(arch_dict(TINY), 0, 0, batch, 40, seed=11)
        try:
            got = [fp.fp_prefill(h, prompt).copy()]
            for i, t in enumerate(forced):  # unread: only the last step waits
                out = fp.fp_decode_step(h, t, want_out=read or i == len(forced) - 1)
            got.append(out.copy())
            for _ in range(3):  # greedy steps: their own tokens
                got.append(fp.fp_decode_step(h, None, batch=batch).copy())
            fp.fp_decode_steps(h, 2)
            got.append(fp.fp_decode_step(h, got[0], batch=batch).copy())
            got.append(fp.fp_get_tensor(h, fp.FP_G_TOKENS, dtype=np.int32).copy())
            got.append(fp.fp_get_tensor(h, fp.FP_G_LOGITS, dtype=np.float32).copy())
        finally:
            fp.fp_destroy(h)
        results.append(got)
    for a, b in zip(*results):
        assert np.array_equal(a, b)
    assert np.array_equal(results[0][-2], results[0][-3])
    logits = results[0][-1].reshape(batch, -1)
    assert np.array_equal(results[0][-2], logits.argmax(1))

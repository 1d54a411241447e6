"""What fm_generate counts: passes behind the end are neither launched nor in the accept lengths."""
import numpy as np
import pytest

import fm_synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("faces,keep,eos", [(2, 3, 0), (3, 1, 0), (2, 3, 1)])
def test_nothing_is_launched_behind_the_end(faces, keep, eos):
    from paper_2511_15618_b200 import FlashMesh
    cfg = S.get_config("tiny").with_(allow_eos=eos)
    dev = FlashMesh(cfg, S.make_weights(cfg))
    cond, D = np.stack([S.make_condition(cfg)]), cfg.draft_len

    def run(**kw):
        dev.prefill(cond, [[]])
        l0 = dev.launch_count()
        tok, ln, st = dev.generate(faces, **kw)
        return tok, int(ln[0]), st, dev.launch_count() - l0

    tok, n, _, _ = run(plain=True)
    truth = tok[:, :n].contiguous()
    sched = np.full((1, 1), keep, np.int32)
    passes = -(-n // (keep + 1))
    _, m, st, launches = run(truth=truth, keep=sched)
    assert m == n == st.emitted and sum(st.accept_hist) == passes and st.steps == -(-passes // 8) * 8
    assert st.mean_accept_len == n / passes
    one, two, exact = (run(truth=truth, keep=sched, max_steps=k) for k in (1, 2, passes))
    assert exact[1] == n and exact[2].steps == passes
    # the loop notices the end up to two passes late; whole passes are all it launches
    assert (launches - exact[3]) % (two[3] - one[3]) == 0 and launches - exact[3] <= 2 * (two[3] - one[3])

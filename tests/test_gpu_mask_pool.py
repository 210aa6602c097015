"""The memory pool of the masks: what it holds goes back to the device with the last handle, whichever that is."""
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

PROGRAM = """
import torch
import paper_2303_10837_b200 as he
import synthetic_inputs as si

def cycle(score, mask_last):
    ctx = he.he_ctx_create(8192, list(si.PRIMES_N8192), 40)
    masks = [he.he_select_mask(ctx, score, score.numel() // 10) for _ in range(2)]
    inside = torch.cuda.mem_get_info()[0]
    del masks[0]
    if mask_last:
        del ctx
        mask = masks.pop()
        assert he.he_mask_indices(mask).numel() == mask.k
        del mask
    else:
        masks.clear()
        del ctx
    torch.cuda.synchronize()
    return inside

score = torch.rand(60_000_000, device="cuda")
cycle(score[:1000], False)                      # loads the library's device code
for mask_last in (False, True, False):
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    inside = cycle(score, mask_last)
    torch.cuda.empty_cache()
    after = torch.cuda.mem_get_info()[0]
    assert before - inside > 70 << 20, (before, inside)
    # the figures are the device's, so other programs move them a little; the pool would hold all of what was used inside
    assert before - after < 8 << 20, (mask_last, before, after)
print("ok")
"""


def test_the_pool_is_given_back_with_the_last_handle():
    run = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0 and run.stdout.strip().endswith("ok"), run.stdout[-2000:] + run.stderr[-3000:]

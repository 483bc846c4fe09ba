"""The attention kernel's bounded waits on grids of more than one wave: two tiles per CTA (adjacent ones, and the same rows of
two heads), and later CTAs that find the status record set and leave with only their first copies to wait for."""
import pytest
import torch

from paper_2608_17336_b200 import synth
from tests import helpers as H
from tests.test_gpu_timeout import drop  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("Hk,d", [(80, 128), (20, 128), (80, 64)])
def test_wait_runs_out_with_two_tiles_per_cta(drop, Hk, d):  # noqa: F811
    from paper_2608_17336_b200 import binding as tm
    w = synth.Workload("timeout", 1, 80, 700, d, d, 1, seed=92, routing="bernoulli", int8_fraction=0.5)
    q, k, v = (t.to(DEV) for t in synth.make_qkv(w))
    k, v = k[:, :Hk].contiguous(), v[:, :Hk].contiguous()
    route = torch.from_numpy(synth.make_route(w)).to(DEV)[:, :Hk].contiguous()
    p = tm.problem(1, 80, Hk, 700, d, d, d, 1)
    codes = tm.tilemix_quantize_qk(p, q, k)
    words, _ = tm.tilemix_pack_routing_mask(p, route, False)
    good = tm.tilemix_attention_fwd(p, q, k, v, *codes, words)
    assert tm.tilemix_read_status(good["workspace"])[0] == 0
    drop(1, 2_000_000)
    bad = tm.tilemix_attention_fwd(p, q, k, v, *codes, words, workspace=good["workspace"])
    assert tm.tilemix_read_status(bad["workspace"])[0] == tm.ERR_DEVICE_TIMEOUT
    drop(0)
    again = tm.tilemix_attention_fwd(p, q, k, v, *codes, words, workspace=good["workspace"])
    assert tm.tilemix_read_status(again["workspace"])[0] == 0
    assert torch.equal(again["out"], good["out"])

"""The backward at sides above 32, whose CTAs wait for one another, on a stream that has a part of the device's SMs only: fewer and smaller gangs,
the same gradients."""
import pytest
import torch

import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.workloads import make_inputs, small_config

pytestmark = pytest.mark.gpu
driver = pytest.importorskip("cuda.bindings.driver")

CASES = [(1, 70, 130, 2, 64, 64, 32, 32, 0, 1), (3, 35, 140, 7, 64, 40, 20, 20, 0, 1), (1, 128, 128, 1, 128, 128, 64, 0, 0, 1)]


def _ok(result):
    assert result[0] == driver.CUresult.CUDA_SUCCESS, result[0]
    return result[1] if len(result) == 2 else result[1:]


@pytest.fixture(params=[8, 72], scope="module")
def partition(request):
    torch.cuda.init()
    torch.zeros(1, device="cuda")
    device = _ok(driver.cuDeviceGet(torch.cuda.current_device()))
    sms = _ok(driver.cuDeviceGetDevResource(device, driver.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    groups, _, _ = _ok(driver.cuDevSmResourceSplitByCount(1, sms, 0, request.param))
    desc = _ok(driver.cuDevResourceGenerateDesc(groups, 1))
    context = _ok(driver.cuGreenCtxCreate(desc, device, driver.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    stream = _ok(driver.cuGreenCtxStreamCreate(context, driver.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))
    yield torch.cuda.ExternalStream(int(stream))
    torch.cuda.synchronize()
    driver.cuStreamDestroy(stream)
    driver.cuGreenCtxDestroy(context)


@pytest.mark.parametrize("case", CASES, ids=["_".join(map(str, c)) for c in CASES])
def test_backward_on_a_part_of_the_device(case, partition):
    cfg = small_config("partition", *case)
    x = {k: v.cuda() for k, v in make_inputs(cfg).items()}
    d = terra.make_desc(cfg)
    o, lse = terra.terra_swin_attn_fwd(d, x["q"], x["k"], x["v"], x["bias"])
    ref = terra.terra_swin_attn_bwd(d, x["q"], x["k"], x["v"], x["bias"], o, lse, x["do"])
    torch.cuda.synchronize()
    with torch.cuda.stream(partition):
        o2, _ = terra.terra_swin_attn_fwd(d, x["q"], x["k"], x["v"], x["bias"])
        got = terra.terra_swin_attn_bwd(d, x["q"], x["k"], x["v"], x["bias"], o, lse, x["do"])
    partition.synchronize()
    terra.terra_swin_check()
    assert torch.equal(o, o2)
    # Where CTAs no longer start at different chunks of the queries, all sums have another order: 32-bit sums, of which dQ, dK and dV are then rounded
    # to the 8 bits of bf16 (a sum that lies near the middle of two may go to the other one: at most 2^-8 of it)
    for a, b, tol in zip(got, ref, (4e-3, 4e-3, 4e-3, 1e-5)):
        assert (a.double() - b.double()).norm() <= tol * b.double().norm()

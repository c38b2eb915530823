"""The stencil gradient's blocks take equal shares of the units and stay for the whole call: there are as many as are
resident at once, no more (a second, partial wave of them would double the call). A block writes its sums to a
column of its own of the workspace, so that the columns that a call on one level writes are its blocks."""
import numpy as np
import pytest
import torch

import aprsynth as S
import paper_2112_03592_gb300 as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,resident", [(3, 2), (5, 3)])
def test_one_wave_of_blocks(k, resident):
    apr = S.uniform_level_apr((120, 128, 128), 7, l_min=7)      # 480 work items, 960 units
    lay = G.AprLayout.from_apr(apr, G.APR_VALIDATE | G.APR_REQUIRE_BALANCE)
    v = torch.as_tensor(apr.values, device="cuda")
    tree = torch.empty(0, device="cuda")
    g = torch.ones_like(v)
    ws = torch.full((int(lay._lib.apr_stencil_grad_workspace_bytes(lay.handle, k)) // 4,), float("nan"), device="cuda")
    gw = torch.empty(k ** 3, device="cuda")
    assert lay._lib.apr_convolve_stencil_grad(lay.handle, v.data_ptr(), tree.data_ptr(), k, G.APR_BC_REFLECT, g.data_ptr(), gw.data_ptr(),
                                              ws.data_ptr(), 4 * ws.numel(), G._stream_ptr()) == 0
    items = len(lay.export(4))
    written = ws[:k ** 3 * items].view(k ** 3, items).isfinite()
    assert torch.equal(written.all(0), written.any(0))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert int(written.any(0).sum()) == min(resident * sms, items)
    assert abs(float(gw[k ** 3 // 2]) - float(v.double().sum())) <= 1e-5 * float(v.double().abs().sum())

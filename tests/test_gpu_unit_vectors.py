"""GPU check of the node build's column parts and of the unit vectors' launch through whole
networks: widths below and above a part, of no whole parts, many
rows, and output vectors off 16-byte boundaries."""
import ctypes

import numpy as np
import pytest
import torch

import workloads
from test_gpu_fused import _ll, _oracle_check, _topk
from _helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,K,D,shift", [(1, 2, 3, 64, 0), (1, 5, 4, 320, 0), (2, 3, 2, 1024, 0),
                                           (40, 8, 2, 512, 0), (1, 4, 4, 512, 1)])
def test_columns_and_alignment(B, L, K, D, shift):
    ll = _ll()
    wl = workloads.Workload(f"unit_b{B}_d{D}", B=B, L=L, V=500, K=K, d=D, H=64, dtype="bf16",
                            logit_kind="normal_planted", logit_param=(3.0, 8.0), seed_base=9700 + D)
    W = workloads.head_weights(wl)
    inp = workloads.batch_inputs(wl, wl.seeds())
    ids, logp = _topk(wl, inp["logits"])
    head = ll.Head.from_workload(wl, W, workloads.embed_table(wl.V, wl.H, wl.dtype))
    try:
        i32, lp = to_dev(ids.astype(np.int32), "f32"), to_dev(logp.astype(np.float32), "f32")
        hid, tgt = to_dev(inp["hidden"], wl.dtype), to_dev(inp["target"], wl.dtype)
        n = B * L * K * D
        buf = torch.zeros(2 * n + B * D + 16, device="cuda")
        out, inn, anc = buf[shift:], buf[n + shift:], buf[2 * n + shift:]
        ws = head.workspace(B)
        st = ll.lib().lilicorr_embed_in_out(head._h, B, i32.data_ptr(), lp.data_ptr(),
                                            hid.data_ptr(), tgt.data_ptr(), out.data_ptr(),
                                            inn.data_ptr(), anc.data_ptr(), ws.ptr, ws.nbytes,
                                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == 0
        torch.cuda.synchronize()
        shape = (B, L, K, D)
        res = [x.cpu().numpy() for x in (out[:n].view(shape), inn[:n].view(shape),
                                         anc[:B * D].view(B, D))]
        assert np.allclose(np.linalg.norm(res[0], axis=-1), 1, atol=1e-5)
        _oracle_check(wl, W, inp, ids, logp, *res, range(min(B, 3)))
    finally:
        head.close()

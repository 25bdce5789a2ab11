"""Two host threads call one kernel at sizes that take different amounts of
shared memory, each on its own stream: every call launches, and the results are
those of the calls made alone.  (The limit belongs to the kernel: set to what one
launch takes, it fails the other thread's larger launch.)"""
import threading

import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import _lib, inputs

pytestmark = pytest.mark.gpu

F32, BF16, FP8 = _lib.ET_F32, _lib.ET_BF16, _lib.ET_FP8
CALLS = 1500


def _in_threads(calls):
    """calls: one function per thread, each made CALLS times."""
    errors = []

    def work(fn):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(CALLS):
                    fn()
                torch.cuda.current_stream().synchronize()
        except Exception as e:      # noqa: BLE001 -- reported below
            errors.append(e)

    threads = [threading.Thread(target=work, args=(fn,)) for fn in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


@pytest.mark.parametrize("dtype,C,forms", [
    (F32, 20, [(0, 2, 1, 3), (0, 4, 1, 3)]),      # evsnet.cu
    (F32, 8, [(1, 3, 3, 1), (1, 7, 9, 1)]),       # evsnet_pix.cu
    (FP8, 16, [(0, 2, 1, 3), (0, 4, 1, 3)]),      # evsnet_tc.cu, 16 channels
    (BF16, 32, [(0, 2, 1, 3), (0, 3, 1, 3)]),     # evsnet_tc.cu, 32 channels
])
def test_forward_in_two_threads(dtype, C, forms):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import api
    H, W = 5, 9
    calls, checks = [], []
    for kind, L, kt, ks in forms:
        net = api.EvsNetDev.from_dict(inputs.random_evsnet(kind, L, C, kt, ks, seed=L, vth=0.3, beta=0.9), dtype)
        lf = torch.as_tensor(inputs.random_logl_clip(L, 2, H, W, step_std=0.4)).cuda()
        st, buf = api.EvsStateDev(net, H, W), api.EventBuffer(4 * H * W)

        def call(net=net, lf=lf, st=st, buf=buf):
            st.initialized = 0
            return api.evsnet_forward(lf, net, st, buf=buf, want_I=True)[1]

        zero = (st.V.clone(), st.hist.clone())
        ref = call().clone()
        st.V.copy_(zero[0])
        st.hist.copy_(zero[1])
        calls.append(call)
        checks.append((call, st, zero, ref))
    torch.cuda.synchronize()
    _in_threads(calls)
    torch.cuda.synchronize()
    for call, st, zero, ref in checks:
        st.V.copy_(zero[0])
        st.hist.copy_(zero[1])
        assert torch.equal(call(), ref)


def test_bf16_training_in_two_threads():
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import api, training as tr
    calls, refs = [], []
    for kt in (1, 7):                             # train_tct.cu below 16 channels
        meta = api.EvsNetDev.from_dict(inputs.random_evsnet(0, 2, 8, kt, 1, seed=kt, vth=0.3, beta=0.9), BF16)
        lf = torch.as_tensor(np.stack([inputs.random_logl_clip(kt, 4, 5, 9, step_std=0.4)])).cuda()
        ws = tr.Workspace()
        ws.get(meta, meta.w, meta.b, tr.L.et_train_shape(1, 3, 5, 9, 4))

        def call(meta=meta, lf=lf, ws=ws):
            lib, C = _lib.load(), tr.C
            sh = tr.L.et_train_shape(1, 3, 5, 9, 4)
            I = torch.empty((1, 3, 5, 9), device="cuda")
            spikes = torch.empty((1, 3, 5, 9), dtype=torch.int8, device="cuda")
            V = torch.empty((1, 1, 5, 9), device="cuda")
            rc = lib.et_evsnet_train_forward(lf.data_ptr(), C.byref(sh), C.byref(tr._net_struct(meta, meta.w, meta.b)),
                                             spikes.data_ptr(), None, None, V.data_ptr(), I.data_ptr(),
                                             ws.buf.data_ptr(), ws.buf.numel(),
                                             torch.cuda.current_stream().cuda_stream)
            _lib.check("et_evsnet_train_forward", rc)
            return I

        refs.append(call().clone())
        calls.append(call)
    torch.cuda.synchronize()
    _in_threads(calls)
    torch.cuda.synchronize()
    for call, ref in zip(calls, refs):
        assert torch.equal(call(), ref)

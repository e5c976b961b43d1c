"""Prediction on device rows as part of a caller's own CUDA graph: a captured call (also a context's first
prediction) is accepted, and a replay predicts with the parameters as they are by then, whether they were set,
drawn anew or trained since.  Same kernel on the same operands: the same bits as an ordinary call."""
import numpy as np
import pytest

from paper_2509_24742_gb300 import srbe

pytestmark = pytest.mark.gpu


def test_captured_prediction_follows_the_parameters():
    import torch
    rng = np.random.default_rng(2)
    D = torch.from_numpy(rng.gamma(2.0, 0.15, (333, srbe.N_DESC)).astype(np.float32)).cuda()
    out, ref = (torch.empty(D.shape[0], dtype=torch.float32, device="cuda") for _ in range(2))
    st = torch.cuda.Stream()
    with srbe.Context((2.0, 2.0, 12.0), 3.5, 0.05, 1.2, 10, 2) as c:
        c.set_stream(st.cuda_stream)
        c.mlp_init(seed=1)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            c.mlp_predict_dev(D.data_ptr(), D.shape[0], out.data_ptr())
        P = c.mlp_params()
        seen = []
        for change in (lambda: None, lambda: c.mlp_init(seed=2), lambda: c.mlp_set_params(P * 1.5),
                       lambda: c.mlp_train(D.cpu().numpy(), np.linspace(0, 1, 333, dtype=np.float32), epochs=2,
                                           batch=64, lr=1e-3, seed=3)):
            change()
            with torch.cuda.stream(st):
                out.fill_(0)
                g.replay()
            st.synchronize()
            got = out.cpu().numpy()
            c.mlp_predict_dev(D.data_ptr(), D.shape[0], ref.data_ptr())
            st.synchronize()
            assert np.array_equal(got, ref.cpu().numpy())
            assert all(not np.array_equal(got, s) for s in seen)
            seen.append(got)

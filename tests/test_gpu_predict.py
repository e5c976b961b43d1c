"""The network's calls in a caller's own CUDA graph and from several threads.  Same kernels on the same operands
as an ordinary call: the same bits."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2509_24742_gb300 import srbe

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_captured_prediction_follows_the_parameters():
    """A captured prediction (also a context's first one) is accepted, and a replay predicts with the parameters
    as they are by then, whether they were set, drawn anew or trained since."""
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


FIRST_CALLS = """
import sys, threading, time
import numpy as np
from paper_2509_24742_gb300 import srbe
train = sys.argv[1] == "train"
ctxs = [srbe.Context((2.0, 2.0, 12.0), 3.5, 0.05, 1.2, 10, 2) for _ in range(12)]
D = np.random.default_rng(0).gamma(2.0, 0.15, (700, srbe.N_DESC)).astype(np.float32)
out, errors, start = [None] * len(ctxs), [], threading.Barrier(len(ctxs))
for c in ctxs:
    c.mlp_init(seed=1)
def work(i):
    try:
        start.wait()
        time.sleep(5e-5 * i)
        out[i] = ctxs[i].mlp_gradients(D, D[:, 0])[0] if train else ctxs[i].mlp_predict(D)
    except Exception as e:
        errors.append(repr(e))
threads = [threading.Thread(target=work, args=(i,)) for i in range(len(ctxs))]
[t.start() for t in threads]
[t.join() for t in threads]
assert not errors, errors
assert all(np.array_equal(o, out[0]) for o in out)
"""


@pytest.mark.parametrize("what", ["predict", "train"])
def test_first_calls_of_several_threads(what):
    """A process's first predictions (gradients), by twelve threads at once: none launches a kernel whose
    shared-memory limit another thread is still setting."""
    r = subprocess.run([sys.executable, "-c", FIRST_CALLS, what], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]

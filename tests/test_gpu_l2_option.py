"""TURSCA_OPT_L2_RESIDENT sets its access-policy window on the scene's stream for
a solve inside tursca_run as it does for tursca_solve: a thread that reads the
stream's attribute meanwhile sees it, and afterwards it is gone."""
import ctypes as C
import threading

import numpy as np
import pytest

from paper_2503_16037_gb300 import scenes
from paper_2503_16037_gb300 import tursca as T

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ACCESS_POLICY_WINDOW = 1  # cudaLaunchAttributeAccessPolicyWindow; num_bytes is the value's second 8 bytes


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_16037_gb300 import build
    build.build()


@pytest.mark.parametrize("whole", [True, False])
def test_the_window_is_set_while_a_solve_runs(whole):
    T.lib()
    rt = C.CDLL("libcudart.so.13")
    stream = torch.cuda.Stream()

    def window():
        value = (C.c_uint64 * 8)()
        assert rt.cudaStreamGetAttribute(C.c_void_p(stream.cuda_stream), ACCESS_POLICY_WINDOW, C.byref(value)) == 0
        return value[1]

    with torch.cuda.stream(stream):
        rn = T.Runner(scenes.make_plume(nx=32, ny=32, nz=24), T.FP32_REFINE, stream=stream)
        mu_a, mu_s = rn.fields("cuda")
        ref = rn.run(mu_a, mu_s)[0].clone()
        T.tursca_set_option(rn.handle, T.OPT_L2_RESIDENT, 1)
        seen, stop = [], threading.Event()

        def watch():
            while not stop.is_set():
                if window():
                    seen.append(True)

        th = threading.Thread(target=watch)
        th.start()
        try:
            for _ in range(200):
                if whole:
                    rad = rn.run(mu_a, mu_s)[0]
                else:
                    rn.set_medium(mu_a, mu_s)
                    rn.assemble()
                    rn.solve()
                    rad = rn.render()[0]
        finally:
            stop.set()
            th.join()
        assert seen and window() == 0
        stream.synchronize()
        assert np.array_equal(ref.cpu().numpy(), rad.cpu().numpy())  # where K is read changes, no bit does
        rn.close()

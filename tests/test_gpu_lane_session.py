"""Circuits of small states applied while another thread starts and stops
serving sessions: every result is right, whichever pass each call took, and the
cluster pass is back once no session is live."""
import threading

import numpy as np
import pytest

import oracle
import paper_2608_09733_gb300 as sv
from paper_2608_09733_gb300.binding import SmallSession, SvError
from workloads import serving_circuit

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_sessions_start_between_plan_and_launch(svlib, cuda_dev):
    n, circ = 12, serving_circuit(12, 6, 1)
    ref = oracle.run(n, circ)
    gates = sv.Gates(circ)
    errors = []

    def sessions():
        try:
            for _ in range(20):
                s = SmallSession(sv.SV_C64, wait_limit_s=0.01)
                try:
                    s.stop()
                except SvError:
                    pass  # it sat idle
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            errors.append(e)

    t = threading.Thread(target=sessions)
    t.start()
    st = torch.empty(2 ** n, dtype=torch.complex64, device="cuda")
    runs = 0
    while t.is_alive() or runs < 50:
        sv.sv_init_basis(st, 0)
        sv.sv_apply_circuit(st, gates)
        assert np.abs(st.cpu().numpy() - ref).max() < 1e-5  # the state tolerance of the other parity tests
        runs += 1
    t.join()
    assert not errors
    sv.sv_profile_enable(True)
    sv.sv_apply_circuit(st, gates)
    torch.cuda.synchronize()
    fam = set(sv.sv_profile_read())
    sv.sv_profile_enable(False)
    assert fam == {"sweep_lane"}

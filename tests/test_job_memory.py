"""Device memory of a job (nne_job_bytes: the state's and its workspaces' allocation plan)
against an earlier plan of the library.  A server or context with a memory budget
admits what fits in it, so a workspace that grows refuses jobs that used to run."""
import numpy as np
import pytest

from paper_2501_13237_gb300 import nne


# dtype, qubits, bond, levels, bytes; exact truncation, one gate, ten observables
@pytest.mark.parametrize("dtype,n,chi,levels,most", [
    (0, 2, 1, 1, 620032), (0, 8, 16, 4, 6333696), (0, 8, 24, 8, 19045888), (0, 12, 40, 4, 19596800),
    (0, 12, 41, 4, 20353280), (0, 16, 64, 8, 83505664), (0, 16, 128, 4, 136744704), (0, 40, 512, 8, 5272381696),
    (0, 40, 4096, 1, 39462912256),
    (1, 2, 1, 1, 1191936), (1, 8, 16, 4, 11242752), (1, 8, 24, 8, 32079360), (1, 12, 40, 4, 31124992),
    (1, 12, 41, 4, 32213248), (1, 16, 64, 8, 126308864), (1, 16, 128, 4, 192936704), (1, 40, 512, 8, 7979094272),
    (1, 40, 4096, 1, 58450701568),
])
def test_job_memory_does_not_grow(dtype, n, chi, levels, most):
    job = nne.Job(n, [([0], np.eye(4, dtype=complex)[None], 1)], np.arange(1.0, levels + 1), np.zeros((levels, 4)), chi,
                  np.zeros((10, n), np.uint8), dtype=dtype)
    assert 0 < job.bytes() <= most

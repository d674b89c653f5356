"""Device memory of a shell-pair handle: a precision's copies of the Hermite
coefficients are held only by handles that read them."""
import pytest

import molgen

pytestmark = pytest.mark.gpu


def test_copies_of_the_coefficients():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required")
    import paper_2407_21445_gb300 as fk
    p = molgen.problem(2)

    def held(**kw):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        b = fk.JKBuilder(p.basis, p.tau, fk.make_opts(**kw))
        torch.cuda.synchronize()
        n = free - torch.cuda.mem_get_info()[0]
        b.close()
        return n

    held()  # tables, streams, kernels
    off, fp64, mixed = held(two_float=False), held(), held(precision=fk.FOCK_MIXED)
    ff = fp64 - off  # 8 bytes per coefficient and 16 per primitive pair
    assert ff > 16 << 20
    assert 0.3 * ff < mixed - fp64 < 0.6 * ff  # 4 bytes per coefficient, for the FP32 path alone

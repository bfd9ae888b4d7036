"""The network's loss is a 64-bit sum: as many bits as FP64 sums of its terms keep."""
from fractions import Fraction

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


# With all parameters 0 the outputs are 0 and the value loss is the mean square of the
# targets.  Every thread of the loss kernel sees the same 16 targets (rows 16 apart, four
# columns), so that its rounding does not average out, and each draw is one on which sums
# of 48 bits are 60 to 120 units of 2^-53 off.  Allowed: one unit for each FP64 operation
# on the way of a term, 3 to join a thread's words, 10 in the block, 1 division, 11 in the
# sum over blocks.
@pytest.mark.parametrize("m", [128, 384])
@pytest.mark.parametrize("seed", [4, 34])
def test_value_loss(m, seed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1307_3424_gb300 import wproj
    net = wproj.MLP(torch.zeros(int(wproj.lib().wproj_mlp_num_params())))
    pat = np.random.default_rng(seed).uniform(0.5, 1.5, 16).astype(np.float32)
    tv = pat.reshape(4, 4)[(np.arange(m)[:, None] // 16) % 4, np.arange(2048)[None, :] % 4]
    loss, _ = net.gradients(torch.zeros(m, 3, device="cuda"), torch.from_numpy(np.ascontiguousarray(tv)).cuda(),
                            torch.zeros(m, 1024, device="cuda"), mask_weight=0.0)
    want = sum(Fraction(float(v)) ** 2 for v in pat) / 16
    assert abs(Fraction(loss) - want) <= 25 * want / 2 ** 53
    net.close()

"""GPU parity of the tensor-core scorer at head size 64 (one half of 64 channels per tile, a deeper key ring): one and two
row blocks, ragged tails, several items per CTA, sequences of different lengths."""
import pytest
import torch

from gpu_helpers import assert_scores_close, bits, gpu_score
from paper_2602_08585_b200 import lukv
from test_gpu_parity import _rand_qkv
from test_gpu_ragged import _case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,L,H,G,T,w,kp", [(1, 1, 1, 1, 129, 1, 1), (1, 1, 2, 4, 1300, 32, 7), (2, 1, 1, 7, 1111, 32, 5),
                                            (1, 1, 1, 4, 2048, 64, 7), (1, 4, 8, 2, 9000, 16, 3)])
def test_score_head64(oracle, S, L, H, G, T, w, kp):
    q, k, _ = _rand_qkv(S, L, H, G, 64, T, w, torch.bfloat16, seed=T + w, scale=2.0)
    p = lukv.make_params(S, L, H, G, 64, T, w, kp, torch.bfloat16, 2)
    assert_scores_close(gpu_score(p, q.cuda(), k.cuda()).cpu().numpy(), oracle.score(bits(q), bits(k), G, kp))


@pytest.mark.parametrize("G,w", [(4, 32), (8, 32)])
def test_ragged_head64(oracle, G, w):
    _case(oracle, 3, 1, 2, G, 64, 2048, w, 5, 17, torch.bfloat16, [2048, 640, 1216], [0.3, 0.1], seed=G, n_sink=4,
          min_keep=0.02)

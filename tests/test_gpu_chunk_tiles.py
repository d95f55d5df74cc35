"""GPU parity of chunked prefill, chunk-end and streaming, at the edges of the d = 64 / 32 prefill kernel's 96-key tiles: pools and window spans of one
and two tiles and a key more or less, chunks around an item of 128 queries and around a tile, and logits so wide that the reference moves
and the accumulator is rescaled, between tiles and under the streaming reading's leave times."""
import pytest

from tests.test_gpu_chunk import _cfg, _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,W,R,T0,Tc", [
    (64, 65, 95, 500, 128), (64, 66, 96, 520, 129), (64, 64, 97, 560, 127), (64, 33, 192, 700, 96), (64, 96, 97, 600, 95),
    (32, 65, 193, 760, 97), (32, 97, 96, 600, 1),
])
@pytest.mark.parametrize("scale", [0.0, 4.0])                     # logits of N(0,1) / d^(1/2) and of N(0,16)
@pytest.mark.parametrize("streaming", [False, True])
def test_chunks_at_tiles_of_96(d, W, R, T0, Tc, scale, streaming):
    _compare(_cfg(B=1, H=2, d=d, W=W, R=R), [("prefill", T0), ("chunk", Tc), ("decode", 2)], seed=6, scale=scale, streaming=streaming)

"""The native argument marshalling behind the per-step calls refuses wrong arguments on the host."""
import pytest
import torch

from paper_2511_22481_b200 import binding as B
from paper_2511_22481_b200 import build as builder


@pytest.fixture(scope="module", autouse=True)
def built():
    builder.build()


def _desc():
    return B.make_desc(1, 16, 4, 4, 64, 0.1)


def test_dtype_device_and_kind_are_checked():
    f32, bf16, i32 = torch.zeros(4), torch.zeros(4, dtype=torch.bfloat16), torch.zeros(4, dtype=torch.int32)
    with pytest.raises(TypeError, match=r"q must be torch.bfloat16, got torch.float32"):
        B.omni_sparse_mla_decode(_desc(), f32, bf16, i32, i32, i32, bf16, f32)
    with pytest.raises(ValueError, match="q must live on cuda"):
        B.omni_sparse_mla_decode(_desc(), bf16, bf16, i32, i32, i32, bf16, f32)
    with pytest.raises(TypeError, match="q must be a tensor"):
        B.omni_sparse_mla_decode(_desc(), 3, bf16, i32, i32, i32, bf16, f32)
    with pytest.raises(TypeError):
        B.omni_sparse_mla_decode(None, bf16, bf16, i32, i32, i32, bf16, f32)
    with pytest.raises(TypeError, match="desc must be an OmniDesc"):
        B.omni_sparse_mla_decode(b"short", bf16, bf16, i32, i32, i32, bf16, f32)
    with pytest.raises(ValueError, match="q_host must be contiguous"):
        B.omni_sparse_mla_decode_host(_desc(), torch.zeros(4, 4, dtype=torch.bfloat16).t(), None, i32, i32, i32, bf16, f32, bf16)


class _Stream:
    cuda_stream = 0


def test_status_codes_become_exceptions():
    """With a stream given, nothing asks the device: the library's own null check answers."""
    for call in (lambda: B.omni_sparse_mla_decode(_desc(), *([None] * 7), stream=_Stream()),
                 lambda: B.omni_sparse_mla_decode_sink_recent(_desc(), None, None, None, None, 64, 64, None, None, stream=_Stream()),
                 lambda: B.omni_kv_append_rolling(_desc(), None, None, None, None, 64, 64, stream=_Stream())):
        with pytest.raises(B.OmniError) as e:
            call()
        assert e.value.code == 1

"""Which tensors ``iconv_plan_stack`` refuses to run a stack of layers on: the addresses alone decide, no GPU is touched."""
import numpy as np
import pytest

from paper_2006_11735_b200 import binding as B

A, C, D = 0x7F0000000000, 0x7F0000100000, 0x7F0000200000        # tensors far apart


def _layer(k=1, c=64, c_out=None, **kw):
    c_out = c if c_out is None else c_out
    return dict(n=2, h=16, w=16, c_in=c, c_out=c_out, kh=k, kw=k, pad=k // 2, weights=np.ones((c_out, k, k, c), np.int8),
                bias=np.zeros(c_out, np.int32), mul=[200], shift=[16], h_i=[83558], **kw)


def _refusal(layers):
    """The reason why these layers' tensors are refused, or None (planning them then goes on to the device)."""
    try:
        B.iconv_stack_destroy(B.iconv_plan_stack(layers))
    except B.IconvError as e:
        text = str(e)
        if "another layer's output" in text or "writes a tensor" in text:
            assert e.status == B.ERR_UNSUPPORTED
            return text
    return None


WIDE = dict(in_c_total=128, out_c_total=128)
READS, WRITES = "reads part of another layer's output", "writes a tensor"


@pytest.mark.parametrize("layers,why", [
    ([(_layer(), A, C), (_layer(), C, D)], None),
    ([(_layer(), A, C), (_layer(), C + 1024, D)], READS),                       # from the second image row on
    ([(_layer(), A, C), (_layer(), C - 1024, D)], READS),
    ([(_layer(**WIDE), A, C), (_layer(**WIDE), C + 64, D)], None),              # the wide tensor's other half, by its address
    ([(_layer(**WIDE), A, C), (_layer(**WIDE), C + 48, D)], READS),             # sixteen of its channels
    ([(_layer(**WIDE), A, C), (_layer(in_c_total=64), C + 128, D)], READS),     # of another stride
    ([(_layer(), A, C), (_layer(), C, A + 64)], WRITES),                        # overwrites the first layer's input
    ([(_layer(), A, C), (_layer(), C, C + 2048)], WRITES),                      # ... and its output
    ([(_layer(), A, C), (_layer(), C, C + 2 * 16 * 16 * 64)], None),            # right behind it
    ([(_layer(), A, A + 4096), (_layer(), A + 4096, D)], WRITES),               # the first layer into its own input
    ([(_layer(**WIDE), A, A + 64), (_layer(**WIDE), A + 64, D)], None),         # into the channels that it does not read
    ([(_layer(), A, C), (_layer(skip_dtype=B.U8, skip_c_total=64, skip_shift=8), C, D, C + 64)], READS),
    ([(_layer(skip_dtype=B.U8, skip_c_total=64, skip_shift=8), A, C, D), (_layer(), C, D + 128)], WRITES),
], ids=lambda v: "" if isinstance(v, list) else None)
@pytest.mark.parametrize("k", [1, 3], ids=["flow", "equal_layers"])
def test_layers_of_a_stack_do_not_share_memory_but_by_their_slices(layers, why, k):
    layers = [(dict(e[0], kh=k, kw=k, pad=k // 2, weights=np.ones((e[0]["c_out"], k, k, e[0]["c_in"]), np.int8)),) + e[1:] for e in layers]
    got = _refusal(layers)
    assert (got is None) if why is None else (got is not None and why in got), got


@pytest.mark.parametrize("k", [1, 3])
def test_an_empty_batch_without_tensors_is_left_to_single_launches(k):
    """Its tensors have no address: no argument error, the caller runs the layers apart."""
    empty = dict(_layer(k), n=0)
    with pytest.raises(B.IconvError) as e:
        B.iconv_plan_stack([(empty, 0, 0), (empty, 0, 0)])
    assert e.value.status == B.ERR_UNSUPPORTED and e.value.layer is None
    with pytest.raises(B.IconvError) as e:
        B.iconv_plan_stack([(_layer(k), 0, C), (_layer(k), C, D)])
    assert e.value.status == B.ERR_ARG

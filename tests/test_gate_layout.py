"""How the columns of a token row lie in shared memory between the router GEMM and the row-per-warp selection:
a column is read where it was stored, no two columns share a word and no word lies outside the row, for every
gate the library accepts.  Host arithmetic that the kernels share; nothing is launched."""
import ctypes

import pytest

from paper_2608_14205_b200 import binding as B


def _layout(E, gate, n_group, topk_group):
    cfg = B.FbConfig(128, 64, E, 1, 1, gate, n_group, topk_group, 1, 1.0)
    words, stored, read = ctypes.c_int32(), (ctypes.c_int32 * 256)(), (ctypes.c_int32 * 256)()
    assert B.lib().fb_staged_row_layout(ctypes.byref(cfg), ctypes.byref(words), stored, read) == B.FB_OK
    return words.value, list(stored), list(read)


def _gates():
    for E in range(1, 257):
        yield E, 0, 1, 1
        for n_group in range(1, 33):
            if E % n_group == 0:
                for topk_group in {1, min(8, max(1, n_group - 1)), min(8, n_group)}:
                    yield E, 1, n_group, topk_group


def test_columns_of_a_staged_row_for_every_gate():
    for gate in _gates():
        E = gate[0]
        words, stored, read = _layout(*gate)
        padded = (E + 15) // 16 * 16
        assert read[:E] == stored[:E], gate
        assert len(set(stored[:E])) == E, gate
        assert all(0 <= w < words for w in stored[:padded]), gate
        assert not set(stored[:E]) & set(stored[E:padded]), gate
        assert words % 4 == 0 and all(stored[c] % 4 == 0 for c in range(0, padded, 4)), gate     # 16-byte stores


@pytest.mark.parametrize("bad", [dict(E=300), dict(gate=1, n_group=3)])
def test_layout_query_refuses_what_create_refuses(bad):
    base = dict(T_max=128, d=64, E=8, k=2, R=4, gate=0, n_group=1, topk_group=1, renorm=1, route_scale=1.0)
    base.update(bad)
    cfg = B.FbConfig(*[base[f] for f, _ in B.FbConfig._fields_])
    words, table = ctypes.c_int32(), (ctypes.c_int32 * 256)()
    assert B.lib().fb_staged_row_layout(ctypes.byref(cfg), ctypes.byref(words), table, table) == B.FB_ERR_UNSUPPORTED_SHAPE

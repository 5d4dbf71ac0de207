"""The attention kernel's plain rules (csrc/attn_rules.h), compiled for the host."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_08721_gb300", "csrc")


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, lib = d / "rules.cpp", d / "rules.so"
    src.write_text('#include "attn_rules.h"\n'
                   'extern "C" int part_bufs() { return libraspec::kAttnPartBufs; }\n'
                   'extern "C" int buf_free(const int* done, int layer, int chunks) {\n'
                   '  return libraspec::part_buf_free(done, layer, chunks);\n}\n'
                   'extern "C" int part(int tiles, int k, int p) { return libraspec::group_part(tiles, k, p); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    return ctypes.CDLL(str(lib))


def _overwrites(bufs, free, chunks, layers, warps=2):
    """Every interleaving of a CTA's merge warps (claim the next chunk of a layer whose barrier has passed, read it,
    count it done) with its own arrivals at the layers' barriers (arrival `layer` lets layer + 1 write the buffer of
    layer + 1 - bufs, and waits for free(done, layer)): (a read or unclaimed chunk can be overwritten, all layers can
    be reached)."""
    start = (0, 0, (None,) * warps, (0,) * bufs)  # barriers passed, chunks claimed, chunk held by each warp, done
    seen, todo, bad, end = {start}, [start], False, False
    while todo:
        passed, claimed, held, done = todo.pop()
        nxt = []
        for w, u in enumerate(held):
            put = lambda x: held[:w] + (x,) + held[w + 1:]  # noqa: E731
            if u is None and claimed < passed * chunks:
                nxt.append((passed, claimed + 1, put(claimed), done))
            elif u is not None:
                k = u // chunks % bufs
                nxt.append((passed, claimed, put(None), done[:k] + (done[k] + 1,) + done[k + 1:]))
        if passed < layers and free(done, passed):
            old_end = (passed + 2 - bufs) * chunks  # chunks of the layers up to the one overwritten
            bad |= claimed < old_end or any(u is not None and u < old_end for u in held)
            nxt.append((passed + 1, claimed, held, done))
        end |= passed == layers and claimed == layers * chunks and not any(u is not None for u in held)
        todo += [s for s in nxt if s not in seen]
        seen.update(nxt)
    return bad, end


@pytest.mark.parametrize("chunks", [1, 2, 3])
def test_partials_are_not_overwritten_before_they_are_merged(rules, chunks):
    bufs = rules.part_bufs()

    def free(done, layer):
        return bool(rules.buf_free((ctypes.c_int * bufs)(*done), layer, chunks))

    assert _overwrites(bufs, free, chunks, 8) == (False, True)
    # one count over all buffers lets a chunk in hand be overwritten
    assert _overwrites(bufs, lambda done, layer: sum(done) >= (layer + 2 - bufs) * chunks, chunks, 8)[0]


def test_a_cta_without_merge_chunks_never_waits(rules):
    assert all(rules.buf_free((ctypes.c_int * 3)(0, 0, 0), layer, 0) for layer in range(64))


@pytest.mark.parametrize("tiles", [1, 151, 152, 2049, 15_000_000, (1 << 31) // 64])
@pytest.mark.parametrize("p", [1, 2, 7, 152, 192])
def test_the_parts_of_a_row_group_cover_it_evenly(rules, tiles, p):
    p = min(p, tiles)
    assert [rules.part(tiles, k, p) for k in range(p + 1)] == [tiles * k // p for k in range(p + 1)]

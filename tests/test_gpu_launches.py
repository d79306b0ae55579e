"""The edges of the content address's launches: heads per norm-key thread, tree levels at the
edge of a block (which hands its digests to their parent) with several fragments in one
launch, leaves on both sides of the switch from four lanes each to one, and the sizes at which
cm_ingest_render starts its render beside the leaf hash, as the leaves end, or beside it again.
Ids and norm keys equal the oracle's; the merges' bytes
equal those of the separate calls."""
import numpy as np
import pytest
import torch

from parity_util import THETA, empty_out, oracle_fragment

pytestmark = pytest.mark.gpu

cm = pytest.importorskip("paper_2607_01308_gb300")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cm.Context(0, THETA)
    yield c
    c.close()


def _fragment(seed, L, H, T, d):
    g = torch.Generator(device="cuda:0").manual_seed(seed)
    shape = (L, H, T, d)
    return tuple((torch.randn(shape, generator=g, device="cuda:0") * s).to(torch.bfloat16)
                 for s in (0.7 + 0.01 * (seed % 50), 1.0))


# 128 threads to a norm block: H < 32 gives 128 // H tokens of H threads, more heads loop
@pytest.mark.parametrize("H,T", [(1, 127), (1, 129), (3, 42), (3, 43), (12, 10), (12, 11),
                                 (31, 5), (32, 4), (33, 9), (70, 3)])
def test_norm_key_over_head_counts(ctx, H, T):
    K, V = _fragment(H * 100 + T, 2, H, T, 16)
    fid, Q = ctx.fragment_id(K, V)
    ref = oracle_fragment(K, V)
    assert fid == ref.fid and np.array_equal(np.array(Q, dtype=np.uint64), ref.Q)
    # the allocation-free call takes the same launches
    out = torch.zeros(16, dtype=torch.uint8, device="cuda:0")
    key = torch.full((T,), -1, dtype=torch.int64, device="cuda:0")
    cm.cm_fragment_id_static(cm.fragment_from_tensors(K, V), out.data_ptr(), key.data_ptr())
    torch.cuda.synchronize()
    assert bytes(out.cpu().numpy()) == ref.fid
    assert np.array_equal(key.cpu().numpy().view(np.uint64), ref.Q)


# a token is 1 KiB = one leaf here, so T tokens have ceil(T / 16) level-1 nodes
@pytest.mark.parametrize("lengths", [(1, 16, 17), (256, 257, 255), (511, 512, 513), (9600, 128), (9600, 129),
                                     (8191, 1, 8193), (4096, 4097, 300)])
def test_tree_levels_at_block_edges(ctx, lengths):
    frags = [_fragment(7 * T + i, 1, 1, T, 256) for i, T in enumerate(lengths)]
    S = cm.FragmentSet(ctx)
    res = S.ingest_batch(frags)
    assert [fid for fid, _ in res] == [oracle_fragment(K, V).fid for K, V in frags]
    S.close()


# 114,688 bytes a token: 120 MiB at 1,098 tokens, 1,216 leaf blocks (one partial wave) up to
# about 1,389, 272 MiB at 2,487; the re-sent copies reach that, what is rendered does not
@pytest.mark.parametrize("lengths,prior,copies", [
    ((540, 550), 0, ()), ((548, 550), 0, ()), ((690, 690), 0, ()), ((700, 705), 0, ()),
    ((1240, 1246), 0, ()), ((1240, 1247), 0, ()), ((1500, 1500, 1700), 0, ()), ((300, 300), 400, ()),
    ((300, 300), 1900, ()), ((800, 810), 400, ()), ((800, 810), 3100, ()), ((600, 700), 0, (1, 0))])
def test_ingest_render_start_rules_give_the_separate_calls_bytes(ctx, lengths, prior, copies):
    frags = [_fragment(31 * T + i, 28, 8, T, 128) for i, T in enumerate(lengths)]
    frags += [tuple(x.clone() for x in frags[i]) for i in copies]
    old = [_fragment(5, 28, 8, prior, 128)] if prior else []
    total = sum(lengths) + prior
    half = (len(frags) + 1) // 2
    outs = []
    for fused in (True, False):
        A, B = cm.FragmentSet(ctx), cm.FragmentSet(ctx)
        if old:
            A.ingest_batch(old)
        k, v = empty_out(28, 8, total, 128, fill=0x3C3C)
        where = [A.handle] * half + [B.handle] * (len(frags) - half)
        fd = [cm.fragment_from_tensors(K, V) for K, V in frags]
        if fused:
            _, n, order, overlapped = cm.cm_ingest_render(where, fd, A.handle, k.data_ptr(),
                                                          v.data_ptr(), total)
            assert overlapped
        else:
            cm.cm_ingest_many(where, fd)
            A.union(B)
            n, order = A.render(k, v)
        torch.cuda.synchronize()
        assert n == total
        outs.append((order, k.view(torch.int16), v.view(torch.int16)))
        A.close()
        B.close()
    assert outs[0][0] == outs[1][0]
    assert torch.equal(outs[0][1], outs[1][1]) and torch.equal(outs[0][2], outs[1][2])


# planes that are no multiple of a 1 KiB leaf: leaves that run into one or many further
# segments, short last leaves, alone and in one launch with whole ones
@pytest.mark.parametrize("shape", [(2, 1, 1, 16), (40, 1, 1, 16), (9, 1, 3, 32), (3, 3, 11, 16),
                                   (4, 2, 37, 64), (5, 1, 63, 128), (6, 3, 5, 512),
                                   (8, 3, 3201, 64)])
def test_leaves_that_straddle_segments(ctx, shape):
    L, H, T, d = shape
    K, V = _fragment(sum(shape), L, H, T, d)
    whole = _fragment(3, L, H, 1024, d)   # 1024 rows to a head: every plane whole leaves
    # (the last shape has more leaves than are hashed by four lanes each)
    S = cm.FragmentSet(ctx)
    res = S.ingest_batch([(K, V)])
    assert res[0][0] == oracle_fragment(K, V).fid
    both = cm.FragmentSet(ctx)
    res = both.ingest_batch([whole, (K, V)])
    assert [fid for fid, _ in res] == [oracle_fragment(*whole).fid, oracle_fragment(K, V).fid]
    S.close()
    both.close()


# item sizes of the renders' widths (2 KiB, 4 KiB and 16 KiB of rows) at, below and above a
# plane's rows, fewer pairs than warps, and every head_dim, against the oracle
@pytest.mark.parametrize("L,H,d,lengths", [(1, 1, 128, (8, 7)), (1, 2, 128, (9, 64, 65)), (2, 1, 16, (63, 64, 65)),
                                           (1, 1, 512, (1, 2, 3)), (3, 2, 64, (16, 17, 31)), (2, 2, 32, (32, 33, 257)),
                                           (2, 3, 256, (4, 5, 40))])
@pytest.mark.parametrize("warps", [16, 8])
def test_render_items_at_their_edges(ctx, L, H, d, lengths, warps):
    import oracle
    import synthetic
    from parity_util import assert_k_parity
    frags = [_fragment(17 * T + i, L, H, T, d) for i, T in enumerate(lengths)]
    S = cm.FragmentSet(ctx)
    S.ingest_batch(frags)
    k, v = empty_out(L, H, sum(lengths) + 3, d, fill=0x3C3C)
    cm.cm_context_set_render_warps(ctx.handle, warps)
    n, order = S.render(k, v)
    torch.cuda.synchronize()
    cm.cm_context_set_render_warps(ctx.handle, 16)
    K_ref, V_ref, o_order = oracle.render(oracle.from_deliveries([oracle_fragment(K, V) for K, V in frags]), THETA)
    assert n == sum(lengths) and order == [f.fid for f in o_order]
    assert np.array_equal(synthetic.to_bits(v[:, :, :n]), V_ref)
    assert assert_k_parity(synthetic.to_bits(k[:, :, :n]), K_ref) == 0
    assert (k.view(torch.int16)[:, :, n:] == 0x3C3C).all() and (v.view(torch.int16)[:, :, n:] == 0x3C3C).all()
    S.close()


# the lines between the full-SM render's two kernels on 152 SMs: 1,216 pairs of 1 KiB items (8
# to 152 planes of K at a time), 48, 62 and 192 MiB of fragments, half of the tokens rotated
@pytest.mark.parametrize("L,H,d,lengths", [
    (19, 8, 128, (16, 16)), (19, 8, 128, (16, 17)), (19, 8, 128, (33, 7, 65)), (19, 8, 512, (4, 4)),
    (19, 8, 512, (4, 5)), (19, 8, 64, (31, 34)), (16, 4, 64, (300, 333, 271)),
    (19, 8, 16, (300, 290)), (8, 4, 256, (39, 41, 43)),
    (28, 8, 128, (283, 283)), (28, 8, 128, (284, 283)), (28, 8, 128, (280, 282, 5)), (28, 8, 128, (878, 877)),
    (28, 8, 128, (878, 878)), (12, 12, 64, (1201, 700, 800)), (24, 8, 32, (1100, 948)), (24, 8, 32, (1100, 949))])
def test_full_width_renders_on_both_sides_of_their_lines(ctx, L, H, d, lengths):
    frags = [_fragment(13 * T + i, L, H, T, d) for i, T in enumerate(lengths)]
    S = cm.FragmentSet(ctx)
    S.ingest_batch(frags)
    total = sum(lengths)
    outs = {}
    for warps in (16, 8):
        cm.cm_context_set_render_warps(ctx.handle, warps)
        k, v = empty_out(L, H, total + 1, d, fill=0x3C3C)
        S.render(k, v)
        outs[warps] = (k.view(torch.int16), v.view(torch.int16))
        for block in (16, 24):
            blocks = -(-total // block)
            table = torch.randperm(blocks + 2, device="cuda:0")[:blocks].to(torch.int32)
            pools = [torch.zeros((L, blocks + 2, block, H, d), dtype=torch.bfloat16, device="cuda:0") for _ in range(2)]
            cm.cm_render_paged(S.handle, cm.cm_paged_cache(
                pools[0].data_ptr(), pools[1].data_ptr(), table.data_ptr(), blocks, block,
                pools[0].stride(1), pools[0].stride(0), pools[0].stride(3), pools[0].stride(2)))
            pos = torch.arange(total, device="cuda:0")
            for pool, flat in zip(pools, outs[warps]):
                got = pool[:, table.long()[pos // block], pos % block].permute(0, 2, 1, 3).view(torch.int16)
                assert torch.equal(got, flat[:, :, :total])
            del pools
        assert all((x[:, :, total:] == 0x3C3C).all() for x in outs[warps])
    cm.cm_context_set_render_warps(ctx.handle, 16)
    assert all(torch.equal(a, b) for a, b in zip(outs[16], outs[8]))
    if L * H * total * d < 4 << 20:
        import oracle
        import synthetic
        K_ref, V_ref, _ = oracle.render(oracle.from_deliveries([oracle_fragment(K, V) for K, V in frags]), THETA)
        assert np.array_equal(synthetic.to_bits(outs[16][1][:, :, :total].view(torch.bfloat16)), V_ref)
        assert np.array_equal(synthetic.to_bits(outs[16][0][:, :, :total].view(torch.bfloat16)), K_ref)
    S.close()

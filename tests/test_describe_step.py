"""mona_describe_step(): the launches of a step, worked out on the host by the code the step itself goes by."""
import random

import pytest
import torch

import paper_2605_26842_b200 as pkg
from paper_2605_26842_b200.binding import FORM_FEW_TILES, FORM_MANY_TILES, FORM_WHOLE_MATRICES, describe_step


def descs(shapes):
    return [pkg.MatrixDesc(r, c, b, 0, 0, 0) for b, r, c in shapes]


@pytest.mark.parametrize("shape,T,form,products", [((1, 256, 512), 5, FORM_FEW_TILES, [15]), ((93, 768, 2048), 5, FORM_MANY_TILES, [16]), ((148, 256, 768), 5, FORM_WHOLE_MATRICES, [16]),
                                                   ((93, 768, 2048), 7, FORM_MANY_TILES, [16, 6]), ((1, 256, 512), 0, None, []), ((1, 250, 512), 5, None, [])])
def test_launches_of_one_bucket(shape, T, form, products):
    got = describe_step(descs([shape]), pkg.default_hparams(ns_steps=T))
    assert [g.products for g in got] == products
    assert all((g.rows, g.cols, g.matrices, g.form) == (shape[1], shape[2], shape[0], form) for g in got)
    assert [g.update_columns > 0 for g in got] == [i == len(products) - 1 for i in range(len(products))]


def test_chunks_and_options():
    got = describe_step(descs([(100, 768, 2048)]))
    assert [(g.matrices, g.slot) for g in got] == [(93, 0), (7, 1)]
    assert [g.slot for g in describe_step(descs([(100, 768, 2048)]), options=pkg.default_options(chunk_overlap=0))] == [0, 0]
    assert describe_step(descs([(100, 768, 2048)]), pkg.default_hparams(ns_precision=1)) == []
    odd = [pkg.MatrixDesc(256, 512, 2, 256 * 512 + 1, 0, 0)]                # a stride that no 16-byte access divides: a separate update
    assert [g.update_columns for g in describe_step(odd)] == [0]
    with pytest.raises(pkg.MonaError):
        describe_step(descs([(1, 256, 512)]), sm_pairs=0)


@pytest.mark.parametrize("shape,sm_pairs,inside", [((40, 256, 256), 8, False), ((24, 512, 512), 16, False), ((40, 1088, 256), 16, False), ((8, 1024, 1024), 4, False),
                                                   ((300, 72, 648), 74, False), ((40, 256, 256), 32, True), ((13, 128, 128), 8, True), ((1, 64, 64), 1, True),
                                                   ((93, 768, 2048), 74, True), ((512, 256, 768), 74, True), ((2, 2048, 2048), 74, True)])
def test_few_pairs_leave_the_update_of_many_tiles_to_a_pass_of_its_own(shape, sm_pairs, inside):
    assert [g.update_columns > 0 for g in describe_step(descs([shape]), sm_pairs=sm_pairs)] == [inside]


WHOLE_PAYS = {(256, 256): [9, 12, 74, 100, 148, 222, 370, 512], (128, 128): [8, 100, 160, 222, 300, 512], (64, 64): [8, 40], (192, 256): [222, 370, 512],
              (256, 512): [74, 100, 148, 222, 370, 512], (256, 768): [111, 148, 222, 370, 512], (768, 256): [148], (128, 1024): [148], (1024, 256): [148],
              (72, 648): [148], (96, 1024): [148], (64, 512): [512]}
SPREADING_PAYS = {(256, 256): [1, 4, 8, 160, 185, 260], (192, 256): [160], (64, 64): [4], (256, 768): [74, 90, 185, 296], (256, 1280): [74, 90, 111, 185],
                  (72, 648): [300], (96, 1024): [512], (128, 1024): [512], (128, 1280): [300], (192, 2048): [74], (256, 4096): [74, 222], (264, 264): [8, 148]}


@pytest.mark.parametrize("whole,shape,count", [(w, s, c) for w, table in ((True, WHOLE_PAYS), (False, SPREADING_PAYS)) for s, cs in table.items() for c in cs])
def test_whole_matrices_where_they_were_measured_faster(whole, shape, count):
    assert all((g.form == FORM_WHOLE_MATRICES) == whole for g in describe_step(descs([(count, *shape)])))


@pytest.mark.parametrize("shapes,bucket,whole", [([(40, 256, 256), (4, 1024, 1024), (2, 2816, 1024)], 0, False), ([(8, 256, 200), (4, 1024, 1024)], 0, False),
                                                 ([(2, 848, 608), (2, 320, 1472), (42, 256, 256)], 2, False), ([(37, 896, 192), (4, 576, 1024)], 0, False),
                                                 ([(26, 192, 256), (8, 192, 128), (8, 448, 128)], 0, True), ([(6, 384, 128), (10, 256, 128)], 1, True)])
def test_whole_matrices_on_a_share_of_the_pairs(shapes, bucket, whole):
    got = {(g.rows, g.cols): g.form for g in describe_step(descs(shapes))}
    assert (got[shapes[bucket][1:]] == FORM_WHOLE_MATRICES) == whole


def random_small_set(rng):
    shapes = {}
    for _ in range(rng.randint(2, 9)):
        r, c = (8 * int(8 * 32 ** rng.random()) for _ in range(2))
        shapes[(r, c)] = rng.randint(1, 6)
    return [(b, r, c) for (r, c), b in shapes.items()]


@pytest.mark.parametrize("shapes", [[(13, 128, 128), (5, 2048, 2048), (3, 192, 128), (2, 448, 96)], [(40, 256, 256), (4, 1024, 1024), (2, 2816, 1024)]]
                         + [random_small_set(random.Random(seed)) for seed in range(40)])
def test_launches_that_run_side_by_side_fit_the_device(shapes):
    """Where a set has small buckets only, one launch of every slot can run at a time: together they use no more SM pairs than there
    are, so that none has to wait until another has ended."""
    for sm_pairs in (74, 20, 5):
        launches = describe_step(descs(shapes), sm_pairs=sm_pairs)
        widest = {}
        for g in launches:
            widest[g.slot] = max(widest.get(g.slot, 0), g.sm_pairs)
        assert all(w >= 1 for w in widest.values()) and sum(widest.values()) <= sm_pairs, [(g.rows, g.cols, g.slot, g.sm_pairs) for g in launches]


@pytest.mark.gpu
@pytest.mark.parametrize("shapes,T", [([(1, 256, 512)], 5), ([(100, 768, 2048)], 7), ([(40, 256, 256), (4, 1024, 1024), (2, 2816, 1024)], 5), ([(60, 512, 512), (8, 256, 256)], 5)])
def test_a_step_launches_what_is_described(shapes, T):
    dev = torch.device("cuda", 0)
    p, g = [torch.zeros(s, device=dev) for s in shapes], [torch.full(s, 1e-3, device=dev) for s in shapes]
    hp = pkg.default_hparams(ns_steps=T)
    opt = pkg.MonaOptimizer(p)
    opt.step(hp, p, g)
    assert opt.poll_status()[0] == 0
    launches = describe_step(opt.descs, hp)
    chunks = len({(x.rows, x.cols, x.slot, x.matrices) for x in launches})
    updates = chunks - sum(x.update_columns > 0 for x in launches)
    assert opt.last_launch_count() == chunks + len(launches) + updates        # a prologue per chunk, and an update where none is inside
    opt.close()

"""Half or whole 8 x 8 blocks a compositing warp: for every batch measured on the
GPU, the variant the library chooses takes at most 8% longer than the better one
(the lines are drawn over many batches; these are the ones its comment lists).
Host arithmetic only."""
import ctypes as C

import numpy as np
import pytest

# points, view sizes in turn, views, visible point-views, (tile, point) pairs of
# 16 x 16 tiles, then forward half / whole and backward half / whole, in us:
# streamed, streamed with the stored list, persistent, persistent with the list,
# and the first two with the pairs counted
MEASURED = [
    (227000, "101x339,1270x365,400x300,640x480", 7, 1185092, 1896506,
     (325, 452, 451, 609), (451, 763, 645, 1083), (362, 510, 540, 756),
     (498, 914, 677, 1217), (349, 451, 499, 691), (467, 765, 673, 1078)),
    (7000, "97x120,150x130,200x100,128x256", 4, 27502, 37613,
     (32, 41, 60, 85), (43, 73, 89, 137), (53, 77, 81, 114),
     (70, 130, 106, 162), (35, 41, 62, 92), (43, 73, 89, 137)),
    (500000, "800x800", 4, 2000000, 3965121,
     (178, 181, 405, 344), (238, 279, 493, 484), (189, 190, 369, 363),
     (244, 321, 455, 485), (199, 188, 472, 416), (261, 281, 538, 509)),
    (272000, "640x480,333x777,1000x500", 33, 8611548, 15105001,
     (885, 850, 2057, 1688), (1179, 1326, 2475, 2341), (855, 785, 1907, 1554),
     (1246, 1329, 2217, 2046), (944, 909, 2572, 2008), (1260, 1335, 2780, 2466)),
    (1000000, "1920x1080", 1, 957750, 4020948,
     (138, 131, 383, 284), (254, 305, 454, 398), (146, 141, 336, 262),
     (296, 351, 415, 374), (151, 134, 398, 307), (289, 306, 461, 401)),
    (45000, "1024x768", 1, 44913, 106308,
     (25, 24, 56, 52), (38, 44, 70, 72), (44, 51, 58, 78),
     (64, 78, 71, 107), (42, 29, 67, 67), (61, 53, 78, 78)),
    (808000, "235x230,1737x835,800x600,500x900", 8, 6197545, 12616347,
     (568, 609, 1131, 945), (766, 1005, 1355, 1390), (556, 676, 1019, 1011),
     (836, 1165, 1232, 1564), (582, 634, 1260, 1056), (794, 1011, 1430, 1420)),
    (136000, "300x300,800x400,500x333", 8, 1011110, 1554938,
     (147, 164, 299, 299), (214, 281, 385, 445), (182, 204, 279, 324),
     (254, 349, 375, 534), (160, 171, 332, 328), (226, 281, 416, 449)),
    (136000, "300x300,800x400,500x333", 43, 5479007, 8403685,
     (552, 535, 1356, 1128), (766, 889, 1619, 1561), (560, 538, 1226, 1012),
     (868, 913, 1461, 1388), (587, 566, 1829, 1401), (852, 910, 1975, 1615)),
]


@pytest.mark.parametrize("row", MEASURED, ids=[f"{r[0]}x{r[2]}" for r in MEASURED])
def test_the_choice_is_the_faster_one(row):
    from paper_2205_14330_gb300 import build
    build.build()
    from paper_2205_14330_gb300 import pbr
    n, sizes, views, n_vis, n_pairs = row[:5]
    sizes = [tuple(int(x) for x in s.split("x")) for s in sizes.split(",")]
    cams = []
    for v in range(views):
        w, h = sizes[v % len(sizes)]
        f = np.float32(w / 2.0 / np.tan(np.radians(25.0)))
        cams.append(dict(fx=f, fy=f, cx=w / 2.0, cy=h / 2.0, R=np.eye(3), t=np.zeros(3), width=w,
                         height=h))
    p = C.c_void_p(16)  # not read
    pts = pbr.Points(p, p, p, p, n, 0, 0)
    f = pbr.lib().pbr_test_raster_lanes
    f.argtypes = [C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p, C.c_int32,
                  C.c_int64, C.c_int64, C.c_void_p]
    for k, t in enumerate(row[5:]):
        o = pbr.default_opts(persistent=int(k in (2, 3)), no_pair_stats=int(k < 4))
        two = (C.c_int32 * 2)()
        assert f(C.byref(pts), 1, None, pbr.make_cameras(cams), views, C.byref(o), k % 2, n_vis,
                 n_pairs, two) == 0
        for phase in (0, 1):
            half, whole = t[2 * phase:2 * phase + 2]
            assert (whole if two[phase] else half) <= 1.08 * min(half, whole), (k, phase)

// The box code of the BVH (csrc/hpt_boxes.cuh) compiled with the host compiler, for the tests.
#include "hpt_boxes.cuh"

using namespace hpt;

struct Coder {
    BoxGrid grid;
    float pad, bound;
    int wide;
    Box all;
};

static Box box_of(const float *lo, const float *hi)
{
    Box b;
    for (int k = 0; k < 3; ++k) { b.lo[k] = lo[k]; b.hi[k] = hi[k]; }
    return b;
}

// wide: -1 by the growth of the boxes
extern "C" void *coder_new(int n, const float *lo, const float *hi, float max_abs, int wide)
{
    std::vector<Box> pb;
    std::vector<int> prims;
    for (int i = 0; i < n; ++i) {
        pb.push_back(box_of(lo + 3 * i, hi + 3 * i));
        prims.push_back(i);
    }
    Coder *c = new Coder;
    c->pad = box_pad(max_abs);
    c->bound = max_abs + c->pad;
    c->grid = box_grid(pb, prims, c->pad);
    c->all.reset();
    for (const Box &b : pb) c->all.grow(b);
    BoxGrowth g;
    for (const Box &b : pb) {
        unsigned q, h[3];
        for (int k = 0; k < 3; ++k) box_code(c->grid, c->pad, b.lo[k], b.hi[k], k, q, h[k]);
        g.add(box_growth(c->grid, c->pad, b, h));
    }
    c->wide = wide < 0 ? g.wide() : wide;
    if (c->wide) c->grid = WIDE_GRID;
    return c;
}
extern "C" void coder_free(void *p) { delete (Coder *)p; }

extern "C" int coder_wide(const void *p) { return ((const Coder *)p)->wide; }
extern "C" int coder_near(const void *p, const float *lo, const float *hi)
{
    const Coder *C = (const Coder *)p;
    return origins_near(C->grid, C->wide, C->bound, box_of(lo, hi));
}

// per box i, as child 0 beside an empty child 1: entry and exit distance of the ray from o[i] along d[i] with the
// reciprocals inv[i]; far: started near the geometry first, as such jobs do; returns how many times the
// empty child was entered
extern "C" int box_test(const void *p, int far, int n, const float *lo, const float *hi, const float *o, const float *d,
                        const float *inv, float *tmin, float *tmax)
{
    const Coder *C = (const Coder *)p;
    int bad = 0;
    for (int i = 0; i < n; ++i) {
        float2 cc[3], hh[3];
        for (int k = 0; k < 3; ++k) {
            if (C->wide) {
                box_code_wide(C->pad, lo[3 * i + k], hi[3 * i + k], cc[k].x, hh[k].x);
                cc[k].y = 0.0f;
                hh[k].y = -INFINITY;
                continue;
            }
            unsigned c, h;
            box_code(C->grid, C->pad, lo[3 * i + k], hi[3 * i + k], k, c, h);
            cc[k] = centres(c);
            hh[k] = extents(h | NO_BOX << 16);
        }
        float3 oi = make_float3(o[3 * i], o[3 * i + 1], o[3 * i + 2]);
        const float3 di = make_float3(d[3 * i], d[3 * i + 1], d[3 * i + 2]);
        double x = oi.x, y = oi.y, z = oi.z;
        for (int k = 0; far && k < 2; ++k) {
            const double t = far_start(C->all, oi, di);
            x += t * di.x;
            y += t * di.y;
            z += t * di.z;
            oi = make_float3((float)x, (float)y, (float)z);
        }
        const GridRay r = grid_ray<true>(*C, oi, make_float3(inv[3 * i], inv[3 * i + 1], inv[3 * i + 2]));
        float e0, e1;
        box_pair(cc, hh, r, 1e30f, tmin[i], tmax[i], e0, e1);
        bad += e0 <= e1;
    }
    return bad;
}

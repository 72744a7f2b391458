// The row walk's host arrays (RowImage) of a host-only handle, for
// tests/test_row_trees.py: host.cpp is compiled in, and its kernels' launchers
// are left unresolved.
#include "host.cpp"

// rows.cu's: every vocabulary here fits
int domino::row_smem_bytes(int32_t, bool, bool) { return 0; }

namespace {

struct Array {
    const void* p;
    int64_t bytes;
};
template <typename T>
Array array_of(const std::vector<T>& v) {
    return Array{v.data(), (int64_t)(v.size() * sizeof(T))};
}

}  // namespace

extern "C" {

// nullptr: make_row_image() refuses the handle.
void* row_image_make(domino_t h) {
    RowImage* im = new RowImage;
    if (make_row_image(h, *im)) return im;
    delete im;
    return nullptr;
}
void row_image_free(void* p) { delete static_cast<RowImage*>(p); }

// Array `which` of an image, and {record strides, loop sets, wide, dense, visits}.
int row_image_get(void* p, int which, const void** data, int64_t* bytes) {
    const RowImage& im = *static_cast<RowImage*>(p);
    const Array all[] = {array_of(im.rb.node),  array_of(im.rb.ncls), array_of(im.rb.dtok), array_of(im.roots),
                         array_of(im.loopbits), array_of(im.keeps),   array_of(im.srec),    array_of(im.srec_next),
                         array_of(im.trec),     array_of(im.xrange),  array_of(im.exits),   array_of(im.start),
                         array_of(im.loop_of),  array_of(im.ret)};
    if (which < 0 || which >= (int)(sizeof(all) / sizeof(all[0]))) return -1;
    *data = all[which].p;
    *bytes = all[which].bytes;
    return 0;
}
void row_image_info(void* p, int64_t* out) {
    const RowImage& im = *static_cast<RowImage*>(p);
    out[0] = im.stride;
    out[1] = im.stride_next;
    out[2] = (int64_t)im.roots.size();
    out[3] = im.rb.wide;
    out[4] = im.cost.dense;
    out[5] = im.cost.visits;
}

// The automaton's own table and pop targets, as the wide form reads them.
int row_image_table(domino_t h, const void** data, int64_t* bytes, const void** ret, int64_t* ret_bytes) {
    const Array t = h->stack ? array_of(h->t32) : array_of(h->t16), r = array_of(h->ret);
    *data = t.p;
    *bytes = t.bytes;
    *ret = r.p;
    *ret_bytes = r.bytes;
    return 0;
}

}  // extern "C"
